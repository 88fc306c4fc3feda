"""AUTO's binary32 kernel (three-way split operands on the tensor cores) at the edges of its variants, against the oracle.

Bounds: the split products are exact to 2^-24 and every tile's sum is rounded to nearest, so the error is binary32's: 2e-6 of
max |V| and 2e-6 relative L2 (measured at most 5e-7), a fifth of the path's stated tolerance.  Scores carry their own
rounding into the weights, 2^-24 of a score: those cases have bounds of their own, the stated 1e-5 for scores of up to 20 (1e-6 of a
weight) and 1e-4 for scores of up to a thousand (6e-5).  AUTO reports SIMT for both binary32 kernels and the plain one would meet these
bounds too; which one ran shows in the bits."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bd():
    from paper_2304_11267_b200 import binding
    from paper_2304_11267_b200 import build
    build.build()
    binding.load()
    return binding


def draw(seed, B, H, Nq, Nk, d):
    g = np.random.default_rng(seed)
    return tuple(g.standard_normal((B, H, n, d), dtype=np.float32) for n in (Nq, Nk, Nk))


def run(bd, q, k, v, scale, tokens_first=False):
    a = bd.Attention(layout=bd.LAYOUT_BNHD if tokens_first else bd.LAYOUT_BHND)
    t = [torch.from_numpy(np.ascontiguousarray(x.transpose(0, 2, 1, 3)) if tokens_first else x).cuda() for x in (q, k, v)]
    out = a.forward(*t, scale=scale)
    a.check()
    assert a.last_mode == bd.MODE_SIMT
    out = out.cpu().numpy()
    return out.transpose(0, 2, 1, 3) if tokens_first else out


def check(got, ref, v, bound=2e-6):
    got = got.astype(np.float64)
    assert np.all(np.isfinite(got))
    err, rel = np.abs(got - ref).max() / np.abs(v).max(), np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err <= bound and rel <= bound, (err, rel)


# head dims at the edges of the variants (48, 64, 96, 160) and of the 4-, 8- and 16-column granules; rows around one and two
# query tiles; keys around the 32- and 64-key tiles
@pytest.mark.parametrize("d", [4, 8, 20, 40, 44, 48, 52, 64, 68, 80, 96, 100, 160])
@pytest.mark.parametrize("Nq,Nk", [(1, 1), (127, 64), (129, 65), (257, 33), (300, 191)])
def test_variants(bd, d, Nq, Nk):
    q, k, v = draw(d + Nq, 1, 3, Nq, Nk, d)
    scale = float(np.float32(d ** -0.5))
    check(run(bd, q, k, v, scale), oracle.forward(q, k, v, scale)[0], v)


# one head dim for every count of eight columns, and some that end in half of one: the contraction of Q K^T is compiled for each
@pytest.mark.parametrize("d", list(range(8, 168, 8)) + [12, 36, 76, 84, 92, 108, 124, 140, 148, 156])
def test_every_count_of_columns(bd, d):
    scale = float(np.float32(d ** -0.5))
    for H, Nq in ((3, 150),) + (((16, 1250),) if d <= 48 else ()):   # (one and two query tiles a CTA)
        q, k, v = draw(d, 1, H, Nq, 150, d)
        check(run(bd, q, k, v, scale), oracle.forward(q, k, v, scale)[0], v)


@pytest.mark.parametrize("d,Nq", [(40, 1300), (36, 2500)])
def test_two_query_tiles_per_cta(bd, d, Nq):
    q, k, v = draw(d, 2, 8, Nq, 200, d)   # more tiles than SMs; the last CTA of a head has one
    scale = float(np.float32(d ** -0.5))
    ref = oracle.forward(q, k, v, scale)[0]
    check(run(bd, q, k, v, scale), ref, v)
    check(run(bd, q, k, v, scale, tokens_first=True), ref, v)


FOUR = pytest.mark.parametrize("d,H,Nq", [(40, 2, 150), (40, 16, 1250), (80, 2, 150), (160, 2, 150)])   # the variants


@FOUR
@pytest.mark.parametrize("scale", [-0.4, 0.0])
def test_negative_and_zero_scale(bd, d, H, Nq, scale):
    q, k, v = draw(d, 1, H, Nq, 150, d)
    check(run(bd, q, k, v, scale), oracle.forward(q, k, v, scale)[0], v, 1e-5)


@pytest.mark.parametrize("d,H,Nq", [(40, 2, 260), (40, 16, 1250), (80, 2, 260), (160, 2, 260)])   # the four variants
def test_scores_that_leave_the_anchor_behind(bd, d, H, Nq):
    """The anchor is the first key tile's maximum; keys that grow 40-fold twice raise some rows' scores by hundreds, past the
    2^64 at which a row is re-anchored (and lower others', whose weights vanish)."""
    q, k, v = draw(d, 1, H, Nq, 260, d)
    k[:, :, 100:] *= 40.0
    k[:, :, 210:] *= 6.0
    scale = float(np.float32(d ** -0.5))
    ref = oracle.forward(q, k, v, scale)[0]
    scores = np.einsum("bhid,bhjd->bhij", q.astype(np.float64), k.astype(np.float64)) * scale
    assert (scores[..., 210:].max(-1) - scores[..., :32].max(-1)).max() > 64 * np.log(2.0)
    check(run(bd, q, k, v, scale), ref, v, 1e-4)


@pytest.mark.parametrize("d,H,Nq", [(40, 2, 150), (40, 8, 2500), (80, 2, 150), (160, 2, 150)])   # the four variants
@pytest.mark.parametrize("what", ["inf in V", "largest V", "inf in K", "largest K", "nan in Q", "V and rising scores"])
def test_the_ends_of_the_range(bd, what, d, H, Nq):
    """Values without three bfloat16 parts, and weights whose products overflow although the result is finite: what the plain kernel
    returns comes back, infinities and NaNs included."""
    g = torch.Generator().manual_seed(d + Nq)
    q, k, v = (torch.randn(1, H, n, d, generator=g) for n in (Nq, 200, 200))
    if what == "inf in V":
        v[0, 1, 70, 3] = float("inf")
        v[0, 1, 9, d - 1] = float("-inf")
    elif what == "largest V":
        v[0, 1, 70, 3] = v[0, 0, 9, d - 1] = torch.finfo(torch.float32).max
    elif what == "inf in K":        # a score of -inf: weight zero
        q[0, 1, :, 5] = q[0, 1, :, 5].abs() + 0.1
        k[0, 1, 70, 5] = float("-inf")
    elif what == "largest K":       # scores of some 1e38, of either sign
        k[0, 1, 70, 5] = torch.finfo(torch.float32).max
        q[0, 1, :, 5] *= 0.1
    elif what == "nan in Q":
        q[0, 0, Nq - 1, 0] = q[0, 1, 17, 2] = float("nan")
    else:                           # weights near 2^47 against the first key tile's maximum times V near 2^90
        q = 0.5 + 0.5 * torch.rand(q.shape, generator=g)
        k *= 0.01
        k[:, :, 150] += 33.0 / 0.75 / d ** 0.5
        v *= 2.0 ** 90
    q, k, v = q.cuda(), k.cuda(), v.cuda()
    plain = bd.Attention(mode=bd.MODE_SIMT).forward(q, k, v)
    a = bd.Attention()
    got = a.forward(q, k, v)
    a.check()
    assert bool(torch.isfinite(plain).all()) == (what not in ("inf in V", "nan in Q"))
    torch.testing.assert_close(got, plain, rtol=1e-5, atol=1e-5 * float(v[v.isfinite() & (v.abs() < 1e37)].abs().max()), equal_nan=True)


@pytest.mark.parametrize("d,H,Nq", [(40, 2, 150), (40, 8, 2500), (80, 2, 150), (160, 2, 150)])   # the four variants
def test_auto_runs_on_the_tensor_cores(bd, d, H, Nq):
    """The two kernels add in different orders and round differently: over thousands of values their bits differ; the plain
    kernel in AUTO's place would give its own."""
    t = [torch.from_numpy(x).cuda() for x in draw(d + 7, 1, H, Nq, 400, d)]
    auto, plain = bd.Attention(), bd.Attention(mode=bd.MODE_SIMT)
    got, want = auto.forward(*t), plain.forward(*t)
    assert auto.last_mode == plain.last_mode == bd.MODE_SIMT
    assert float((got != want).float().mean()) > 0.1
    torch.testing.assert_close(got, want, rtol=1e-5, atol=1e-5)


@FOUR
def test_small_values(bd, d, H, Nq):
    """V near 2^-100 has its three parts, and Q near 2^-60 against K near 2^60."""
    q, k, v = draw(d + 1, 1, H, Nq, 150, d)
    scale = float(np.float32(d ** -0.5))
    ref = oracle.forward(q, k, v, scale)[0]
    got = run(bd, q * np.float32(2.0 ** -60), k * np.float32(2.0 ** 60), v * np.float32(2.0 ** -100), scale)
    check(got.astype(np.float64) * 2.0 ** 100, ref, v)


@pytest.mark.parametrize("d,Nq,Nk", [(40, 2500, 65), (48, 1250, 200), (4, 1250, 64), (44, 1250, 130)])   # two query tiles per CTA
def test_columns_of_v_far_apart(bd, d, Nq, Nk):
    """Columns of V from 2^-90 to 2^90, keys that grow 2^10-fold: a column's error is relative to that column."""
    q, k, v = draw(d + Nq, 1, 16, Nq, Nk, d)
    v *= np.float32(2.0) ** np.linspace(-90, 90, d).round().astype(np.float32)
    v[:, :, 64:] *= np.float32(2.0 ** 10)
    scale = float(np.float32(d ** -0.5))
    ref = oracle.forward(q, k, v, scale)[0]
    got = run(bd, q, k, v, scale).astype(np.float64)
    assert np.all(np.isfinite(got))
    assert (np.abs(got - ref).max(axis=(0, 1, 2)) / np.abs(v).max(axis=(0, 1, 2))).max() <= 2e-6


@pytest.mark.parametrize("growth", [2.0 ** 5, 2.0 ** 12, 2.0 ** 15])
def test_weights_past_the_range_of_a_part(bd, growth):
    """Two query tiles per CTA: keys along q itself give the second and third key tiles a largest weight of about `growth` times the first
    one's and its square, in rows of some warps only."""
    q, k, v = draw(77, 1, 16, 1300, 190, 40)
    q /= np.linalg.norm(q, axis=-1, keepdims=True)
    k *= 0.01
    for at, x in ((100, growth), (150, growth * growth)):
        k[:, :, at] = q[:, :, 640] * np.float32(np.log(x) * 40 ** 0.5)
    scale = float(np.float32(40 ** -0.5))
    check(run(bd, q, k, v, scale), oracle.forward(q, k, v, scale)[0], v, 1e-5)


def around_one_key(seed, Nk, at, spread):
    """Sixteen heads in which key `at` lies 10 to 40 binary orders above all the others (`spread`: their deviation, in such orders).
    More query tiles than SMs; d = 40."""
    g = np.random.default_rng(seed)
    q, k = np.zeros((1, 16, 1250, 40), np.float32), g.standard_normal((1, 16, Nk, 40), dtype=np.float32)
    scale = float(np.float32(40 ** -0.5))
    order = np.float32(np.log(2.0) / scale)
    q[..., 0] = g.uniform(0.95, 1.05, q.shape[:3])
    k[..., 0] *= spread * order
    k[0, :, at, 0] = np.linspace(10, 40, 16) * order
    return q, k, scale


@pytest.mark.parametrize("Nk,at,spread", [(4096, 0, 0), (4096, 0, 1), (4096, 2000, 0), (9216, 5, 0)])
@pytest.mark.parametrize("value", [0.01, 0.0])
def test_keys_far_below_one(bd, Nk, at, spread, value):
    """Thousands of keys far below a dominant one whose V is small, or zero: each weighs next to nothing, and together they are the
    output.  The result is right relative to itself, head by head: 1e-5, the path's bound (scores of up to 40 binary orders carry 4e-6 of a
    weight)."""
    q, k, scale = around_one_key(Nk + at, Nk, at, spread)
    v = np.random.default_rng(1).uniform(0.5, 1.0, k.shape).astype(np.float32)
    v[:, :, at] = value
    rows = (np.arange(16)[:, None] * 1250 + np.arange(0, 1250, 25)).ravel()
    ref = oracle.forward(q, k, v, scale, rows=rows)[0].reshape(16, -1, 40)
    got = run(bd, q, k, v, scale)[0, :, ::25].astype(np.float64)
    assert np.abs(got - ref).max() <= 2e-6
    rel = np.linalg.norm(got - ref, axis=(1, 2)) / np.linalg.norm(ref, axis=(1, 2))
    assert rel.max() <= 1e-5, rel


@pytest.mark.parametrize("outlier", [2.0 ** 26, 2.0 ** 30])
def test_an_outlier_in_v_without_weight(bd, outlier):
    """A column of V whose largest value, by far, belongs to a key without weight: the others' products are as exact as ever."""
    q, k, v = draw(11, 1, 16, 1250, 200, 40)
    q[..., 0], k[..., 0] = 1.0, 0.0
    k[:, :, 3, 0] = -100.0 * 40 ** 0.5 * np.log(2.0)
    v[:, :, 3, ::3] = outlier
    scale = float(np.float32(40 ** -0.5))
    check(run(bd, q, k, v, scale), oracle.forward(q, k, v, scale)[0], np.delete(v, 3, axis=2))


def test_one_key_comes_back_as_it_is(bd):
    """One key of weight one: V's three parts add up to V, bit by bit."""
    q, k, v = draw(5, 1, 16, 1250, 1, 40)
    assert np.array_equal(run(bd, q, k, v, 0.0), np.broadcast_to(v, q.shape))


# two query tiles per CTA: a last half or whole key tile without a key, head dims around the 4-, 8- and 16-column granules
@pytest.mark.parametrize("d", [4, 8, 20, 28, 44, 48])
@pytest.mark.parametrize("Nk", [1, 31, 33, 63, 97])
def test_two_query_tiles_at_the_edges(bd, d, Nk):
    q, k, v = draw(d + Nk, 1, 16, 1250, Nk, d)
    scale = float(np.float32(d ** -0.5))
    check(run(bd, q, k, v, scale), oracle.forward(q, k, v, scale)[0], v)
