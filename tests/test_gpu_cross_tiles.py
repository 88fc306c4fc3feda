"""The one-tile cross-attention kernel over its key tiles, row tiles, fetches and head dims, against the oracle (tolerances of
test_gpu_parity.py), and both CROSS kernels on the same problem."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import test_gpu_parity as parity  # noqa: E402


@pytest.fixture(scope="module")
def bd():
    from paper_2304_11267_b200 import binding
    from paper_2304_11267_b200 import build
    build.build()
    binding.load()
    return binding


def run(bd, q, k, v, scale, tokens_first=False, **options):
    a = bd.Attention(layout=bd.LAYOUT_BNHD if tokens_first else bd.LAYOUT_BHND, options=bd.Options(**options))
    t = [torch.from_numpy(np.ascontiguousarray(x.transpose(0, 2, 1, 3)) if tokens_first else x).cuda() for x in (q, k, v)]
    out = a.forward(*t, scale=float(scale))
    a.check()
    assert a.last_mode == bd.MODE_CROSS
    out = out.cpu().numpy()
    a.close()
    return out.transpose(0, 2, 1, 3) if tokens_first else out


# keys around the tiles of 64, 80 and 128; head dims at the edges of the chunks and of the untiled fetch; rows that leave a
# tile of 64 with one row, a warp with none
@pytest.mark.parametrize("Nk", [1, 16, 63, 64, 65, 77, 80, 81, 127, 128])
@pytest.mark.parametrize("d,Nq", [(8, 65), (40, 64), (48, 97), (56, 129), (64, 33), (80, 200), (128, 64), (136, 31), (160, 130)])
def test_key_tiles_and_head_dims(bd, d, Nq, Nk):
    q, k, v = parity.rand_qkv(d + Nk, 2, 3, Nq, Nk, d, qmult=3.0)   # (some rows' maximum lies far above their first score)
    scale = np.float32(d ** -0.5)
    ref, _, _ = oracle.forward(q, k, v, scale)
    got = run(bd, q, k, v, scale, cross_one_tile=1)
    parity.check(got, ref, v, what="d=%d Nq=%d Nk=%d" % (d, Nq, Nk))
    assert np.array_equal(got, run(bd, q, k, v, scale, tokens_first=True, cross_one_tile=1))


# more tiles than the GPU holds at once: 128-row tiles; the problem right at the line between the two kernels
@pytest.mark.parametrize("B,Nq,d", [(2, 4733, 40), (2, 2304, 80), (2, 4736, 40), (3, 1500, 160)])
def test_row_tiles_and_the_line_between_the_kernels(bd, B, Nq, d):
    q, k, v = parity.rand_qkv(Nq, B, 8, Nq, 77, d)
    scale = np.float32(d ** -0.5)
    rows = np.arange(0, B * 8 * Nq, 11, dtype=np.int64)
    ref, _, _ = oracle.forward(q, k, v, scale, rows=rows)
    for opts in ({}, {"cross_one_tile": 1}):
        parity.check(run(bd, q, k, v, scale, **opts).reshape(-1, d)[rows], ref, v, what="%d x 77 d=%d %s" % (Nq, d, opts))


# token-major calls at the line between the kernels: one tile, half an SM's worth of tiles and one more; groups at two per SM
@pytest.mark.parametrize("dtype", ["float16", "bfloat16"])
@pytest.mark.parametrize("n,Nq,Nk,d", [(1, 1, 65, 40), (1, 1153, 77, 40), (1, 1183, 80, 48), (1, 1185, 77, 8), (3, 700, 77, 40),
                                       (5, 947, 80, 24), (4, 1300, 65, 48)])
def test_token_major_line_between_the_kernels(bd, n, Nq, Nk, d, dtype):
    g = torch.Generator(device="cuda").manual_seed(Nq + d)
    sets = [tuple(torch.randn(1, m, 8, d, generator=g, device="cuda").to(getattr(torch, dtype)) for m in (Nq, Nk, Nk)) for _ in range(n)]
    results = []
    for options in ({}, {"cross_one_tile": 1}):
        a = bd.Attention(layout=bd.LAYOUT_BNHD, options=bd.Options(**options))
        outs = [torch.zeros_like(q) for q, _, _ in sets]
        problems = bd.make_problems([(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), 1, 8, Nq, Nk, d, d ** -0.5)
                                     for (q, k, v), o in zip(sets, outs)])
        code = bd.F16 if dtype == "float16" else bd.BF16
        assert bd.sd_attn_forward_batch(a.handle, problems, code, torch.cuda.current_stream().cuda_stream) == bd.OK
        results.append(outs + [a.forward(*t) for t in sets])
        a.check()
    for i in range(n):
        assert torch.equal(results[0][i], results[0][n + i])                                              # the group and the call alone
        assert torch.equal(results[0][i], results[1][i]) and torch.equal(results[0][i], results[1][n + i])   # either kernel
        q, k, v = (t.transpose(1, 2).double() for t in sets[i])
        ref = (torch.softmax(q @ k.transpose(-1, -2) * d ** -0.5, -1) @ v).transpose(1, 2)
        assert float((results[0][i].double() - ref).norm() / ref.norm()) < (2e-3 if dtype == "float16" else 1.6e-2)


@pytest.mark.parametrize("dtype", ["float16", "bfloat16"])
@pytest.mark.parametrize("Nk", [2, 64, 81, 128])
def test_the_largest_weight_is_exact(bd, Nk, dtype):
    """Up to 64 and from 81 keys a row's exponents are anchored at its maximum, so the largest weight is 1 and only the others
    are rounded, by u = 2^-11 (bfloat16: 2^-8) of themselves.  Where the others make up less than a quarter of the row's sum, a
    constant V = 1 comes back as 1 +- u / 4 (+ 128 half steps of binary16's subnormals, 2^-18), which rounds to 1: the next value
    below is u away.  With the anchor at another score the largest weight itself is off by up to u, and a fifth of the rows are
    not 1.  Here the second key leads the first by 1.5 to 2.25 and the others by 7.5 to 11.25."""
    r = 1.0 + 0.5 * torch.rand(2, 4, 512, 1, generator=torch.Generator().manual_seed(Nk))
    q = (r * torch.ones(64)).to(getattr(torch, dtype))
    k = torch.full((2, 4, Nk, 64), -6.0 / 8.0).to(q.dtype)
    k[:, :, 0], k[:, :, 1] = 0.0, 1.5 / 8.0
    p = torch.softmax(q.double() @ k.double().transpose(-1, -2) / 8.0, -1)
    assert p.max(-1).values.min() > 0.75
    a = bd.Attention()
    out = a.forward(q.cuda(), k.cuda(), torch.ones_like(k).cuda())
    a.check()
    assert a.last_mode == bd.MODE_CROSS
    assert bool((out == 1.0).all())
