"""The direct 3x3 convolution at the edges of its tiles and of its plan, and the transformed domain behind the same class
for images it does not cover, against the oracle.

The direct kernel multiplies the binary16 values as they are, accumulates in binary32 and rounds once: |err| <= 2^-11 |y|
plus binary32 accumulation over 9 C products (2e-6 of the sum of their magnitudes, about sqrt(9 C) r.m.s. here).
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import test_gpu_winograd as wg  # noqa: E402


@pytest.fixture(scope="module")
def bd():
    from paper_2304_11267_b200 import binding
    from paper_2304_11267_b200 import build
    build.build()
    binding.load()
    return binding


# one position and one channel group; just under, at and over 128 positions of the padded raster (W + 2) (H + 1); three
# images in one tile; the widest image (126) and rows that leave a tile one position; channel counts around 64 and K around
# the 16-filter granule, one and several filter tiles; few tiles and many channels (the steps split two- to eightfold)
@pytest.mark.parametrize("N,H,W,C,K", [
    (1, 1, 1, 8, 8), (1, 6, 15, 8, 8), (1, 7, 14, 16, 24), (1, 7, 15, 64, 40), (3, 3, 3, 72, 16), (2, 2, 126, 64, 32),
    (1, 1, 126, 8, 264), (2, 5, 125, 56, 72), (1, 8, 8, 1280, 64), (2, 9, 12, 640, 328), (1, 16, 16, 320, 1280),
    (1, 33, 43, 128, 200), (4, 12, 11, 320, 320), (2, 31, 29, 192, 648), (1, 9, 9, 832, 640), (1, 16, 16, 512, 968),
])
def test_against_the_oracle(bd, N, H, W, C, K):
    assert bd.sd_winograd_direct_supported(N, H, W, C, K)
    x, w, b = wg.make(500 + H + W + C + K, N, H, W, C, K)
    ref = oracle.conv3x3_forward(x, w, b)
    got = wg.run(bd, x, w, b).astype(np.float64)
    err = np.abs(got - ref)
    assert np.all(err <= 2.0 ** -11 * np.abs(ref) + 2e-5), float((err - 2.0 ** -11 * np.abs(ref)).max())


def test_guard_bytes_and_repeated_bits(bd):
    x, w, b = wg.make(3, 2, 9, 13, 640, 72)
    layer = bd.WinogradConv3x3(torch.from_numpy(w).cuda(), torch.from_numpy(b).cuda())
    tx = torch.from_numpy(x).cuda()
    n, guard = 2 * 9 * 13 * 72, 4096
    buf = torch.full((n + 2 * guard,), 55.0, dtype=torch.float16, device="cuda")
    out = buf[guard:guard + n].view(2, 9, 13, 72)
    layer(tx, out=out)
    again = layer(tx)
    torch.cuda.synchronize()
    assert torch.equal(out, again)
    assert bool((buf[:guard] == 55.0).all()) and bool((buf[guard + n:] == 55.0).all())


def test_wide_images_take_the_transformed_domain(bd):
    assert not bd.sd_winograd_direct_supported(1, 6, 127, 72, 40)
    x, w, b = wg.make(11, 1, 6, 127, 72, 40)
    wg.check(wg.run(bd, x, w, b), oracle.conv3x3_forward(x, w, b), "127 wide")


@pytest.mark.parametrize("N,H,W,C,K", [(2, 32, 32, 320, 320), (1, 13, 10, 40, 24), (3, 7, 9, 200, 328), (1, 1, 5, 16, 16)])
def test_the_transformed_domain_itself(bd, N, H, W, C, K):
    x, w, b = wg.make(700 + H + C, N, H, W, C, K)
    layer = bd.WinogradConv3x3(torch.from_numpy(w).cuda(), torch.from_numpy(b).cuda())
    assert torch.equal(layer._filter().cpu(), torch.from_numpy(w))
    y = layer._transformed(torch.from_numpy(x).cuda(), None, None)
    rc, detail = bd.sd_winograd_query_status()
    assert rc == bd.OK, detail
    wg.check(y.cpu().numpy(), oracle.conv3x3_forward(x, w, b), str((N, H, W, C, K)))


def test_arguments(bd):
    f = bd.sd_winograd_direct_forward
    assert f(256, 256, 0, 256, 1, 8, 8, 0, 16, 0) == bd.ERR_INVALID_VALUE
    assert f(256, 256, 0, 256, 1, 8, 8, 12, 16, 0) == bd.ERR_UNSUPPORTED
    assert f(256, 256, 0, 256, 1, 8, 127, 16, 16, 0) == bd.ERR_UNSUPPORTED
    assert f(256, 256, 0, 256, 0, 8, 8, 16, 16, 0) == bd.OK
    assert f(0, 256, 0, 256, 1, 8, 8, 16, 16, 0) == bd.ERR_INVALID_VALUE
    assert f(264, 256, 0, 256, 1, 8, 8, 16, 16, 0) == bd.ERR_ALIGNMENT
    assert bd.sd_winograd_direct_pack_filter(0, 256, 16, 16, 0) == bd.ERR_INVALID_VALUE
    assert bd.sd_winograd_direct_pack_filter(256, 256, 12, 16, 0) == bd.ERR_UNSUPPORTED


def test_the_faster_of_the_two(bd):
    """Small images and few channels go to the direct kernel, the largest calls to the transformed domain."""
    assert bd.sd_winograd_direct_preferred(2, 64, 64, 320, 320) and bd.sd_winograd_direct_preferred(2, 8, 8, 1280, 1280)
    assert not bd.sd_winograd_direct_preferred(1, 6, 127, 72, 40) and not bd.sd_winograd_direct_preferred(0, 8, 8, 64, 64)
    N, H, W, C, K = 4, 24, 24, 2560, 1280
    assert not bd.sd_winograd_direct_preferred(N, H, W, C, K)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(N, H, W, C, generator=g, device="cuda").half()
    w = (torch.randn(K, 3, 3, C, generator=g, device="cuda") / (9 * C) ** 0.5).half()
    layer = bd.WinogradConv3x3(w)
    y = layer(x)
    assert torch.equal(y, layer._transformed(x, None, None))
    direct = torch.empty_like(y)
    assert bd.sd_winograd_direct_forward(x.data_ptr(), layer._packed.data_ptr(), 0, direct.data_ptr(), N, H, W, C, K,
                                         torch.cuda.current_stream().cuda_stream) == bd.OK
    assert float((y.float() - direct.float()).norm() / direct.float().norm()) < 6e-3


@pytest.mark.parametrize("N,H,W,C,K", [(1, 6, 130, 72, 40), (1, 16, 16, 64, 64)])   # through either domain
def test_a_layers_first_call_may_be_captured(bd, N, H, W, C, K):
    """What the capture leaves behind must serve an eager call although the graph has not run yet."""
    x, w, b = wg.make(90, N, H, W, C, K)
    layer = bd.WinogradConv3x3(torch.from_numpy(w).cuda(), torch.from_numpy(b).cuda())
    tx = torch.from_numpy(x).cuda()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        captured = layer(tx)
    ref = oracle.conv3x3_forward(x, w, b)
    wg.check(layer(tx).cpu().numpy(), ref, "eager call after the capture")
    g.replay()
    wg.check(captured.cpu().numpy(), ref, "replay")
    rc, detail = bd.sd_winograd_query_status()
    assert rc == bd.OK, detail


def test_the_transformed_domains_workspace_belongs_to_one_call(bd):
    """Calls on two streams at once do not share it, nor does a captured call keep memory that a larger one has given back."""
    g = torch.Generator(device="cuda").manual_seed(5)
    w = (torch.randn(64, 3, 3, 64, generator=g, device="cuda") / 24.0).half()
    layer = bd.WinogradConv3x3(w)
    small, large = (torch.randn(1, h, 200, 64, generator=g, device="cuda").half() for h in (24, 96))
    want_small, want_large = layer(small), layer(large)
    assert not bd.sd_winograd_direct_supported(*large.shape, 64)
    side = torch.cuda.Stream()
    outs = [torch.empty_like(small) for _ in range(40)]
    torch.cuda.synchronize()
    got = []
    for out in outs:
        with torch.cuda.stream(side):
            got.append((layer(large), want_large))
        got.append((layer(small), want_small))
        got.append((layer(small, out=out, stream=side.cuda_stream), want_small))
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in got)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = layer(small)
    layer(large)
    held = [torch.full((1 << 20,), 7.0, device="cuda") for _ in range(40)]   # whatever was given back is someone else's now
    captured.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(captured, want_small)
    assert all(bool((t == 7.0).all()) for t in held)


def test_a_steps_shapes_keep_their_plans(bd):
    """A step goes through its shapes one after another: each must find its plan, as a layer that runs alone does."""
    import time
    shapes = [(2, 64 >> lv, 64 >> lv, C, K) for lv, Ks in enumerate((320, 640, 1280, 1280)) for K in (Ks, 2 * Ks)
              for C in (320, 640, 1280)]
    ask = bd.sd_winograd_direct_preferred

    def us(sequence):
        best = 1e9
        for _ in range(5):
            begin = time.perf_counter()
            for s in sequence:
                ask(*s)
            best = min(best, (time.perf_counter() - begin) / len(sequence))
        return best * 1e6

    one, step = us(shapes[:1] * 2000), us(shapes * 80)
    print("a layer alone %.2f us, %d shapes in turn %.2f us" % (one, len(shapes), step))
    assert step < 1.4 * one   # (0.82 and 0.85 us; 1.56 when every call plans anew)
