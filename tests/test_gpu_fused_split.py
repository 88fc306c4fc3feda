"""The variants of the single-pass kernel.  The lone query tile's: two, three and four parts, score buffers that are no multiple of
the parts, a K/V ring as deep as the buffers, against the oracle (tolerances of test_gpu_parity.py)."""
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


# head dims at the edges of the parts (64 -> 4, 72..96 -> 3, 104..160 -> 2); key tiles from one per launch to several times
# round the buffers and the ring (3 at d = 160), the last one ragged or not
@pytest.mark.parametrize("d", [8, 40, 64, 72, 80, 96, 104, 128, 136, 160])
@pytest.mark.parametrize("Nk", [129, 192, 257, 320, 400, 1000])
def test_parts_buffers_and_ring(bd, d, Nk):
    a = bd.Attention()
    q, k, v = parity.rand_qkv(d + Nk, 1, 3, 150, Nk, d, qmult=2.0)
    scale = float(np.float32(d ** -0.5))
    ref, _, _ = oracle.forward(q, k, v, scale)
    parity.check(parity.run(a, bd, bd.MODE_AUTO, q, k, v, scale), ref, v, what="d=%d Nk=%d" % (d, Nk))
    a.close()


@pytest.mark.parametrize("d,Nk", [(40, 1024), (80, 1024), (160, 1024), (136, 130), (160, 192), (160, 256)])   # (d > 128: a ring of three stages)
def test_parts_that_re_anchor_at_every_key_tile(bd, d, Nk):
    """Scores that rise along the keys: the rescale of a part's accumulator waits for its own last product."""
    a = bd.Attention()
    q, k, v = parity.rand_qkv(d, 1, 4, 128, Nk, d)
    k = (k.astype(np.float32) * np.repeat(np.geomspace(0.1, 12.0, 16), 64)[:1024:1024 // Nk][:Nk, None].astype(np.float32)).astype(np.float16)
    scale = float(np.float32(d ** -0.5))
    ref, _, _ = oracle.forward(q, k, v, scale)
    for _ in range(5):
        parity.check(parity.run(a, bd, bd.MODE_FUSED, q, k, v, scale), ref, v, what="rising d=%d" % d)
    a.close()


@pytest.mark.parametrize("tiles,shares", [(1, 0), (2, 0), (3, 0), (4, 0), (2, 1), (4, 1)])
@pytest.mark.parametrize("Nk", [65, 320, 385, 1024])   # fewer key tiles than score buffers, as many, one more, several rounds
def test_tiles_that_re_anchor_at_every_key_tile(bd, tiles, shares, Nk):
    """Whole units of one to four tiles: the rescale of an accumulator is all that waits for the products before it."""
    a = bd.Attention(bd.MODE_FUSED, options=bd.Options(fused_tiles=tiles, fused_split=1, fused_shares=shares))
    q, k, v = parity.rand_qkv(tiles + Nk, 1, 3, 600, Nk, 40)
    k = (k.astype(np.float32) * np.geomspace(0.1, 12.0, Nk, dtype=np.float32)[None, None, :, None]).astype(np.float16)
    scale = float(np.float32(40 ** -0.5))
    ref, _, _ = oracle.forward(q, k, v, scale)
    for _ in range(5):
        parity.check(parity.run(a, bd, bd.MODE_FUSED, q, k, v, scale), ref, v, what="tiles=%d Nk=%d" % (tiles, Nk))
    a.close()


@pytest.mark.parametrize("tiles,d", [(2, 72), (3, 80), (1, 88), (2, 88), (1, 128), (2, 128), (2, 136), (2, 160)])
@pytest.mark.parametrize("Nk", [65, 193, 257, 449])   # around the score buffers (2 to 4) and the K/V ring (3 to 6)
def test_whole_units_of_wide_heads(bd, tiles, d, Nk):
    """80 < d <= 128 takes every phase of the products' barriers, the others only where a row is re-anchored, here at every key tile."""
    a = bd.Attention(bd.MODE_FUSED, options=bd.Options(fused_tiles=tiles, fused_split=1))
    q, k, v = parity.rand_qkv(d + Nk, 1, 3, 300, Nk, d)
    scale = float(np.float32(d ** -0.5))
    for grow in (1.0, 12.0):
        kk = (k.astype(np.float32) * np.geomspace(0.1 if grow > 1 else 1.0, grow, Nk, dtype=np.float32)[None, None, :, None]).astype(np.float16)
        ref, _, _ = oracle.forward(q, kk, v, scale)
        parity.check(parity.run(a, bd, bd.MODE_FUSED, q, kk, v, scale), ref, v, what="tiles=%d d=%d Nk=%d" % (tiles, d, Nk))
    a.close()
