"""The edges of the dispatch rules of the group normalisation and GEGLU kernels, against the oracle (tolerances of
test_gpu_groupnorm.py and test_gpu_geglu.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import test_gpu_geglu as geglu  # noqa: E402
import test_gpu_groupnorm as gn  # noqa: E402


@pytest.fixture(scope="module")
def bd():
    from paper_2304_11267_b200 import binding
    from paper_2304_11267_b200 import build
    build.build()
    binding.load()
    return binding


# (channels per group, values per channel, groups), in values of the dtype; a 16-byte piece is 8 (fp16) or 4 (fp32) of them
@pytest.mark.parametrize("dtype", [np.float16, np.float32], ids=["f16", "f32"])
@pytest.mark.parametrize("pieces_times", [
    (1024, 0), (1024, 1),            # one block / the same with a remainder
    (6144, 0), (6144, 1),            # clusters of four, without and with a remainder
    (12288, 1), (24576, 0), (24576, 1), (49152, 0), (49152, 1),   # clusters of four, of eight, streaming form
])
def test_groupnorm_group_sizes_at_the_edges_of_a_plan(bd, dtype, pieces_times):
    pieces, more = pieces_times
    vec = 16 // np.dtype(dtype).itemsize
    x, gamma, beta = gn.make(pieces + more, (2, 2, (pieces + more) * vec), dtype, scale=1.3, shift=-0.7)
    gn.check(gn.run(bd, x, 2, 1e-5, gamma, beta), x, 2, 1e-5, gamma, beta, what=str(pieces_times))


# (groups, 16-byte pieces of each): blocks per group and threads per block, on either side of every line of the plan on 148 SMs
@pytest.mark.parametrize("dtype", [np.float16, np.float32], ids=["f16", "f32"])
@pytest.mark.parametrize("groups,pieces", [(33, 5119), (33, 5120), (34, 5120), (74, 2559), (74, 2560), (75, 2560), (74, 10240), (74, 10241),
                                           (33, 20480), (33, 20481), (148, 2561), (148, 4097), (148, 6144), (148, 6145), (149, 4097), (149, 6145),
                                           (33, 8192), (33, 8196), (74, 4096), (74, 4098), (149, 2048), (149, 2049), (149, 3072), (149, 3073), (149, 4096),
                                           (149, 5120), (149, 5121), (222, 5121), (223, 5121), (75, 8193), (111, 8193), (112, 8193), (149, 6146), (222, 6147)])
@pytest.mark.parametrize("odd", [0, 3])   # values more than whole pieces: ragged groups
def test_groupnorm_blocks_of_a_group(bd, dtype, groups, pieces, odd):
    vec = 16 // np.dtype(dtype).itemsize
    x, gamma, beta = gn.make(groups + pieces, (1, groups, pieces * vec - odd), dtype, scale=0.9, shift=0.5)
    gn.check(gn.run(bd, x, groups, 1e-5, gamma, beta), x, groups, 1e-5, gamma, beta, what=str((groups, pieces, odd)))


# (groups, pieces): threads and registers of a block where blocks outnumber the SMs: up to four an SM and more, every count of pieces a thread
@pytest.mark.parametrize("dtype", [np.float16, np.float32], ids=["f16", "f32"])
@pytest.mark.parametrize("groups,pieces", [(592, 512), (593, 512), (592, 513), (593, 1024), (300, 1025), (300, 1536), (149, 1537), (300, 2048), (300, 2049)])
@pytest.mark.parametrize("odd", [0, 3])
def test_groupnorm_small_blocks_in_many_waves(bd, dtype, groups, pieces, odd):
    vec = 16 // np.dtype(dtype).itemsize
    x, gamma, beta = gn.make(groups + pieces, (1, groups, pieces * vec - odd), dtype, scale=1.1, shift=-0.2)
    gn.check(gn.run(bd, x, groups, 1e-5, gamma, beta), x, groups, 1e-5, gamma, beta, what=str((groups, pieces, odd)))


# ragged and whole groups on either side of the 16 MB from which blocks ask ahead
@pytest.mark.parametrize("dtype", [np.float16, np.float32], ids=["f16", "f32"])
@pytest.mark.parametrize("groups", [511, 512])
@pytest.mark.parametrize("odd", [0, 3])
def test_groupnorm_asking_ahead(bd, dtype, groups, odd):
    per_group = (32 << 10) // np.dtype(dtype).itemsize + (8 if odd else 0)
    x, gamma, beta = gn.make(groups, (1, groups, per_group - odd), dtype, scale=1.2, shift=0.3)
    gn.check(gn.run(bd, x, groups, 1e-5, gamma, beta), x, groups, 1e-5, gamma, beta, what=str((groups, odd)))


@pytest.mark.parametrize("dtype", [np.float16, np.float32], ids=["f16", "f32"])
@pytest.mark.parametrize("C,HW,G", [(12, 9, 3), (6, 5, 1), (40, 31, 8), (10, 5525, 1), (20, 4757, 2), (64, 37, 32), (1030, 9, 1),
                                    (2, 24577, 1), (2, 8, 2), (4, 4, 1),
                                    (300, 16, 1), (300, 13, 1), (1024, 8, 1), (1024, 9, 1)])   # more channels in a group than threads
def test_groupnorm_ragged_channels(bd, dtype, C, HW, G):
    x, gamma, beta = gn.make(C + HW, (3, C, HW), dtype, scale=0.8, shift=5.0)
    gn.check(gn.run(bd, x, G, 1e-5, gamma, beta), x, G, 1e-5, gamma, beta, what=str((C, HW, G)))


@pytest.mark.parametrize("dtype", [np.float16, np.float32], ids=["f16", "f32"])
def test_groupnorm_of_an_outlier_in_front(bd, dtype):
    """The statistics are summed about a thread's first value: a group whose first values lie far from the rest."""
    x, gamma, beta = gn.make(5, (1, 4, 4096), dtype, scale=0.01, shift=0.0)
    x[:, :, :8] = dtype(300.0)
    gn.check(gn.run(bd, x, 4, 1e-5, gamma, beta), x, 4, 1e-5, gamma, beta, what="outlier")


@pytest.mark.parametrize("dtype", [np.float16, np.float32], ids=["f16", "f32"])
@pytest.mark.parametrize("rows,C", [(1, 8), (255, 8), (257, 8), (148 * 16, 2048), (148 * 16 - 1, 2048), (4737, 1288)])
def test_geglu_sizes_at_the_edges(bd, dtype, rows, C):
    x = geglu.make(rows + C, rows, C, dtype)
    geglu.check(bd.geglu(torch.from_numpy(x).cuda()).cpu().numpy(), x, what=str((rows, C)))


@pytest.mark.parametrize("dtype", [torch.float16, torch.float32], ids=["f16", "f32"])
def test_inputs_written_by_the_kernel_before(bd, dtype):
    """Blocks ask for their input in the L2 while the kernel that writes it still runs: what they read is what it wrote."""
    g = torch.Generator(device="cuda").manual_seed(3)
    xs = [torch.randn(4096, 8192, generator=g, device="cuda").to(dtype) for _ in range(3)]
    gn_x = torch.randn(12, 128, 64, 64, generator=g, device="cuda").to(dtype)
    want, got = [], []
    for x in xs:
        a = bd.geglu(x)
        torch.cuda.synchronize()
        want.append(bd.geglu(a))
        torch.cuda.synchronize()
    b = bd.groupnorm(gn_x, 32)
    torch.cuda.synchronize()
    want.append(bd.groupnorm(b, 32))
    torch.cuda.synchronize()
    a, b = torch.empty_like(a), torch.empty_like(b)   # rewritten by every call
    for x in xs:
        got.append(bd.geglu(bd.geglu(x, out=a)))
    got.append(bd.groupnorm(bd.groupnorm(gn_x, 32, out=b), 32))
    assert all(torch.equal(w, o) for w, o in zip(want, got))


@pytest.mark.parametrize("dtype", [np.float16, np.float32], ids=["f16", "f32"])
@pytest.mark.parametrize("more", [-1, 0])
def test_geglu_input_marked_to_go_first(bd, dtype, more):
    """Either side of the size from which the input's lines are marked: 16 MB of output."""
    rows = (16 << 20) // (1024 * np.dtype(dtype).itemsize) + more
    x = geglu.make(rows, rows, 1024, dtype)
    geglu.check(bd.geglu(torch.from_numpy(x).cuda()).cpu().numpy(), x, what=str(rows))


@pytest.mark.parametrize("dtype", [torch.float16, torch.float32], ids=["f16", "f32"])
@pytest.mark.parametrize("share", [8, 2])
def test_geglu_either_side_of_the_lines_of_the_l2(bd, dtype, share):
    """An output of an eighth (of half) of the L2, a row less and a row more: the same bits as by parts, which are far below the lines."""
    C = 1024
    line = torch.cuda.get_device_properties(0).L2_cache_size // share // (C * torch.finfo(dtype).bits // 8)
    g = torch.Generator(device="cuda").manual_seed(share)
    x = torch.randn(line + 1, 2 * C, generator=g, device="cuda").to(dtype)
    parts = torch.cat([bd.geglu(p.contiguous()) for p in x.split(1024)])
    for rows in (line - 1, line, line + 1):
        assert torch.equal(bd.geglu(x[:rows]), parts[:rows]), rows
