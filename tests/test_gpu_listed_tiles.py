"""The tcgen05 ring GEMM over a list of column tiles, the form that the serving loop replays: CTAs that
compute one tile after another (the sums of a tile pass through the shared memory that the next tile's
query copies fill)."""
import numpy as np
import pytest

from gpu_common import lib, tags_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.mark.parametrize("tile_cols,chosen", [(128, [0, 2, 3, 6, 7]), (256, [0, 2, 3])])
@pytest.mark.parametrize("l,segments", [(128, 2), (256, 1), (640, 2)])
def test_tiles_one_after_another(torch, tile_cols, chosen, l, segments):
    """157 row tiles (the last ragged) x 5 or 6 listed tiles of 128 columns: five to seven tiles a CTA, and K of a
    few stages, so that a tile's copies follow at once on the one before. Whole numbers: equal to the int32
    kernel's; columns that are not listed keep what they held."""
    ipc = lib()
    rows, cols, n_pad, K = 20003, 1000, 1024, segments * l
    g = torch.Generator(device="cpu").manual_seed(l + segments)
    limbs = lambda *shape: torch.randint(-128, 128, shape, dtype=torch.int8, generator=g).cuda()
    x, b = [limbs(rows, l) for _ in range(2 * segments)], [limbs(n_pad, K) for _ in range(2)]
    b16 = [t.to(torch.float16).view(torch.int16).contiguous() for t in b]
    tags = torch.from_numpy(tags_for(3, 33, 31).view(np.int32)).cuda()
    ldz = 20008
    ref = torch.zeros((cols, ldz), dtype=torch.int16, device="cuda")
    z = torch.full((cols, ldz), 77, dtype=torch.int16, device="cuda")
    tiles = torch.tensor(chosen, dtype=torch.int32, device="cuda")
    count = torch.tensor([len(chosen)], dtype=torch.int32, device="cuda")
    if segments == 2:
        ipc.ipc_ring_gemm("i32", x[0:2], x[2:4], rows, b[0], b[1], cols, n_pad, l, tags, 5, 6, 1, ref, ldz, 8)
        ipc.ipc_ring_gemm_tc_tiles(tile_cols, x[0:2], x[2:4], rows, b16[0], b16[1], cols, n_pad, l, tags, 5, 6, 1, z,
                                   ldz, 8, tiles, count)
    else:
        # K = l as the int32 kernel's two segments of l / 2
        h = l // 2
        xl, xh = ([t[:, :h].contiguous(), t[:, h:].contiguous()] for t in x)
        ipc.ipc_ring_gemm("i32", xl, xh, rows, b[0], b[1], cols, n_pad, h, tags, 5, 6, 1, ref, ldz, 8)
        ipc.ipc_ring_gemm_tc_galois(tile_cols, x[0], x[1], rows, b16[0], b16[1], cols, n_pad, l, tags, 5, 6, 1, z, ldz,
                                    8, tiles, count)
    torch.cuda.synchronize()
    ipc.ipc_status()
    for t in range(-(-cols // tile_cols)):
        at = slice(t * tile_cols, min(cols, (t + 1) * tile_cols))
        if t in chosen:
            assert (z[at, :rows] == ref[at, :rows]).all(), t
            assert (z[at, rows:] == 77).all(), t
        else:
            assert (z[at] == 77).all(), t
