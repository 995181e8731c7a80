"""Column counts whose last 256-column tile is nearly full, for which the ring GEMM keeps both operands in shared
memory (and their neighbours, for which it does not): equal to the int32 kernel's whole numbers, at both ends of the
limbs' range, at short and long K; and a context's six passes, against the same database in small chunks."""
import numpy as np
import pytest

import synth
from gpu_common import lib, load_workload, make_ctx, plain_mask_u16, query_shares_gpu, tags_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def _case(torch, rows, cols, l, segments, fill=None, same_lo=False):
    ipc = lib()
    n_pad, K = (cols + 127) // 128 * 128, segments * l
    g = torch.Generator(device="cuda").manual_seed(rows + cols)

    def limbs(*shape):
        if fill is not None:
            return torch.full(shape, fill, dtype=torch.int8, device="cuda")
        return torch.randint(-128, 128, shape, dtype=torch.int8, generator=g, device="cuda")

    x, b = [limbs(rows, l) for _ in range(2 * segments)], [limbs(n_pad, K) for _ in range(2)]
    if same_lo:
        x[1] = x[0]  # both segments' lo limbs in one plane, their hi limbs in two
    tags = torch.from_numpy(tags_for(3, (cols + 30) // 31, 31).view(np.int32)).cuda()
    ldz = (rows + 7) // 8 * 8
    ref = torch.zeros((cols, ldz), dtype=torch.int16, device="cuda")
    z = torch.full((cols, ldz), 77, dtype=torch.int16, device="cuda")
    b16 = [t.to(torch.float16).view(torch.int16).contiguous() for t in b]
    if segments == 2:
        ipc.ipc_ring_gemm("i32", x[0:2], x[2:4], rows, b[0], b[1], cols, n_pad, l, tags, 5, 6, 1, ref, ldz, 8)
        ipc.ipc_ring_gemm_tc(x[0:2], x[2:4], rows, b16[0], b16[1], cols, n_pad, l, tags, 5, 6, 1, z, ldz, 8)
    else:
        h = l // 2  # K = l as the int32 kernel's two segments of l / 2
        xl, xh = ([t[:, :h].contiguous(), t[:, h:].contiguous()] for t in x)
        ipc.ipc_ring_gemm("i32", xl, xh, rows, b[0], b[1], cols, n_pad, h, tags, 5, 6, 1, ref, ldz, 8)
        ipc.ipc_ring_gemm_tc_galois(256, x[0], x[1], rows, b16[0], b16[1], cols, n_pad, l, tags, 5, 6, 1, z, ldz, 8)
    torch.cuda.synchronize()
    ipc.ipc_status()
    assert (z[:, :rows] == ref[:, :rows]).all()
    assert (z[:, rows:] == 77).all()


@pytest.mark.parametrize("cols", [225, 240, 241, 248, 255, 256, 257, 496, 512])
@pytest.mark.parametrize("rows,l,segments", [(19456, 1280, 2), (38901, 256, 1), (9601, 512, 2)])
def test_columns_about_a_full_tile(torch, cols, rows, l, segments):
    _case(torch, rows, cols, l, segments)


@pytest.mark.parametrize("l,segments,fill", [(16384, 2, -128), (16384, 2, 127), (16384, 1, -128), (128, 2, None)])
def test_ends_of_limbs_and_k(torch, l, segments, fill):
    _case(torch, 19456, 250, l, segments, fill)


def test_planes_are_told_apart_by_both_limbs(torch):
    _case(torch, 19456, 248, 256, 2, same_lo=True)


@pytest.mark.parametrize("path,plain", [("tc", False), ("tcg", False), ("tcg", True), ("tc", True)])
def test_passes_of_a_launch(torch, path, plain):
    """30,003 rows x 248 columns: a launch of six (four) passes over two tiles of 128 or one of 256 columns; in chunks
    of 4,096 rows always the former."""
    ipc = lib()
    gal = path == "tcg"
    w = synth.Workload("wide", s=30003, Q=8, planted=3, seed=0x71DE)
    qc, qm = w.query_bits()
    got = []
    for chunk_rows in (0, 4096):
        ctx = make_ctx(w, path=path, chunk_rows=chunk_rows, plain_mask=plain)
        try:
            load_workload(ctx, w, galois_shares=gal, plain_mask=plain)
            code, mask = query_shares_gpu(w, qc, qm, galois_shares=gal)
            masks = [plain_mask_u16(qm, w.l), None, None] if plain else [mask[j] for j in range(3)]
            rid = ipc.submit_queries(ctx, [code[j] for j in range(3)], masks, w.Q, 1)
            sh = np.zeros((3, w.Q), np.uint8)
            ipc.fetch_bit_shares(ctx, rid, sh, w.Q, 60000)
            got.append((rid, sh))
        finally:
            ipc.ipc_destroy(ctx)
    assert got[0][0] == got[1][0] and (got[0][1] == got[1][1]).all()
    bits = got[0][1][0] ^ got[0][1][1] ^ got[0][1][2]
    assert np.nonzero(bits)[0].tolist() == sorted(w.planted_set())
