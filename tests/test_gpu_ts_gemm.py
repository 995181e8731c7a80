"""The tcgen05 ring GEMM at the edges of its shapes: every tile width it is built for and one column
on either side, ragged rows, short and long K (split over a cluster or not), the limbs at the ends of
their range, and several passes in one launch (through a context). Integer results: equal to the int32
kernel's, or to the plain dot products, without tolerance."""
import numpy as np
import pytest

import synth
from gpu_common import db_bits_device, lib, load_workload, make_ctx, plain_mask_u16, query_shares_gpu, tags_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def _case(torch, rows, cols, l, segments, fill=None):
    ipc = lib()
    n_pad, K = (cols + 127) // 128 * 128, segments * l
    g = torch.Generator(device="cpu").manual_seed(rows * 1009 + cols)

    def limbs(*shape):
        if fill is not None:
            return torch.full(shape, fill, dtype=torch.int8, device="cuda")
        return torch.randint(-128, 128, shape, dtype=torch.int8, generator=g).cuda()

    x = [limbs(rows, l) for _ in range(2 * segments)]  # lo of each segment, then hi of each
    b = [limbs(n_pad, K) for _ in range(2)]
    tags = torch.from_numpy(tags_for(3, (cols + 30) // 31, 31).view(np.int32)).cuda()
    ldz = (rows + 7) // 8 * 8
    ref = torch.zeros((cols, ldz), dtype=torch.int16, device="cuda")
    z = torch.full((cols, ldz), 77, dtype=torch.int16, device="cuda")
    b16 = [t.to(torch.float16).view(torch.int16).contiguous() for t in b]
    if segments == 2:
        ipc.ipc_ring_gemm("i32", x[0:2], x[2:4], rows, b[0], b[1], cols, n_pad, l, tags, 5, 6, 1, ref, ldz, 8)
        ipc.ipc_ring_gemm_tc(x[0:2], x[2:4], rows, b16[0], b16[1], cols, n_pad, l, tags, 5, 6, 1, z, ldz, 8)
    else:
        # K = l as the int32 kernel's two segments of l / 2
        h = l // 2
        xl, xh = ([t[:, :h].contiguous(), t[:, h:].contiguous()] for t in x)
        ipc.ipc_ring_gemm("i32", xl, xh, rows, b[0], b[1], cols, n_pad, h, tags, 5, 6, 1, ref, ldz, 8)
        ipc.ipc_ring_gemm_tc_galois(256, x[0], x[1], rows, b16[0], b16[1], cols, n_pad, l, tags, 5, 6, 1, z, ldz, 8)
    torch.cuda.synchronize()
    ipc.ipc_status()
    assert (z[:, :rows] == ref[:, :rows]).all()
    assert (z[:, rows:] == 77).all()


@pytest.mark.parametrize("cols", [1, 16, 17, 31, 32, 33, 64, 65, 96, 97, 127, 128, 129, 160, 161, 192, 193, 208, 209,
                                  223, 224, 225, 279, 416, 417, 449, 2100])
def test_every_tile_width(torch, cols):
    _case(torch, 200, cols, 1280, 2)


@pytest.mark.parametrize("cols,rows", [(31, 1), (31, 127), (31, 129), (248, 1001), (31, 20000), (208, 20000)])
def test_rows_and_splits_of_k(torch, cols, rows):
    _case(torch, rows, cols, 2560, 2)


@pytest.mark.parametrize("l,segments", [(128, 2), (256, 1), (256, 2), (512, 1), (640, 2), (1280, 1), (12800, 1), (16384, 2)])
@pytest.mark.parametrize("cols", [40, 130, 200])
def test_lengths_of_k(torch, cols, l, segments):
    _case(torch, 130, cols, l, segments)


@pytest.mark.parametrize("cols", [16, 100, 150, 208])
@pytest.mark.parametrize("fill", [-128, 127])
def test_limbs_at_their_ends(torch, cols, fill):
    """The accumulators reach their bound: 512 k of C and, with -128, 2^24 exactly. 20,000 rows keep K in one CTA."""
    _case(torch, 20000, cols, 16384, 2, fill)


@pytest.mark.parametrize("path,plain,Q", [("tc", False, 2), ("tc", True, 7), ("tcg", True, 9), ("tc", False, 40)])
def test_passes_of_a_launch(torch, path, plain, Q):
    """A context launches a chunk's GEMMs together (of equal or unequal K): the dot products and mask lengths of a
    column are the plain ones. Two chunks of 1,024 rows (the second ragged)."""
    ipc = lib()
    gal = path == "tcg"
    w = synth.Workload("passes", s=1500, Q=Q, rot_lo=-2, R=5, seed=0x7A55 + Q)
    ctx = make_ctx(w, path=path, keep=True, chunk_rows=1024, max_queries=Q, plain_mask=plain)
    try:
        load_workload(ctx, w, galois_shares=gal, plain_mask=plain)
        qc, qm = w.query_bits()
        code, mask = query_shares_gpu(w, qc, qm, galois_shares=gal)
        masks = [plain_mask_u16(qm, w.l), None, None] if plain else [mask[j] for j in range(3)]
        rid = ipc.submit_queries(ctx, [code[j] for j in range(3)], masks, Q, 1)
        got = [np.zeros(w.s, np.int16) for _ in range(2)]
        q, rho = Q - 1, 3
        ipc.fetch_distances(ctx, rid, q, rho, 0, w.s, got[0], got[1].view(np.uint16))
        bits = np.zeros(Q, np.uint8)
        ipc.fetch_match_bits(ctx, rid, bits, Q, 60000)
    finally:
        ipc.ipc_destroy(ctx)
    cb, mb = db_bits_device(w, 0, w.s)

    def values(c, m):
        s = torch.arange(64, device="cuda")
        m = ((m[:, :, None] >> s) & 1).reshape(m.shape[0], -1)[:, :w.l]
        c = ((c[:, :, None] >> s) & 1).reshape(c.shape[0], -1)[:, :w.l]
        return (m - 2 * (c & m)).double(), m.double()

    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()
    dc, dm = values(cb, mb)
    yc, ym = values(dev(qc), dev(qm))
    roll = lambda v: torch.roll(v[q].reshape(w.rows, w.cols, w.cell), w.rot_lo + rho, 1).reshape(-1)
    assert (got[0] == (dc @ roll(yc)).short().cpu().numpy()).all()
    assert (got[1] == (dm @ roll(ym)).short().cpu().numpy()).all()
