"""The tcgen05 ring GEMM over Z_2^32 at the edges of its shapes: tile widths and one column on either side, ragged
rows, short and long K (split over a cluster or not), and the limbs at the ends of their range, against 64-bit integer
products mod 2^32 (equal seeds make the zero share vanish; one case has unequal ones)."""
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


def _run(torch, x, b, rows, cols, l, segments, seeds=(5, 5)):
    """x, b: four int8 limb tensors each, [rows][K] and [n_pad][K] on the device -> z [cols][ldz] int32."""
    ipc = lib()
    xs = [t[:, s * l:(s + 1) * l].contiguous() for s in range(segments) for t in x]
    b16 = [t.to(torch.float16).view(torch.int16).contiguous() for t in b]
    tags = torch.from_numpy(tags_for(3, (cols + 30) // 31, 31).view(np.int32)).cuda()
    ldz = (rows + 3) // 4 * 4
    z = torch.full((cols, ldz), 77, dtype=torch.int32, device="cuda")
    ipc.ipc_ring_gemm_tc32(segments, xs, rows, b16, cols, b[0].shape[0], l, tags, seeds[0], seeds[1], 1, z, ldz, 8)
    torch.cuda.synchronize()
    ipc.ipc_status()
    assert (z[:, rows:] == 77).all()
    return z[:, :rows]


def _case(torch, rows, cols, l, segments):
    n_pad, K = (cols + 127) // 128 * 128, segments * l
    g = torch.Generator(device="cpu").manual_seed(rows * 1009 + cols)
    limbs = lambda n: [torch.randint(-128, 128, (n, K), dtype=torch.int8, generator=g) for _ in range(4)]
    x, b = limbs(rows), limbs(n_pad)
    value = lambda v: sum(t.long() << (8 * i) for i, t in enumerate(v))
    want = (value(b)[:cols] @ value(x).T).int()
    got = _run(torch, [t.cuda() for t in x], [t.cuda() for t in b], rows, cols, l, segments)
    assert torch.equal(got.cpu(), want)


@pytest.mark.parametrize("cols", [1, 16, 17, 31, 48, 80, 81, 96, 97, 160, 161, 192, 193, 300])
def test_tile_widths(torch, cols):
    _case(torch, 130, cols, 640, 2)


@pytest.mark.parametrize("rows,cols", [(1, 31), (127, 96), (129, 80), (1001, 33)])
def test_rows(torch, rows, cols):
    _case(torch, rows, cols, 384, 2)


@pytest.mark.parametrize("l,segments", [(128, 2), (256, 1), (256, 2), (512, 1), (1280, 1), (2048, 2)])
@pytest.mark.parametrize("cols", [40, 90])
def test_lengths_of_k(torch, cols, l, segments):
    _case(torch, 70, cols, l, segments)


@pytest.mark.parametrize("cols", [31, 80, 96])
@pytest.mark.parametrize("fill", [-128, 127])
@pytest.mark.parametrize("rows", [100, 20000])
def test_limbs_at_their_ends(torch, rows, cols, fill):
    """The accumulators reach their bound of 2^24; 20,000 rows keep K in one CTA, 100 split it."""
    l, n_pad = 16384, 128
    x = [torch.full((rows, 2 * l), fill, dtype=torch.int8, device="cuda")] * 4
    b = [torch.full((n_pad, 2 * l), fill, dtype=torch.int8, device="cuda")] * 4
    v = sum(fill << (8 * i) for i in range(4))
    want = np.uint32(2 * l * v * v % (1 << 32)).astype(np.int32)
    assert (_run(torch, x, b, rows, cols, l, 2) == int(want)).all()


def test_zero_shares_do_not_depend_on_the_split(torch):
    """F(seed_own) - F(seed_prev) of every cell: a run with unequal seeds less one with equal seeds is the same for a
    few rows (K split over a cluster) and for many (unsplit)."""
    diffs = []
    for rows in (64, 20000):
        z = [_run(torch, [torch.zeros((rows, 512), dtype=torch.int8, device="cuda")] * 4,
                  [torch.ones((128, 512), dtype=torch.int8, device="cuda")] * 4, rows, 62, 256, 2, s)
             for s in ((5, 6), (5, 5))]
        diffs.append((z[0] - z[1])[:, :64])
        assert (z[1] == 0).all()
    assert torch.equal(diffs[0], diffs[1])
