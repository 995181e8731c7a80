"""The OR tree's two halves, inside comparison blocks and above them, at every way of cutting it: the tree's shape
is fixed, so the bit shares must not depend on the block size, nor on how many threads share a block. Blocks of one
word leave the whole tree to ipc_or_finalize (up to 1,250 roots a column: several batches of 32 pairs a level)."""
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu

SEEDS = (0x51EED0, 0x51EED1, 0x51EED2)


@pytest.fixture(scope="module")
def torch():
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.mark.parametrize("mode", ["lift", "plain", "const"])
@pytest.mark.parametrize("rows,Q,R", [(1, 1, 1), (33, 2, 2), (1000, 3, 31), (1025, 1, 5), (2080, 4, 17), (4129, 2, 30),
                                      (40000, 1, 3), (65536, 33, 31)])
def test_bits_do_not_depend_on_the_cut(torch, mode, rows, Q, R):
    ipc = lib()
    N, ldz = Q * R, (rows + 7) // 8 * 8
    g = torch.Generator(device="cuda").manual_seed(rows + Q)
    rand = lambda dt, b: torch.randint(-(1 << b), 1 << b, (N, ldz), generator=g, dtype=dt, device="cuda")
    zc = [rand(torch.int16, 15) for _ in range(3)]
    zm = [rand(torch.int16 if mode != "const" else torch.int32, 15 if mode != "const" else 31) for _ in range(3)]
    n = torch.arange(N)
    tags = torch.stack([torch.full((N,), 5), ((n // R) << 5) | (n % R)], 1).int().cuda()
    shares = []
    for p in (5, 4, 2, 0):
        if p == 0 and rows > 40000:
            continue
        nb = (rows + (32 << p) - 1) // (32 << p)
        roots = torch.zeros((3, N, nb), dtype=torch.int32, device="cuda")
        if mode == "lift":
            ipc.ipc_compare(zc, zm, ldz, N, rows, 0, tags, SEEDS, 16384, p, roots, nb)
        elif mode == "plain":
            ipc.ipc_compare_plain(zc, zm[0], ldz, N, rows, 0, tags, SEEDS, 16384, p, roots, nb)
        else:
            ipc.ipc_compare_liftfree(zc, None, zm, ldz, N, rows, 0, tags, SEEDS, 16384, 0, p, roots, nb)
        bits = torch.full((3, Q), 9, dtype=torch.uint8, device="cuda")
        ipc.ipc_or_finalize(roots, nb, nb, p, Q, R, tags, SEEDS, bits)
        shares.append(bits)
    torch.cuda.synchronize()
    ipc.ipc_status()
    for s in shares[1:]:
        assert torch.equal(s, shares[0])
    assert int(shares[0].max()) <= 1
