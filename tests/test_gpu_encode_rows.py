"""ipc_encode_share at row lengths that share a block, fill one or take several, and with outputs that allow
16-byte stores or only 8-byte ones: equal to the oracle's components."""
import numpy as np
import pytest

import oracle
from gpu_common import dev_u64, lib, u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("l", [4, 8, 12, 60, 64, 128, 132, 512, 1024, 1028, 2040, 2048, 2056, 4104, 12800])
@pytest.mark.parametrize("n,skew", [(1, 0), (67, 0), (258, 0), (67, 4)])
def test_row_lengths(l, n, skew):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(l + n)
    code, mask = (rng.integers(0, 1 << 63, (n, (l + 63) // 64), dtype=np.uint64) * np.uint64(2) +
                  rng.integers(0, 2, (n, (l + 63) // 64), dtype=np.uint64) for _ in range(2))
    want = oracle.encode_share(code, mask, l, 0xC0DE + l, 1, idx0=3)
    size = 3 * n * l
    bufs = [torch.full((size + 2 * skew,), 77, dtype=torch.int16, device="cuda") for _ in range(2)]
    outs = [b[skew:skew + size] for b in bufs]
    lib().ipc_encode_share(dev_u64(code), dev_u64(mask), n, l, 0xC0DE + l, 1, 3, outs[0], outs[1])
    torch.cuda.synchronize()
    for buf, out, ref in zip(bufs, outs, want):
        assert (u16(out).reshape(3, n, l) == ref).all()
        assert (buf[:skew] == 77).all() and (buf[skew + size:] == 77).all()
