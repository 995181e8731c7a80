"""The Z_2^32 ring GEMM where the column tiles of a launch differ in width (16-column units dealt out unevenly), K in
one CTA or split over a cluster, against products of limbs that are exact in 64-bit floats, combined mod 2^32."""
import numpy as np
import pytest

from gpu_common import lib, tags_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [97, 110, 177, 290, 496, 992])
@pytest.mark.parametrize("rows,l,segments", [(1000, 1280, 2), (20000, 256, 1)])
def test_tiles_of_two_widths(cols, rows, l, segments):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ipc = lib()
    n_pad, K = (cols + 127) // 128 * 128, segments * l
    g = torch.Generator(device="cuda").manual_seed(rows + cols)
    limbs = lambda n: [torch.randint(-128, 128, (n, K), dtype=torch.int8, generator=g, device="cuda") for _ in range(4)]
    x, y = limbs(rows), limbs(n_pad)
    want = torch.zeros((cols, rows), dtype=torch.int64, device="cuda")
    for a in range(4):
        for b in range(4 - a):
            want += (y[b][:cols].double() @ x[a].double().T).long() << (8 * (a + b))
    xs = [t[:, s * l:(s + 1) * l].contiguous() for s in range(segments) for t in x]
    b16 = [t.to(torch.float16).view(torch.int16).contiguous() for t in y]
    tags = torch.from_numpy(tags_for(3, (cols + 30) // 31, 31).view(np.int32)).cuda()
    z = torch.full((cols, rows + 4), 77, dtype=torch.int32, device="cuda")
    ipc.ipc_ring_gemm_tc32(segments, xs, rows, b16, cols, n_pad, l, tags, 5, 5, 1, z, rows + 4, 0)
    torch.cuda.synchronize()
    ipc.ipc_status()
    assert torch.equal(z[:, :rows], want.int()) and (z[:, rows:] == 77).all()
