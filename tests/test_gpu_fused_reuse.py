"""The fused chunk step with items that follow one another at once: K of a few stages, so that the query copies of
the next pass or tile fill the shared memory right after an epilogue and a comparison phase used it."""
import numpy as np
import pytest

import synth
from gpu_common import lib, load_workload, make_ctx, query_shares_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["tc", "tcg"])
@pytest.mark.parametrize("cols", [4, 20])
def test_short_codes_many_tiles_equal_unfused(path, cols):
    """20,003 rows (157 row tiles, the last ragged) x 310 columns (two column tiles): two or three tiles of six
    passes a CTA, K = 256 to 2,560. Every share equals the unfused context's."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ipc = lib()
    w = synth.Workload("reuse", s=20003, Q=10, planted=0, seed=0x4E5E, cols=cols)
    gal = path == "tcg"
    got = []
    for fused in (True, False):
        ctx = make_ctx(w, path=path, fused=fused, chunk_rows=20480, keep=True)
        try:
            load_workload(ctx, w, galois_shares=gal)
            code, mask = query_shares_gpu(w, galois_shares=gal)
            rid = ipc.submit_queries(ctx, [code[j] for j in range(3)], [mask[j] for j in range(3)], w.Q, 1)
            sh = np.zeros((3, w.Q), np.uint8)
            ipc.fetch_bit_shares(ctx, rid, sh, w.Q, 60000)
            got.append((rid, sh, ipc.fetch_transcript_hash(ctx, rid)))
        finally:
            ipc.ipc_destroy(ctx)
    assert got[0][0] == got[1][0] and got[0][2] == got[1][2] and (got[0][1] == got[1][1]).all()
