"""A chunk's six GEMMs go out in one launch, in two of three or in six, by the chunk's size: a request's shares
are the same whichever it was, so they are compared with those of the same database in small chunks."""
import numpy as np
import pytest

import synth
from gpu_common import lib, load_workload, make_ctx, plain_mask_u16, query_shares_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def _shares(w, path, chunk_rows, plain):
    ipc = lib()
    ctx = make_ctx(w, path=path, chunk_rows=chunk_rows, plain_mask=plain)
    try:
        load_workload(ctx, w, galois_shares=path == "tcg", plain_mask=plain)
        qc, qm = w.query_bits()
        code, mask = query_shares_gpu(w, qc, qm, galois_shares=path == "tcg")
        masks = [plain_mask_u16(qm, w.l), None, None] if plain else [mask[j] for j in range(3)]
        rid = ipc.submit_queries(ctx, [code[j] for j in range(3)], masks, w.Q, 1)
        sh = np.zeros((3, w.Q), np.uint8)
        ipc.fetch_bit_shares(ctx, rid, sh, w.Q, 60000)
        return rid, sh
    finally:
        ipc.ipc_destroy(ctx)


# rounds of the chip a pass: 3.1 (all passes together), 6.2 and 9.6 (threes), 20.2 (each alone)
@pytest.mark.parametrize("path,plain,rows,Q", [("tc", False, 20000, 20), ("tc", False, 40000, 20),
                                               ("tc", True, 40000, 20), ("tcg", False, 30000, 40),
                                               ("tc", False, 65536, 40)])
def test_shares_do_not_depend_on_the_launches(torch, path, plain, rows, Q):
    w = synth.Workload("groups", s=rows, Q=Q, planted=3, seed=0x6A0 + rows)
    rid, big = _shares(w, path, 0, plain)
    rid2, small = _shares(w, path, 4096, plain)
    assert rid == rid2 and (big == small).all()
    bits = big[0] ^ big[1] ^ big[2]
    assert np.nonzero(bits)[0].tolist() == sorted(w.planted_set())
