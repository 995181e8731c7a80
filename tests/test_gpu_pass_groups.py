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


@pytest.mark.parametrize("path,rows,pool", [("tc", 4096, 40), ("tc", 40000, 40), ("tcg", 40000, 60)])
def test_serving_steps_of_every_width(torch, path, rows, pool):
    """A wide pool with few and with many columns in use: steps of one launch and of several, whichever of them a
    request shares, give the shares of the same queries submitted alone in small chunks."""
    ipc = lib()
    gal = path == "tcg"
    sizes = [1, 24, 2, pool - 24]
    w = synth.Workload("steps", s=rows, Q=sum(sizes), planted=4, seed=0x57E9 + rows)
    qc, qm = w.query_bits()
    code, mask = query_shares_gpu(w, qc, qm, galois_shares=gal)
    cuts = np.cumsum([0] + sizes)
    runs = {}
    for served in (True, False):
        ctx = make_ctx(w, path=path, chunk_rows=0 if served else 4096, max_queries=max(sizes))
        try:
            load_workload(ctx, w, galois_shares=gal)
            if served:
                ipc.ipc_serve_start(ctx, pool_queries=pool)
            ids = []
            for a, b in zip(cuts, cuts[1:]):
                part = [[v[j, a:b].contiguous() for j in range(3)] for v in (code, mask)]
                if served:
                    ids.append(ipc.ipc_serve_submit(ctx, *[[t.cpu().numpy() for t in v] for v in part], b - a))
                else:
                    ids.append(ipc.submit_queries(ctx, *part, b - a, 1))
            runs[served] = ids, []
            for rid, n in zip(ids, sizes):
                sh = np.zeros((3, n), np.uint8)
                ipc.fetch_bit_shares(ctx, rid, sh, n, 60000)
                runs[served][1].append(sh)
        finally:
            ipc.ipc_destroy(ctx)
    assert runs[True][0] == runs[False][0]
    got, want = (np.concatenate(runs[k][1], 1) for k in (True, False))
    assert (got == want).all()
    assert np.nonzero(got[0] ^ got[1] ^ got[2])[0].tolist() == sorted(w.planted_set())
