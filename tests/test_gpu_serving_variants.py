"""The serving loop with a given table of tile widths: a tuning file of its own making, rewritten to name one variant
for every width, so that what runs does not depend on what the autotuner measures."""
import json

import numpy as np
import pytest

import synth
from gpu_common import lib, load_workload, make_ctx, query_shares_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def _start(ctx, pool, cache, variant):
    """Starts the loop with the table in `cache`, written by a first start, naming `variant` in every bucket."""
    ipc = lib()
    ipc.ipc_serve_start(ctx, pool_queries=pool, tune_cache=str(cache))
    ipc.ipc_serve_stop(ctx)
    table = json.loads(cache.read_text())
    for b in table["buckets"]:
        b["variant"] = variant
    cache.write_text(json.dumps(table) + "\n")
    ipc.ipc_serve_start(ctx, pool_queries=pool, tune_cache=str(cache))
    assert json.loads(ipc.ipc_serve_tuning(ctx)) == table   # read, not measured
    return table["key"]


def test_int8_tables_keep_their_key(torch, tmp_path):
    """The int8 variants are what they were, so a table written before the tcgen05 paths had four is still read."""
    ipc = lib()
    w = synth.Workload("tab8", s=500, Q=1, planted=1, seed=0x7AB8)
    ctx = make_ctx(w, path="i8mix", chunk_rows=1024)
    try:
        load_workload(ctx, w, chunk=500)
        code, mask = (v.cpu().numpy() for v in query_shares_gpu(w))
        key = _start(ctx, 1, tmp_path / "t.json", "mma32")
        assert key.endswith("|l12800|rows1024|path2|pool256")
        rid = ipc.ipc_serve_submit(ctx, list(code), list(mask), 1)
        bits = np.zeros(1, np.uint8)
        ipc.fetch_match_bits(ctx, rid, bits, 1, 60000)
        assert bits[0] == 1 and [s > 0 for s in ipc.ipc_serve_stats(ctx)["variant_steps"]] == [False] * 3 + [True]
        ipc.ipc_serve_stop(ctx)
    finally:
        ipc.ipc_destroy(ctx)
