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


@pytest.mark.parametrize("path,rows", [("tc", 5000), ("tcg", 5000), ("tc", 20000)])
def test_every_tile_width_of_the_loop(torch, tmp_path, path, rows):
    """Every tcgen05 variant (tiles of 256, 128, 208 and 64 columns) serves the same requests: 18 queries x 31
    rotations in a pool of 768 columns, of which 208 does not divide (the last tile reaches past it), alone and
    beside others, several tiles a CTA. Equal to the shares of the same queries submitted alone."""
    ipc = lib()
    gal = path == "tcg"
    w = synth.Workload("widths", s=rows, Q=39, planted=5, seed=0x71D5 + rows)
    code, mask = query_shares_gpu(w, galois_shares=gal)
    sizes = [18, 5, 8, 3, 5]
    cuts = np.cumsum([0] + sizes)

    def run(variant):
        ctx = make_ctx(w, path=path, chunk_rows=4096 if rows < 20000 else 0, max_queries=18)
        try:
            load_workload(ctx, w, galois_shares=gal)
            if variant:
                _start(ctx, 18, tmp_path / f"{variant}.json", variant)
            shares = []
            for burst in ([0], [1, 2, 3], [4]):
                ids = []
                for i in burst:
                    part = [[v[j, cuts[i]:cuts[i + 1]].contiguous() for j in range(3)] for v in (code, mask)]
                    if variant:
                        part = [[t.cpu().numpy() for t in v] for v in part]
                        ids.append((ipc.ipc_serve_submit(ctx, *part, sizes[i]), i))
                    else:
                        ids.append((ipc.submit_queries(ctx, *part, sizes[i], 1), i))
                for rid, i in ids:
                    sh = np.zeros((3, sizes[i]), np.uint8)
                    ipc.fetch_bit_shares(ctx, rid, sh, sizes[i], 60000)
                    ipc.ipc_release(ctx, rid)
                    shares.append((rid, sh))
            steps = ipc.ipc_serve_stats(ctx)["variant_steps"] if variant else None
            return shares, steps
        finally:
            ipc.ipc_destroy(ctx)

    want, _ = run(None)
    bits = np.concatenate([s[0] ^ s[1] ^ s[2] for _, s in want])
    assert np.nonzero(bits)[0].tolist() == sorted(w.planted_set())
    for k, variant in enumerate(("tc256", "tc128", "tc208", "tc64")):
        got, steps = run(variant)
        assert [s > 0 for s in steps] == [i == k for i in range(4)]
        for (rid, sh), (rid2, sh2) in zip(got, want):
            assert rid == rid2 and (sh == sh2).all(), (variant, rid)
