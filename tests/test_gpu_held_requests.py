"""Requests held back while the device is busy with other work: submitting does not wait for that work, a
fetch that may not wait says so, and a full serving queue refuses. The work is a kernel on the caller's
stream (or the context's) that spins for about half a second and ends by itself."""
import os
import subprocess
import sys
import time

import numpy as np
import pytest

import synth
from gpu_common import lib, lift_shares, load_workload, make_ctx, plain_mask_u16, query_shares_gpu, torch_mod

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SPIN = 1_000_000_000  # clock cycles, about 0.5 s
FORMS = {"tc": dict(path="tc"), "tcg": dict(path="tcg"), "plain": dict(path="tc", plain_mask=True),
         "const": dict(path="tc", lift="const"), "none": dict(path="tc", lift="none"),
         "fused": dict(path="tc", fused=True), "i8mix": dict(path="i8mix"), "i8mma": dict(path="i8mma"),
         "i32": dict(path="i32")}


@pytest.fixture(scope="module")
def torch():
    t = torch_mod()
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def _held_request(form):
    """A new context's first request behind a spin on its input stream."""
    torch, ipc, cfg = torch_mod(), lib(), FORMS[form]
    w = synth.Workload("held", s=300, Q=2, planted=1, seed=0xFA14)
    gal, plain, lift = cfg["path"] == "tcg", cfg.get("plain_mask", False), cfg.get("lift")
    qc, qm = w.query_bits()
    ctx = make_ctx(w, **cfg)
    try:
        load_workload(ctx, w, chunk=300, galois_shares=gal, plain_mask=plain, lift=lift)
        code, mask = lift_shares(qc, qm, w.l, w.q_share_seed, 1, lift=lift) if lift else query_shares_gpu(
            w, qc, qm, galois_shares=gal)
        masks = [plain_mask_u16(qm, w.l), None, None] if plain else [mask[j] for j in range(3)]
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            torch.cuda._sleep(SPIN)
        ipc.ipc_set_input_stream(ctx, side.cuda_stream)
        rid = ipc.submit_queries(ctx, [code[j] for j in range(3)], masks, w.Q, 1)
        bits = np.zeros(w.Q, np.uint8)
        rc = 0
        try:
            ipc.fetch_match_bits(ctx, rid, bits, w.Q, 0)
        except ipc.IpcError as e:
            rc = e.rc
        assert not side.query(), "submit or fetch waited for the caller's stream"
        assert rc == ipc.IPC_ETIMEOUT
        ipc.fetch_match_bits(ctx, rid, bits, w.Q, -1)
        assert side.query() and bits.tolist() == [int(q in w.planted_set()) for q in range(w.Q)]
    finally:
        ipc.ipc_destroy(ctx)


@pytest.mark.parametrize("form", FORMS)
def test_first_submit_of_a_context_does_not_wait(torch, form):
    _held_request(form)


def test_first_submits_of_a_process_do_not_wait(torch):
    """The same in a fresh process, where each form launches its kernels for the first time."""
    code = "import test_gpu_held_requests as t\nfor form in t.FORMS: t._held_request(form)"
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


def test_full_serving_queue_refuses_until_a_request_is_admitted(torch):
    """One query slot, one waiting request, and the serving stream held. The loop keeps two steps in flight, so at
    most three requests are admitted before it waits; with one waiting the queue is full, and a further request is
    refused. Released, every accepted request has its bits."""
    ipc = lib()
    w = synth.Workload("held2", s=2000, Q=6, planted=2, seed=0xFA15)
    ctx = make_ctx(w, path="tc", max_queries=1)
    try:
        load_workload(ctx, w)
        code, mask = query_shares_gpu(w)
        hc, hm = (np.ascontiguousarray(v.cpu().numpy()) for v in (code, mask))
        ipc.ipc_serve_start(ctx, pool_queries=1, max_pending=1, variant=0)
        stream = torch.cuda.ExternalStream(ipc.ipc_ctx_stream(ctx))
        with torch.cuda.stream(stream):
            torch.cuda._sleep(SPIN)
        rids, refused, until = [], 0, time.perf_counter() + 0.3
        while len(rids) < 5 and time.perf_counter() < until:
            q = len(rids)
            try:
                rids.append(ipc.ipc_serve_submit(ctx, [hc[j, q:q + 1] for j in range(3)],
                                                 [hm[j, q:q + 1] for j in range(3)], 1))
            except ipc.IpcError as e:
                assert e.rc == ipc.IPC_EAGAIN
                refused += 1
        assert 1 <= len(rids) <= 4 and refused > 0
        for q, rid in enumerate(rids):
            b = np.zeros(1, np.uint8)
            ipc.fetch_match_bits(ctx, rid, b, 1, 60000)
            assert b[0] == int(q in w.planted_set())
        ipc.ipc_serve_stop(ctx)
    finally:
        ipc.ipc_destroy(ctx)


def test_a_request_with_free_slots_does_not_fill_the_queue(torch):
    """One query slot and one waiting request, the loop idle: of two requests submitted at once the first takes the
    slot, so the second may wait, however late the loop's thread wakes up."""
    ipc = lib()
    w = synth.Workload("held3", s=300, Q=1, planted=1, seed=0xFA16)
    ctx = make_ctx(w, path="tc", max_queries=1)
    try:
        load_workload(ctx, w, chunk=300)
        code, mask = (v.cpu().numpy() for v in query_shares_gpu(w))
        ipc.ipc_serve_start(ctx, pool_queries=1, max_pending=1, variant=0)
        for _ in range(400):
            rids = [ipc.ipc_serve_submit(ctx, list(code), list(mask), 1) for _ in range(2)]
            for rid in rids:
                b = np.zeros(1, np.uint8)
                ipc.fetch_match_bits(ctx, rid, b, 1, 60000)
                assert b[0] == 1
        assert ipc.ipc_serve_stats(ctx)["completed"] == 800
        ipc.ipc_serve_stop(ctx)
    finally:
        ipc.ipc_destroy(ctx)
