"""Serving engine: slots that change hands while workers still claim from the request before."""
import time

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inflight,count", [(1, 300), (2, 1200), (7, 1500)])
def test_tiles_of_a_reused_slot_run_once(sg, heapf, inflight, count):
    """One-tile AMOs and puts of several tiles take the same few slots in turn, with every worker after
    each of them: no tile of a request is run by a worker that claimed from the slot's last one."""
    npes, page, big = 4, 64 << 10, 9 * (64 << 10) + 48
    arena = 16 * page
    H = arena + (1 << 20) + 4096
    h = heapf(npes, H)
    h.partitions().zero_()
    for p in range(npes):
        h.view(h.sym(arena + 4096), p, torch.int32, big // 4).copy_(torch.arange(p + 1, p + 1 + big // 4, dtype=torch.int32))
    cfg = sg.ServerCfg(page_bytes=page, max_inflight=inflight, ring_slots=256, arena_offset=0, arena_bytes=arena, amo_offset=arena,
                       amo_words=8)
    q = np.zeros(count, sg.REQ_DTYPE)
    for i in range(count):
        r = q[i]
        if i % 2:
            r["kind"], r["dtype"], r["operand"] = W.OP_FADD, W.DT_INT64, 1
        else:
            r["kind"], r["pe"], r["issuer"], r["src"] = W.OP_PUT, i // 2 % npes, i // 6 % npes, arena + 4096
            r["n"] = (big, 16, 3 * (64 << 10))[i // 2 % 3]
    rec = torch.zeros(sg.COMPLETION_DTYPE.itemsize, dtype=torch.uint8).pin_memory()
    want = {}
    for i in range(0, count, 2):
        key = (int(q[i]["pe"]), int(q[i]["issuer"]), int(q[i]["n"]))
        if key not in want:
            sg.request_run(q[i:i + 1], cfg, rec.data_ptr())
            torch.cuda.synchronize()
            want[key] = rec.numpy().view(sg.COMPLETION_DTYPE)[0]["result"]
    srv = sg.Server(cfg, torch.cuda.Stream())
    recs, got, sent = np.zeros(count, sg.COMPLETION_DTYPE), 0, 0
    end = time.monotonic() + 30
    try:
        while got < count and time.monotonic() < end:
            while sent < count and srv.submit(sg.Req.from_buffer_copy(q[sent].tobytes())) is not None:
                sent += 1
            got += srv.poll(recs[got:])
    finally:
        srv.stop()
    assert got == count and not recs["status"].any()
    assert np.array_equal(np.sort(recs["ticket"]), np.arange(count))
    res = recs["result"][np.argsort(recs["ticket"], kind="stable")]
    assert sorted(res[1::2].tolist()) == list(range(count // 2))
    assert h.view(h.sym(arena), 0, torch.int64, 1).item() == count // 2
    for i in range(0, count, 2):
        assert res[i] == want[(int(q[i]["pe"]), int(q[i]["issuer"]), int(q[i]["n"]))], i
