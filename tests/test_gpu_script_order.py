"""Order of a PE's ops in a device script: what quiet and fence promise a PE that sees a later flag,
and what an op finds that touches what the op before it wrote."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_util import random_heap, upload

pytestmark = pytest.mark.gpu
KiB = 1 << 10


def _rec(**kw):
    r = np.zeros((), dtype=W.OP_DTYPE)
    r["issuer"] = -1
    for k, v in kw.items():
        r[k] = v
    return r


def _dev(ops):
    ops = np.array(ops, dtype=W.OP_DTYPE)
    return ops, torch.from_numpy(ops.view(np.uint8).copy()).cuda()


@pytest.mark.parametrize("mode,cd", [(0, 1), (1, 2)])
@pytest.mark.parametrize("order", [W.OP_QUIET, W.OP_FENCE])
@pytest.mark.parametrize("flag", ["amo", "put8", "put64"])
@pytest.mark.parametrize("n,rounds", [(8, 40), (4 * KiB, 40), (48 * KiB, 24)])
def test_flag_after_quiet_or_fence_follows_the_data(sg, heapf, mode, cd, order, flag, n, rounds):
    """PE 0 puts a payload that stays below the bulk engine's threshold, quiets or fences, and raises a
    flag that any of its threads may issue; PE 1 waits for the flag and copies the payload.  The
    other PEs keep the memory busy meanwhile."""
    npes, H = 24, 8 << 20
    h = heapf(npes, H, pe_mode=mode, cluster_dim=cd)
    init = random_heap(npes, H, n + rounds)
    m = init.reshape(npes, H)
    SRC, FLAGS, DST, FLAG, ACK, LOG, NOISE = 0, 128 * KiB, 256 * KiB, 512 * KiB, 520 * KiB, 1 << 20, 4 << 20
    m[:, FLAGS:FLAGS + 64 * rounds] = 0
    for r in range(rounds):  # the flag's value in the last word of 64 bytes
        m[0, FLAGS + 64 * r + 56:FLAGS + 64 * r + 64].view(np.int64)[0] = r + 1
    m[:, FLAG:FLAG + 64] = 0
    m[:, ACK:ACK + 8] = 0
    word = FLAG + 56
    ops = []
    for r in range(rounds):
        src = SRC + 16 * r if n > 8 else SRC + 8 * r
        ops.append(_rec(kind=W.OP_PUT, issuer=0, pe=1, dst=DST, src=src, n=n))
        ops.append(_rec(kind=order, issuer=0))
        if flag == "amo":
            ops.append(_rec(kind=W.OP_FADD, dtype=W.DT_INT64, issuer=0, pe=1, dst=word, operand=1))
        elif flag == "put8":
            ops.append(_rec(kind=W.OP_PUT, issuer=0, pe=1, dst=word, src=FLAGS + 64 * r + 56, n=8))
        else:
            ops.append(_rec(kind=W.OP_PUT, issuer=0, pe=1, dst=FLAG, src=FLAGS + 64 * r, n=64))
        ops.append(_rec(kind=W.OP_WAIT_UNTIL, issuer=1, sub=W.CMP_EQ, dst=word, operand=r + 1))
        ops.append(_rec(kind=W.OP_PUT, issuer=1, pe=1, dst=LOG + r * n, src=DST, n=n))
        ops.append(_rec(kind=order, issuer=1))
        ops.append(_rec(kind=W.OP_FADD, dtype=W.DT_INT64, issuer=1, pe=0, dst=ACK, operand=1))
        ops.append(_rec(kind=W.OP_WAIT_UNTIL, issuer=0, sub=W.CMP_EQ, dst=ACK, operand=r + 1))
        for p in range(2, npes):
            ops.append(_rec(kind=W.OP_PUT, issuer=p, pe=1 if p % 2 else p, dst=NOISE + (p // 2) * 64 * KiB, src=NOISE, n=64 * KiB - 8))
    upload(h, init)
    fetched = torch.zeros(len(ops), dtype=torch.int64, device="cuda")
    for _ in range(3):
        h.partitions()[:, FLAG:FLAG + 64] = 0
        h.partitions()[:, ACK:ACK + 8] = 0
        h.partitions()[1, LOG:LOG + rounds * n] = 0
        ops_np, dev = _dev(ops)
        sg.run_script(dev, len(ops_np), fetched)
        torch.cuda.synchronize()
        assert sg.get_status()[0] == 0
        got = h.partitions()[1, LOG:LOG + rounds * n].cpu().numpy().reshape(rounds, n)
        for r in range(rounds):
            src = SRC + 16 * r if n > 8 else SRC + 8 * r
            assert np.array_equal(got[r], m[0, src:src + n]), r
