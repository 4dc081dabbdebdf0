"""Order of a PE's ops in a device script: what quiet and fence promise a PE that sees a later flag,
and what an op finds that touches what the op before it wrote."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_util import download, first_diff, random_heap, upload

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


@pytest.mark.parametrize("mode,cd", [(0, 1), (1, 2)])
@pytest.mark.parametrize("sig", [0, 1])
@pytest.mark.parametrize("seed", [1, 2])
@pytest.mark.parametrize("pad", [0, 125, 126, 127])
def test_ops_on_the_signal_word_follow_the_signal(sg, heapf, orc, mode, cd, sig, seed, pad):
    """put_signal, then by the same PE an AMO, a put, a get or another put_signal that reads or writes the
    signal word: the list's result, also across the end of a batch of the list."""
    npes, H = 3, 1 << 18
    rng = np.random.RandomState(seed)
    SIG, DATA, TMP = 64 * KiB, 0, 128 * KiB
    ops = [_rec(kind=W.OP_FADD, dtype=W.DT_INT64, issuer=2, pe=2, dst=8 * (i % 16), operand=3) for i in range(pad)]
    for r in range(120):
        to, w = rng.randint(0, npes), SIG + 8 * rng.randint(0, 2)
        put = dict(kind=W.OP_PUT_SIGNAL, sub=sig, issuer=0, pe=to, aux=w, operand=5 + r)
        # (a put before it turns the ops that follow to other threads)
        ops.append(_rec(kind=W.OP_PUT, issuer=0, pe=1, dst=TMP, src=DATA, n=8 * rng.randint(1, 600)))
        ops.append(_rec(**put, dst=192 * KiB, src=DATA, n=int(rng.choice([0, 8, 4096, 40000]))))
        u = r % 5
        if u == 0:
            ops.append(_rec(kind=W.OP_FADD, dtype=W.DT_INT64, issuer=0, pe=to, dst=w, operand=1 << 20))
        elif u == 1:
            ops.append(_rec(kind=W.OP_PUT, issuer=0, pe=to, dst=w, src=DATA + 8 * (r % 64), n=8))
        elif u == 2:
            ops.append(_rec(kind=W.OP_GET, issuer=0, pe=to, dst=TMP + 32 * KiB + 8 * r, src=w, n=8))
        elif u == 3:  # another put_signal that carries the word
            ops.append(_rec(kind=W.OP_PUT_SIGNAL, sub=sig, issuer=0, pe=2, aux=SIG + 32, operand=1, dst=TMP + 48 * KiB + 8 * r, src=w, n=8)
                       if to == 0 else _rec(**put, dst=w, src=DATA + 8, n=8))
        else:
            ops.append(_rec(kind=W.OP_FXOR, dtype=W.DT_INT64, issuer=0, pe=to, dst=w, operand=r))
            ops.append(_rec(kind=W.OP_GET, issuer=0, pe=to, dst=TMP + 32 * KiB + 8 * r, src=SIG, n=16))
    ops_np, dev = _dev(ops)
    h = heapf(npes, H, pe_mode=mode, cluster_dim=cd)
    init = random_heap(npes, H, seed)
    upload(h, init)
    fetched = torch.zeros(len(ops), dtype=torch.int64, device="cuda")
    sg.run_script(dev, len(ops), fetched)
    torch.cuda.synchronize()
    assert sg.get_status()[0] == 0
    ref = orc.Heap(npes, H, init)
    want = ref.run_script(ops_np)
    assert first_diff(download(h), ref.mem) is None
    amo = np.isin(ops_np["kind"], [W.OP_FADD, W.OP_FXOR])
    assert np.array_equal(fetched.cpu().numpy()[amo], np.asarray(want)[amo])


def test_agent_gives_a_silent_pe_eight_timeouts(sg, heapf):
    """A context agent whose PE shows no sign of life -- here during a short list of long puts --
    reports a timeout after eight of them and not after five."""
    H, n, count = 1 << 30, 256 << 20, 48
    h = heapf(2, H)
    ops = [_rec(kind=W.OP_PUT, issuer=0, pe=1, dst=512 << 20, src=0, n=n) for _ in range(count)]
    _, dev = _dev(ops)
    t = []
    for _ in range(2):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        sg.run_script(dev, count, None)
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b) * 1e6)
    assert sg.get_status()[0] == 0
    h.close()
    for parts, want in ((5, 0), (12, sg.ERR_TIMEOUT)):
        h = heapf(2, H, timeout_ns=int(t[1] / parts))
        sg.run_script(dev, count, None)
        torch.cuda.synchronize()
        status, detail = sg.get_status()
        assert status == want and (status == 0 or detail == -5), (parts, status, detail)
        h.close()
