"""The work a program has this library do, as cases that can be timed and compared.

listed() is the fixed set, draw(rng) gives more cases of the same ranges.  prepare(case,
seed) makes what a program holds before the call (symmetric objects filled with the
inputs, teams, op lists, plans), run(state) makes the call(s) through the public binding,
work(case) counts the bytes the call cannot do without, and exact(case, seed) gives the
floating-point results in 64 bits from plain torch.

The library holds one symmetric heap per process.  States of one heap shape share it
(each allocates its own symmetric objects); a case that needs another shape gets a new
heap once no state of the old one is left.
"""
import math
import time

import numpy as np
import torch

import paper_2607_08006_gb300 as sg

KIB, MIB = 1 << 10, 1 << 20
CAP_BYTES = 800_000_000  # of a drawn case's work

DT = {"int32": (sg.INT32, torch.int32, 4), "int64": (sg.INT64, torch.int64, 8), "float": (sg.FLOAT, torch.float32, 4)}
OPS = {"sum": sg.SUM, "max": sg.MAX, "min": sg.MIN}
FMT = {"bf16": (sg.FMT_BF16, 2), "e4m3": (sg.FMT_E4M3, 1)}
OP_REC = np.dtype([("kind", "<u4"), ("dtype", "u1"), ("sub", "u1"), ("team", "<u2"), ("pe", "<i4"), ("issuer", "<i4"),
                   ("dst", "<u8"), ("src", "<u8"), ("n", "<u8"), ("operand", "<i8"), ("cond", "<i8"), ("aux", "<u8")])
K_PUT, K_GET, K_PUT_NBI, K_ADD, K_CAS, K_XOR, K_BARRIER, K_QUIET, K_BCAST, K_A2A, K_REDUCE = 1, 2, 3, 5, 6, 7, 10, 11, 13, 15, 16


# ------------------------------------------------------------------------------ cases
def listed():
    return [
        # one small message with its arrival flag: the unit of a producer / consumer exchange
        {"name": "put_signal_8B", "kind": "rma", "op": "put_signal", "n": 8, "dshift": 0, "sshift": 0},
        # fetching a remote buffer whose length is no multiple of anything (a packed record block)
        {"name": "get_3MB_ragged", "kind": "rma", "op": "get", "n": 3_000_003, "dshift": 0, "sshift": 0},
        # gathering int32 shards of a 4 Mi-element vector over 48 PEs: the shard length is what the division leaves
        {"name": "fcollect_48x87381_i32", "kind": "fcollect", "P": 48, "n": 4 * 87_381},
        # the transpose step of a distributed matrix / expert dispatch: 64 KiB per pair, 64 PEs
        {"name": "alltoall_64x64KiB", "kind": "alltoall", "P": 64, "n": 64 * KIB},
        # a small global sum (counters, convergence test) over all 64 PEs: latency
        {"name": "reduce_i64_sum_1Ki", "kind": "reduce", "dtype": "int64", "op": "sum", "P": 64, "n": 1024},
        # a gradient-like fp32 sum over 24 PEs, a million values and three
        {"name": "reduce_f32_sum_1M_ragged", "kind": "reduce", "dtype": "float", "op": "sum", "P": 24, "n": 1_000_003},
        # the same kind of sum with 8-bit payloads: quantise, then the dequantising all-reduce
        {"name": "quant_sum_e4m3_1Mi", "kind": "quant", "fmt": "e4m3", "P": 32, "n": 1 << 20},
        # a device-initiated program: 4 PEs, puts / gets of 8 B-64 KiB, atomics, reductions and broadcasts
        {"name": "script_4pe_2000", "kind": "script", "npes": 4, "nops": 2000, "max_words": 8192},
        # many teams' uneven sums (fp32, bf16, E4M3 payloads, int64) in one captured launch
        {"name": "batch_64_teams", "kind": "batch", "npes": 128, "teams": 64, "n_lo": 256, "n_hi": 256 * KIB, "mix_seed": 7},
        # random read-modify-writes on a table spread over 64 PEs, old values fetched
        {"name": "amo_uniform_4Mi", "kind": "amo", "npes": 64, "words_log2": 24, "nops": (1 << 22) - 5, "dist": "unique", "flags": 0},
        # a periodic stencil on 8 x 8 PEs of 256 x 256 points, 20 sweeps with halo exchange
        {"name": "halo_8x8_256_20", "kind": "halo", "px": 8, "py": 8, "nx": 256, "ny": 256, "iters": 20},
        # a burst of mixed requests through the serving engine, from start to stop
        {"name": "serve_burst_1024", "kind": "serve", "npes": 64, "arena": 8 * MIB, "count": 1024},
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _ragged(rng, n, unit):
    """Half of the sizes as they come, half rounded to a multiple of `unit`."""
    return n if rng.random() < 0.5 else max(unit, n // unit * unit)


def draw(rng):
    kind = rng.choice(["rma", "rma", "fcollect", "alltoall", "reduce", "reduce", "quant", "script", "batch", "amo", "halo", "serve"])
    if kind == "rma":
        n = _ragged(rng, _log_int(rng, 1, 16 * MIB), 8)
        shift = rng.random() < 0.25  # a buffer that starts anywhere in its object
        return {"kind": kind, "op": rng.choice(["put", "get", "put_signal"]), "n": n, "dshift": rng.randrange(64) if shift else 0,
                "sshift": rng.randrange(64) if shift else 0}
    if kind == "fcollect":
        P = _log_int(rng, 2, 64)
        total = _log_int(rng, KIB, 8 * MIB)
        n = rng.choice([4, 8]) * _ragged(rng, -(-total // P), 4)
        if rng.random() < 0.5:  # the other replicating collective
            return {"kind": "broadcast", "P": P, "n": min(_log_int(rng, KIB, 64 * MIB) // 4 * 4, CAP_BYTES // (P + 1) // 16 * 16)}
        return {"kind": kind, "P": P, "n": min(n, CAP_BYTES // (P * P + P) // 4 * 4)}
    if kind == "alltoall":
        P = _log_int(rng, 2, 64)
        n = 4 * _ragged(rng, _log_int(rng, 16, 256 * KIB), 4)
        return {"kind": kind, "P": P, "n": min(n, CAP_BYTES // (2 * P * P) // 4 * 4)}
    if kind == "reduce":
        P, dtype = _log_int(rng, 2, 64), rng.choice(["int32", "int64", "float", "float"])
        n = _ragged(rng, _log_int(rng, 256, 4 * MIB), 4)
        return {"kind": kind, "dtype": dtype, "op": rng.choice(["sum", "sum", "max", "min"]), "P": P,
                "n": min(n, CAP_BYTES // (2 * P * DT[dtype][2]))}
    if kind == "quant":
        P = _log_int(rng, 2, 64)
        return {"kind": kind, "fmt": rng.choice(["bf16", "e4m3"]), "P": P,
                "n": min(_ragged(rng, _log_int(rng, KIB, 4 * MIB), 128), CAP_BYTES // (11 * P))}
    if kind == "script":
        if rng.random() < 0.3:  # bulk puts in a ring of two-CTA PEs
            return {"kind": "ring", "npes": 64, "n": min(8 * _log_int(rng, 1, MIB), 6 * MIB)}
        return {"kind": kind, "npes": rng.choice([2, 3, 4, 6, 8]), "nops": _log_int(rng, 100, 2000), "max_words": _log_int(rng, 16, 8192)}
    if kind == "batch":
        n_hi = _log_int(rng, 4 * KIB, 256 * KIB)
        return {"kind": kind, "npes": rng.choice([16, 64, 128]), "teams": _log_int(rng, 8, 64), "n_lo": 256, "n_hi": n_hi,
                "mix_seed": rng.randrange(1 << 30)}
    if kind == "amo":
        words = rng.randint(18, 26)
        zipf = rng.random() < 0.5
        return {"kind": kind, "npes": 1 << rng.randint(4, 10), "words_log2": words, "nops": _log_int(rng, 1 << 14, 1 << min(22, words)) - rng.randrange(8),
                "dist": "zipf" if zipf else "unique", "flags": rng.choice([sg.AMO_AGGREGATE, sg.AMO_COMBINE_BLOCK]) if zipf else 0}
    if kind == "halo":
        px, py = rng.randint(1, 12), rng.randint(1, 12)
        return {"kind": kind, "px": px, "py": py, "nx": 4 * _log_int(rng, 8, 128), "ny": _log_int(rng, 16, 512), "iters": rng.randint(1, 24)}
    return {"kind": "serve", "npes": rng.choice([32, 64]), "arena": rng.choice([4, 8]) * MIB, "count": _log_int(rng, 64, 1024)}


# ------------------------------------------------------------------------------ the heap
class _Shared:
    heap, key, states = None, None, 0


def _align(n):
    return (int(n) + 255) & ~255


class State:
    """One case's symmetric objects on the shared heap; gives them back when it goes."""

    def __init__(self, npes, need, pe_mode=sg.PE_MODE_CTA, cluster_dim=1):
        H = 4 * _align(need) + MIB  # room for the states a program alternates between
        key = (npes, H, pe_mode, cluster_dim)
        if _Shared.key != key:
            if _Shared.states:
                raise MemoryError("out of memory: states of another heap shape are still held")
            if _Shared.heap is not None:
                _Shared.heap.close()
            _Shared.heap = _Shared.key = None
            _Shared.heap = sg.Heap(npes, H, pe_mode=pe_mode, cluster_dim=cluster_dim)
            _Shared.key = key
        self.heap, self.syms, self.teams, self.batches = _Shared.heap, [], [], []
        _Shared.states += 1
        self.counted = True

    def malloc(self, nbytes):
        try:
            s = self.heap.malloc(int(nbytes))
        except sg.ShmemgError as e:
            raise MemoryError("out of memory: %s" % e)
        self.syms.append(s)
        return s

    def team(self, P, npes):
        """P of the heap's PEs: all of them, or every second / every one from PE 1 or 0 on."""
        if P == npes:
            return sg.TEAM_WORLD, 0, 1
        start, stride = (1, 2) if 2 * P <= npes else (npes - P, 1)
        t = sg.team_split_strided(sg.TEAM_WORLD, start, stride, P)
        self.teams.append(t)
        return t, start, stride

    def rows(self, sym, dtype, count, start=0, stride=1, P=None, byte0=0):
        """[P, count] view of the members' copies of a symmetric object."""
        es = torch.empty((), dtype=dtype).element_size()
        P = self.heap.npes if P is None else P
        lo = sym.offset + byte0
        v = self.heap.partitions()[start:start + (P - 1) * stride + 1:stride, lo:lo + count * es]
        return v if dtype == torch.uint8 else v.view(dtype)

    def __del__(self):
        if getattr(self, "counted", False):
            self.counted = False
            _Shared.states -= 1
            if self.heap.live:
                for b in self.batches:
                    b.destroy()
                for t in self.teams:
                    sg.team_destroy(t)
                for s in self.syms:
                    self.heap.free(s)


def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + salt) & 0x7FFFFFFFFFFF)
    return g


def _bytes(seed, *shape):
    return torch.randint(0, 256, shape, dtype=torch.uint8, device="cuda", generator=_gen(seed))


def _values(dtype, seed, P, n):
    if dtype == "float":
        return torch.randn(P, n, device="cuda", generator=_gen(seed))
    return torch.randint(-MIB, MIB + 1, (P, n), dtype=DT[dtype][1], device="cuda", generator=_gen(seed))


def run(state):
    return state.go()


# ------------------------------------------------------------------------------ host RMA
NPES = 64  # the PEs of the host-issued cases


def _prepare_rma(c, seed):
    n, ds, ss = c["n"], c["dshift"], c["sshift"]
    st = State(NPES, 2 * _align(n + 64) + 256)
    dst, src, sig = st.malloc(n + 64), st.malloc(n + 64), st.malloc(8)
    a, b = 5, 42  # the issuing PE and its peer
    put = c["op"] != "get"
    sp, dp = (a, b) if put else (b, a)
    st.heap.view(src, sp, torch.uint8).copy_(_bytes(seed, n + 64))
    st.heap.view(dst, dp, torch.uint8).zero_()
    st.heap.view(sig, b, torch.int64).zero_()
    out = {"dst": st.heap.view(dst, dp, torch.uint8)}
    d, s = dst.ptr + ds, src.ptr + ss
    if c["op"] == "put_signal":
        out["sig"] = st.heap.view(sig, b, torch.int64)

        def go():
            sg.putmem_signal(d, s, n, sig, 1, sg.SIGNAL_ADD, b, a)
            return out
    elif put:
        def go():
            sg.putmem(d, s, n, b, a)
            return out
    else:
        def go():
            sg.getmem(d, s, n, b, a)
            return out
    st.go = go
    return st


# ------------------------------------------------------------------------------ collectives
def _prepare_move(c, seed):
    P, n, kind = c["P"], c["n"], c["kind"]
    nsrc = n * P if kind == "alltoall" else n
    ndst = n if kind == "broadcast" else n * P
    st = State(NPES, _align(nsrc) + _align(ndst))
    team, start, stride = st.team(P, NPES)
    dst, src = st.malloc(ndst), st.malloc(nsrc)
    st.rows(src, torch.uint8, nsrc, start, stride, P).copy_(_bytes(seed, P, nsrc))
    wide = torch.int32 if ndst % 4 == 0 else torch.uint8
    out = {"dst": st.rows(dst, wide, ndst // (4 if wide == torch.int32 else 1), start, stride, P)}
    out["dst"].zero_()
    if kind == "broadcast":
        root = P // 2

        def go():
            sg.broadcastmem(team, dst, src, n, root)
            return out
    elif kind == "fcollect":
        def go():
            sg.fcollectmem(team, dst, src, n)
            return out
    else:
        def go():
            sg.alltoallmem(team, dst, src, n)
            return out
    st.go = go
    return st


def _prepare_reduce(c, seed):
    P, n = c["P"], c["n"]
    dt, tdt, es = DT[c["dtype"]]
    op = OPS[c["op"]]
    st = State(NPES, 2 * _align(n * es))
    team, start, stride = st.team(P, NPES)
    dst, src = st.malloc(n * es), st.malloc(n * es)
    st.rows(src, tdt, n, start, stride, P).copy_(_values(c["dtype"], seed, P, n))
    out = {"dst": st.rows(dst, tdt, n, start, stride, P)}
    out["dst"].zero_()

    def go():
        sg.reduce(team, dst, src, n, dt, op)
        return out
    st.go = go
    return st


def _exact_reduce(c, seed):
    if c["dtype"] != "float":
        return None
    x = _values("float", seed, c["P"], c["n"]).double()
    y = x.sum(0) if c["op"] == "sum" else x.amax(0) if c["op"] == "max" else x.amin(0)
    return {"dst": y.expand(c["P"], c["n"])}


def _prepare_quant(c, seed):
    P, n = c["P"], c["n"]
    fmt, qs = FMT[c["fmt"]]
    nb = -(-n // 128)
    st = State(NPES, 2 * _align(4 * n) + _align(qs * n) + _align(4 * nb))
    team, start, stride = st.team(P, NPES)
    src, dst, q, sc = st.malloc(4 * n), st.malloc(4 * n), st.malloc(qs * n), st.malloc(4 * nb)
    st.rows(src, torch.float32, n, start, stride, P).copy_(_values("float", seed, P, n))
    out = {"codes": st.rows(q, torch.int16 if qs == 2 else torch.uint8, n, start, stride, P),
           "scales": st.rows(sc, torch.float32, nb, start, stride, P), "sum": st.rows(dst, torch.float32, n, start, stride, P)}

    def go():
        sg.quantize(team, q, sc, src, fmt, n)
        sg.qsum_reduce(team, dst, q, sc, fmt, n)
        return out
    st.go = go
    return st


def _exact_quant(c, seed):
    P, n = c["P"], c["n"]
    nb = -(-n // 128)
    R = 448.0 if c["fmt"] == "e4m3" else 1.0
    y = torch.zeros(n, dtype=torch.float64, device="cuda")
    scales = []
    for row in _values("float", seed, P, n):
        x = torch.nn.functional.pad(row, (0, nb * 128 - n)).view(nb, 128)
        amax = x.abs().amax(1)
        s = torch.where(amax == 0, torch.ones_like(amax), amax / torch.full_like(amax, R))  # (a tensor: a true division)
        scales.append(torch.where(amax == 0, torch.ones_like(amax, dtype=torch.float64), amax.double() / R))
        code = (x / s[:, None]).to(torch.float8_e4m3fn if c["fmt"] == "e4m3" else torch.bfloat16)
        y += (code.double() * s.double()[:, None]).view(-1)[:n]
    return {"codes": None, "scales": torch.stack(scales), "sum": y.expand(P, n)}


# ------------------------------------------------------------------------------ device scripts
def _script_zones(npes):
    """Word offsets of a script's zones in a partition: read-only sources, landing slots
    (one per putting PE), the PE's own get buffer, results of collectives, atomics."""
    z, at = {}, 0
    for name, words in (("src", 16384), ("land", npes * 8192), ("got", 8192), ("sum", 4096), ("bcast", 2048), ("amo", 4096)):
        z[name] = at
        at += words
    return z, at


def _script_ops(c, seed, base):
    """An op list in which PEs never race: puts go to the putting PE's own slot, gets to its
    own buffer, every atomic word belongs to one issuer, sources are never written."""
    npes, nops = c["npes"], c["nops"]
    z, _ = _script_zones(npes)
    r = np.random.RandomState(seed & 0x7FFFFFFF)
    ops = np.zeros(nops, OP_REC)
    u, v = r.rand(nops), r.rand(nops)
    words = np.floor(np.exp(r.rand(nops) * math.log(c["max_words"]))).astype(np.int64)
    src = (r.rand(nops) * (16384 - words)).astype(np.int64)
    dst = (r.rand(nops) * (8192 - words + 1)).astype(np.int64)
    pe, issuer = r.randint(0, npes, nops), r.randint(0, npes, nops)
    amo = r.randint(0, 4096 // npes, nops) * npes + issuer
    operand = r.randint(1, 1 << 20, nops)
    csrc = r.randint(0, 16384 - 4096 + 1, nops) // 2 * 2
    for i in range(nops):
        o = ops[i]
        if i % 500 == 499:
            o["kind"], o["issuer"] = K_BARRIER, -1
        elif u[i] < 0.60:
            o["kind"], o["pe"], o["issuer"], o["n"] = K_PUT if u[i] < 0.30 else K_GET, pe[i], issuer[i], 8 * words[i]
            o["src"] = 8 * (z["src"] + src[i])
            o["dst"] = 8 * (z["land"] + issuer[i] * 8192 + dst[i]) if u[i] < 0.30 else 8 * (z["got"] + dst[i])
        elif u[i] < 0.85:
            o["kind"], o["dtype"], o["pe"], o["issuer"] = K_ADD if u[i] < 0.75 else K_CAS, sg.INT64, pe[i], issuer[i]
            o["dst"], o["operand"] = 8 * (z["amo"] + amo[i]), operand[i]
            o["cond"] = amo[i] if v[i] < 0.5 else operand[i] + 1
        elif u[i] < 0.925:
            o["kind"], o["dtype"], o["sub"], o["team"], o["issuer"], o["n"] = K_REDUCE, sg.INT64, sg.SUM, sg.TEAM_WORLD, -1, 4096
            o["src"], o["dst"] = 8 * (z["src"] + csrc[i]), 8 * z["sum"]
        else:
            o["kind"], o["team"], o["pe"], o["issuer"], o["n"] = K_BCAST, sg.TEAM_WORLD, pe[i], -1, 16 * KIB
            o["src"], o["dst"] = 8 * (z["src"] + csrc[i]), 8 * z["bcast"]
    moves = (ops["kind"] != K_BARRIER)
    ops["dst"][moves] += base
    ops["src"][moves] += base
    return ops


def _prepare_script(c, seed):
    npes, nops = c["npes"], c["nops"]
    z, total = _script_zones(npes)
    st = State(npes, 8 * total)
    area = st.malloc(8 * total)
    a = st.rows(area, torch.int64, total)
    a.zero_()
    a[:, z["src"]:z["land"]] = torch.randint(-MIB, MIB + 1, (npes, 16384), dtype=torch.int64, device="cuda", generator=_gen(seed))
    a[:, z["amo"]:] = torch.arange(4096, dtype=torch.int64, device="cuda")
    ops = torch.from_numpy(_script_ops(c, seed, area.offset).view(np.uint8).copy()).cuda()
    fetched = torch.zeros(nops, dtype=torch.int64, device="cuda")

    def go():
        sg.run_script(ops, nops, fetched)
        return {"heap": a, "fetched": fetched}
    st.go = go
    return st


def _script_bytes(c):
    """Bytes the ops read and write, from the op list of seed 0 (the list's shape is the same for every seed)."""
    ops = _script_ops(c, 0, 0)
    k, n = ops["kind"], ops["n"].astype(np.int64)
    P = c["npes"]
    return float(2 * n[(k == K_PUT) | (k == K_GET)].sum() + 24 * ((k == K_ADD) | (k == K_CAS)).sum()
                 + 2 * P * 8 * n[k == K_REDUCE].sum() + (P + 1) * n[k == K_BCAST].sum() + 64 * len(ops))


def _prepare_ring(c, seed):
    npes, n = c["npes"], c["n"]
    st = State(npes, 2 * _align(n), sg.PE_MODE_CLUSTER, 2)
    dst, src = st.malloc(n), st.malloc(n)
    st.rows(src, torch.uint8, n).copy_(_bytes(seed, npes, n))
    out = {"dst": st.rows(dst, torch.int64, n // 8)}
    out["dst"].zero_()
    ops = np.zeros(npes + 1, OP_REC)
    for p in range(npes):
        o = ops[p]
        o["kind"], o["pe"], o["issuer"], o["dst"], o["src"], o["n"] = K_PUT_NBI, (p + 1) % npes, p, dst.offset, src.offset, n
    ops[npes]["kind"], ops[npes]["issuer"] = K_QUIET, -1
    dops = torch.from_numpy(ops.view(np.uint8).copy()).cuda()
    fetched = torch.zeros(npes + 1, dtype=torch.int64, device="cuda")

    def go():
        sg.run_script(dops, npes + 1, fetched)
        return out
    st.go = go
    return st


# ------------------------------------------------------------------------------ batched teams
def _batch_teams(c):
    """(kind, start, P, n, element offset in its kind's area) of each team, and the areas' lengths."""
    r = np.random.RandomState(c["mix_seed"] & 0x7FFFFFFF)
    teams, at = [], {"f32": 0, "bf16": 0, "e4m3": 0, "i64": 0}
    for t in range(c["teams"]):
        kind = ("f32", "bf16", "e4m3", "i64")[t % 4]
        P = int(round(math.exp(r.uniform(math.log(2), math.log(c["npes"])))))
        start = int(r.randint(0, c["npes"] - P + 1))
        n = int(round(math.exp(r.uniform(math.log(c["n_lo"]), math.log(c["n_hi"])))))
        teams.append((kind, start, P, n, at[kind]))
        at[kind] += -(-n // 128) * 128
    return teams, at


def _batch_inputs(c, seed, at):
    w = c["npes"]
    f = torch.randn(w, at["f32"], device="cuda", generator=_gen(seed, 1))
    b = torch.randn(w, at["bf16"], device="cuda", generator=_gen(seed, 2)).to(torch.bfloat16)
    e = (torch.randn(w, at["e4m3"], device="cuda", generator=_gen(seed, 3)) * 100).clamp(-448, 448).to(torch.float8_e4m3fn)
    i = torch.randint(-MIB, MIB + 1, (w, at["i64"]), dtype=torch.int64, device="cuda", generator=_gen(seed, 4))
    bs = torch.rand(w, at["bf16"] // 128, device="cuda", generator=_gen(seed, 5)) + 0.5
    es = (torch.rand(w, at["e4m3"] // 128, device="cuda", generator=_gen(seed, 6)) + 0.5) / 100
    return f, b, e, i, bs, es


def _prepare_batch(c, seed):
    teams, at = _batch_teams(c)
    nf = at["f32"] + at["bf16"] + at["e4m3"]  # one output area for the float teams: fp32, bf16, E4M3 teams' parts
    sizes = {"f": 4 * at["f32"], "b": 2 * at["bf16"], "e": at["e4m3"], "i": 8 * at["i64"], "bs": at["bf16"] // 32,
             "es": at["e4m3"] // 32, "of": 4 * nf, "oi": 8 * at["i64"]}
    st = State(c["npes"], sum(_align(v) + 256 for v in sizes.values()))
    s = {k: st.malloc(v) for k, v in sizes.items()}
    f, b, e, i, bs, es = _batch_inputs(c, seed, at)
    for key, x in (("f", f), ("b", b.view(torch.int16)), ("e", e.view(torch.uint8)), ("i", i), ("bs", bs), ("es", es)):
        st.rows(s[key], x.dtype, x.shape[1]).copy_(x)
    out = {"float": st.rows(s["of"], torch.float32, nf), "int64": st.rows(s["oi"], torch.int64, at["i64"])}
    out["float"].zero_()
    out["int64"].zero_()
    off = {"f32": 0, "bf16": at["f32"], "e4m3": at["f32"] + at["bf16"]}
    descs = []
    for kind, start, P, n, o in teams:
        if kind == "i64":
            descs.append(sg.CollDesc(start, P, sg.INT64, -1, n, s["oi"].ptr + 8 * o, s["i"].ptr + 8 * o, None))
        elif kind == "f32":
            descs.append(sg.CollDesc(start, P, sg.FLOAT, -1, n, s["of"].ptr + 4 * o, s["f"].ptr + 4 * o, None))
        else:
            fmt, qs = FMT[kind]
            q, sc = (s["b"], s["bs"]) if kind == "bf16" else (s["e"], s["es"])
            descs.append(sg.CollDesc(start, P, sg.FLOAT, fmt, n, s["of"].ptr + 4 * (off[kind] + o), q.ptr + qs * o, sc.ptr + o // 32))
    plan = sg.Batch(descs)
    st.batches.append(plan)

    def go():
        plan.launch()
        return out
    st.go = go
    return st


def _exact_batch(c, seed):
    teams, at = _batch_teams(c)
    f, b, e, _, bs, es = _batch_inputs(c, seed, at)
    off = {"f32": 0, "bf16": at["f32"], "e4m3": at["f32"] + at["bf16"]}
    y = torch.zeros(c["npes"], at["f32"] + at["bf16"] + at["e4m3"], dtype=torch.float64, device="cuda")
    for kind, start, P, n, o in teams:
        if kind == "i64":
            continue
        x = (f if kind == "f32" else b if kind == "bf16" else e)[start:start + P, o:o + n].double()
        if kind != "f32":
            sc = (bs if kind == "bf16" else es)[start:start + P, o // 128:o // 128 + -(-n // 128)].double()
            x = x * sc.repeat_interleave(128, 1)[:, :n]
        y[start:start + P, off[kind] + o:off[kind] + o + n] = x.sum(0)
    return {"float": y, "int64": None}


# ------------------------------------------------------------------------------ atomics
def _s64(v):
    return v - (1 << 64) if v >> 63 else v


def _shr(z, k):  # logical shift right of int64 bit patterns
    return (z >> k) & ((1 << (64 - k)) - 1)


def _mix64(x):
    """splitmix64's first output for the states x (int64 bit patterns)."""
    z = x + _s64(0x9E3779B97F4A7C15)
    z = (z ^ _shr(z, 30)) * _s64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _s64(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _prepare_amo(c, seed):
    npes, words = c["npes"], 1 << c["words_log2"]
    wpp, nops, unique = words // npes, c["nops"], c["dist"] == "unique"
    st = State(npes, 8 * wpp)
    table = st.malloc(8 * wpp)
    tseed, oseed = 2 * int(seed) + 1, 3 * int(seed) + 7
    rows = st.rows(table, torch.int64, wpp)
    rows.copy_(_mix64(torch.arange(words, dtype=torch.int64, device="cuda") ^ tseed).view(npes, wpp))
    i = torch.arange(nops, dtype=torch.int64, device="cuda")
    if unique:  # every word at most once (a bijection of the index), so every fetched value is determined
        w = (i * 0x2545F491 + int(seed)) & (words - 1)
        w = (w ^ (w >> (c["words_log2"] // 2))) * 0x9E3779B1 & (words - 1)
        w = w ^ (w >> (c["words_log2"] // 2))
        code = torch.tensor([0, 0, 1, 2], device="cuda")[_shr(_mix64(i ^ (int(seed) + 99)), 62)]  # half adds, a quarter each of the others
    else:  # Zipf(1.1) ranks spread over the table; a word is always added to or always xor-ed, so the table is determined
        u = torch.rand(nops, dtype=torch.float64, device="cuda", generator=_gen(seed))
        rank = ((1 - u * (1 - float(words) ** -0.1)) ** -10.0).floor().long().clamp(1, words) - 1
        w = (rank * 0x9E3779B1 + int(seed)) & (words - 1)
        code = 2 * (_mix64(w) & 1)
    ops = (w | (code << 27)).to(torch.int32).contiguous()
    fetched = torch.zeros(nops, dtype=torch.int64, device="cuda") if unique else None
    out = {"table": rows}
    if unique:
        out["fetched"] = fetched

    def go():
        sg.amo_stream(table, wpp, ops, nops, oseed, tseed, fetched, c["flags"])
        return out
    st.go = go
    return st


# ------------------------------------------------------------------------------ halo exchange
def _prepare_halo(c, seed):
    px, py, nx, ny, iters = c["px"], c["py"], c["nx"], c["ny"], c["iters"]
    npes, hs = px * py, sg.halo_stride(nx, ny)
    st = State(npes, _align(8 * nx * ny) + _align(8 * hs) + 256)
    tiles, halos, sigs = st.malloc(8 * nx * ny), st.malloc(8 * hs), st.malloc(32)
    t = st.rows(tiles, torch.float32, 2 * nx * ny).view(npes, 2, ny, nx)
    t[:, 0].copy_(torch.randn(npes, ny, nx, device="cuda", generator=_gen(seed)))
    t[:, 1].zero_()
    st.rows(sigs, torch.int64, 4).zero_()
    out = {"tile": t[:, iters & 1]}

    def go():
        sg.halo_jacobi(tiles, halos, sigs, px, py, nx, ny, iters)
        return out
    st.go = go
    return st


def _exact_halo(c, seed):
    px, py, nx, ny = c["px"], c["py"], c["nx"], c["ny"]
    g = torch.randn(px * py, ny, nx, device="cuda", generator=_gen(seed)).double()
    g = g.view(py, px, ny, nx).permute(0, 2, 1, 3).reshape(py * ny, px * nx)
    for _ in range(c["iters"]):
        g = 0.25 * ((g.roll(1, 0) + g.roll(-1, 0)) + (g.roll(1, 1) + g.roll(-1, 1)))
    return {"tile": g.view(py, ny, px, nx).permute(0, 2, 1, 3).reshape(px * py, ny, nx)}


# ------------------------------------------------------------------------------ serving
AMO_WORDS = 1024  # table words per PE


def _serve_requests(c, seed):
    """60 % put / get of 8 B-1 MiB, 25 % atomics (each on a word of its own), 10 % fp32 / bf16
    reductions of 16 Ki-256 Ki elements, 5 % alltoall of 4-64 KiB; every payload staged."""
    npes, count, arena = c["npes"], c["count"], c["arena"]
    r = np.random.RandomState(seed & 0x7FFFFFFF)
    q = np.zeros(count, sg.REQ_DTYPE)
    words = r.permutation(npes * AMO_WORDS)

    def log_int(lo, hi):
        return int(math.exp(r.uniform(math.log(lo), math.log(hi))))

    for i in range(count):
        u, o = r.rand(), q[i]
        o["word"] = r.randint(1, 1 << 62)
        if u < 0.60:
            o["kind"], o["flags"], o["pe"], o["issuer"], o["n"] = r.choice([K_PUT, K_GET]), 1, r.randint(npes), r.randint(npes), 8 * log_int(1, 128 * KIB)
        elif u < 0.85:
            o["kind"], o["dtype"], o["word"], o["operand"], o["cond"] = r.choice([K_ADD, K_ADD, K_CAS, K_XOR]), sg.INT64, words[i], r.randint(1, 1 << 20), words[i]
        else:
            P = log_int(2, min(32, npes))
            o["flags"], o["issuer"], o["pe"] = 1, P, r.randint(npes - P + 1)
            if u < 0.95:
                o["kind"], o["dtype"], o["fmt"] = K_REDUCE, sg.FLOAT, sg.FMT_F32 if r.rand() < 0.5 else sg.FMT_BF16
                o["n"] = 4 * log_int(4 * KIB, 64 * KIB)
            else:
                o["kind"], o["n"] = K_A2A, min(16 * log_int(256, 4 * KIB), arena // 4 // P // 16 * 16)
    return q


def _prepare_serve(c, seed):
    npes, count = c["npes"], c["count"]
    st = State(npes, c["arena"] + 8 * AMO_WORDS)
    arena, table = st.malloc(c["arena"]), st.malloc(8 * AMO_WORDS)
    t = st.rows(table, torch.int64, AMO_WORDS)
    t.copy_(torch.arange(npes * AMO_WORDS, dtype=torch.int64, device="cuda").view(npes, AMO_WORDS))
    cfg = sg.ServerCfg(ring_slots=4096, arena_offset=arena.offset, arena_bytes=c["arena"], amo_offset=table.offset, amo_words=AMO_WORDS)
    reqs, due = _serve_requests(c, seed), np.zeros(count, np.uint64)
    recs = np.zeros(count, sg.COMPLETION_DTYPE)
    stream = torch.cuda.Stream()

    def go():
        # (a program's server lives longer; here its whole life is one pass, after what its stream's caller enqueued)
        stream.wait_stream(torch.cuda.current_stream())
        server = sg.Server(cfg, stream)
        try:
            server.feed(reqs, due)
            got, give_up = 0, time.monotonic() + 30
            while got < count and time.monotonic() < give_up:
                got += server.poll(recs[got:])
        finally:
            server.stop()
        order = np.argsort(recs["ticket"], kind="stable")
        return {"result": recs["result"][order].view(np.int64), "status": recs["status"][order], "table": t}
    st.go = go
    return st


def _serve_bytes(c):
    """A request's payload is written, read and its result written (seed 0's list; every seed's has the same mix)."""
    q = _serve_requests(c, 0)
    k, n, P = q["kind"], q["n"].astype(np.int64), q["issuer"].astype(np.int64)
    bf = q["fmt"] == sg.FMT_BF16
    rma = 3 * n[(k == K_PUT) | (k == K_GET)].sum()
    a2a = (3 * P * P * n)[k == K_A2A].sum()
    f32 = (12 * P * n)[(k == K_REDUCE) & ~bf].sum()
    b16 = (2 * 2 * P * n + 4 * P * n)[(k == K_REDUCE) & bf].sum()
    return float(rma + a2a + f32 + b16 + 16 * ((k == K_ADD) | (k == K_CAS) | (k == K_XOR)).sum())


# ------------------------------------------------------------------------------ dispatch
_PREPARE = {"rma": _prepare_rma, "fcollect": _prepare_move, "broadcast": _prepare_move, "alltoall": _prepare_move, "reduce": _prepare_reduce,
            "quant": _prepare_quant, "script": _prepare_script, "ring": _prepare_ring, "batch": _prepare_batch, "amo": _prepare_amo,
            "halo": _prepare_halo, "serve": _prepare_serve}
_EXACT = {"reduce": _exact_reduce, "quant": _exact_quant, "batch": _exact_batch, "halo": _exact_halo}


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def exact(case, seed):
    f = _EXACT.get(case["kind"])
    return f(case, seed) if f else None


def work(case):
    """Bytes of one pass: every input read once, every output written once."""
    c, k = case, case["kind"]
    if k == "rma":
        b = 2 * c["n"] + (8 if c["op"] == "put_signal" else 0)
    elif k == "broadcast":
        b = (c["P"] + 1) * c["n"]
    elif k == "fcollect":
        b = (c["P"] + c["P"] ** 2) * c["n"]
    elif k == "alltoall":
        b = 2 * c["P"] ** 2 * c["n"]
    elif k == "reduce":
        b = 2 * c["P"] * c["n"] * DT[c["dtype"]][2]
    elif k == "quant":
        b = c["P"] * ((8 + FMT[c["fmt"]][1]) * c["n"] + 4 * -(-c["n"] // 128))
    elif k == "script":
        b = _script_bytes(c)
    elif k == "ring":
        b = 2 * c["npes"] * c["n"]
    elif k == "batch":
        per = {"f32": 8, "bf16": 6, "e4m3": 5, "i64": 16}
        b = sum(P * n * per[kind] for kind, _, P, n, _ in _batch_teams(c)[0])
    elif k == "amo":
        b = c["nops"] * (28 if c["dist"] == "unique" else 4) + (0 if c["dist"] == "unique" else 16 * min(c["nops"], 1 << c["words_log2"]))
    elif k == "halo":
        b = 8 * c["px"] * c["py"] * c["nx"] * c["ny"]  # the input tile read, the result written
    else:
        b = _serve_bytes(c)
    return {"bytes": float(b), "flops": 0.0}
