"""GPU parity where a call's work is cut differently from its PEs or vectors: ends of
ranges, remainders, the smallest and largest sizes of each form."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_amo_quant_batch import _check_stream, _table_heap
from test_gpu_halo import _run as _run_halo
from gpu_util import download, first_diff, random_heap, upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("agg", [0, 1])
@pytest.mark.parametrize("npes,wpp,nops", [(1, 2048, 1), (3, 1000, 255), (3, 1000, 257), (1, 2048, 513), (64, 32, 152 * 3 * 256 * 2 + 1)])
def test_amo_stream_ranges_of_the_grid(sg, heapf, orc, agg, npes, wpp, nops):
    """The stream is cut into ranges of 256-op blocks over the resident CTAs, whatever the
    PE count: one op, a block less or more one op, one op past a full round of the GPU."""
    h, init = _table_heap(heapf, npes, wpp, 11)
    _check_stream(sg, orc, h, init, W.amo_stream_np(5, nops, 11), wpp, 21, 11, agg)


@pytest.mark.parametrize("px,py,nx,ny,iters", [
    (1, 1, 16, 16, 3), (1, 1, 16, 15, 2),               # the smallest tile whose words fit, and one below
    (2, 2, 12, 24, 5), (3, 1, 132, 61, 4),              # columns that no warp divides, a ragged last thread row
    (1, 2, 16, 2048, 4), (1, 1, 16, 2050, 3),           # the most rows of a CTA, and two more
    (2, 1, 2048, 16, 3), (1, 1, 2048, 61, 2),           # one thread row per CTA; uneven bands
    (2, 2, 256, 256, 5), (19, 8, 128, 64, 2),           # 16 and 8 rows per thread; a PE on every SM
    (1, 1, 512, 512, 2), (1, 1, 520, 512, 3), (2, 1, 520, 600, 2)])  # the largest in registers; past it, several CTAs per PE
def test_halo_tiles_in_registers(sg, heapf, orc, px, py, nx, ny, iters):
    got, want, sig = _run_halo(sg, heapf, orc, px, py, nx, ny, iters)
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
    assert not sig.any()


@pytest.mark.parametrize("px,py,nx,ny", [(2, 2, 8, 8), (1, 1, 4, 3), (2, 1, 4, 1023), (2, 1, 4, 1024), (1, 2, 1020, 4), (1, 2, 1024, 4)])
def test_halo_tiles_too_thin_for_registers(sg, heapf, orc, px, py, nx, ny):
    """Streamed tiles on either side of 4096 points, from which several CTAs take a PE."""
    got, want, sig = _run_halo(sg, heapf, orc, px, py, nx, ny, 5)
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
    assert not sig.any()


@pytest.mark.parametrize("nx,ny", [(64, 64), (256, 200)])
def test_halo_captured_and_replayed(sg, heapf, orc, nx, ny):
    """A captured run (one CTA per PE; several) replays on what the last replay left."""
    px, py, iters = 2, 2, 4
    hs, n = sg.halo_stride(nx, ny), nx * ny
    h = heapf(px * py, (8 * n + 8 * hs + 64 + 4095) // 4096 * 4096)
    tiles, halos, sigs = h.sym(0, 8 * n), h.sym(8 * n, 8 * hs), h.sym(8 * n + 8 * hs, 32)
    h.partitions().zero_()
    grid = W.normals_np(4, px * py * n).astype(np.float32).reshape(py * ny, px * nx)
    for p in range(px * py):
        t = grid[p // px * ny:(p // px + 1) * ny, p % px * nx:(p % px + 1) * nx]
        h.view(tiles, p, torch.float32, n).copy_(torch.from_numpy(np.ascontiguousarray(t).reshape(-1)))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        sg.halo_jacobi(tiles, halos, sigs, px, py, nx, ny, iters)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert sg.get_status()[0] == 0
    want = orc.halo_jacobi(grid, 3 * iters)
    for p in range(px * py):
        t = want[p // px * ny:(p // px + 1) * ny, p % px * nx:(p % px + 1) * nx]
        assert np.array_equal(h.view(tiles, p, torch.float32, n).cpu().numpy().reshape(ny, nx).view(np.uint32), t.view(np.uint32))


RAGGED = [1, 2, 3, 7, 8, 9, 15, 16, 17, 31, 33, 100, 4095, 8191, 8192, 32767, 32768, 32773, 70004, 262147]


@pytest.mark.parametrize("ds,ss", [(0, 0), (0, 1), (1, 0), (3, 3), (4, 12), (8, 0), (15, 2), (5, 14)])
def test_rma_any_alignment(sg, heapf, ds, ss):
    """Heads, bodies and tails of put, get and put_signal: no byte outside the range changes."""
    npes, H = 3, 1 << 20
    h = heapf(npes, H)
    for k, n in enumerate(RAGGED):
        want = random_heap(npes, H, 100 + k)
        upload(h, want)
        m = want.reshape(npes, H)
        dst, src = 300000 + ds, 4096 + ss   # (300000 is a multiple of 32: the shift alone decides)
        sg.putmem(h.base + dst, h.base + src, n, 2, 0)
        m[2, dst:dst + n] = m[0, src:src + n]
        sg.getmem(h.base + dst, h.base + src, n, 2, 1)
        m[1, dst:dst + n] = m[2, src:src + n]
        sg.putmem_signal(h.base + dst + 300032, h.base + src, n, h.base + 8, 3, sg.SIGNAL_SET, 0, 1)
        m[0, dst + 300032:dst + 300032 + n] = m[1, src:src + n]
        m[0, 8:16].view(np.uint64)[0] = 3
        assert first_diff(download(h), want) is None, n


@pytest.mark.parametrize("P,start,stride", [(1, 4, 1), (3, 1, 2), (16, 0, 1)])
@pytest.mark.parametrize("ds,ss", [(0, 0), (4, 0), (7, 13)])
def test_collectives_of_ragged_blocks(sg, heapf, P, start, stride, ds, ss):
    npes, H = 16, 1 << 20
    h = heapf(npes, H)
    team = sg.team_split_strided(sg.TEAM_WORLD, start, stride, P)
    pes = [start + r * stride for r in range(P)]
    dst, src = 524288 + ds, 1024 + ss
    for k, n in enumerate([1, 3, 4, 20, 130, 4092, 4100, 8195, 20004] + ([32780, 100003] if P < 4 else [])):
        for op in ("broadcast", "fcollect", "alltoall"):
            want = random_heap(npes, H, 7 * k + len(op))
            upload(h, want)
            m = want.reshape(npes, H)
            old = m.copy()
            if op == "broadcast":
                sg.broadcastmem(team, h.base + dst, h.base + src, n, P - 1)
            elif op == "fcollect":
                sg.fcollectmem(team, h.base + dst, h.base + src, n)
            else:
                sg.alltoallmem(team, h.base + dst, h.base + src, n)
            for j, q in enumerate(pes):
                if op == "broadcast":
                    m[q, dst:dst + n] = old[pes[-1], src:src + n]
                    continue
                for i, p in enumerate(pes):
                    s = src if op == "fcollect" else src + j * n
                    m[q, dst + i * n:dst + (i + 1) * n] = old[p, s:s + n]
            assert first_diff(download(h), want) is None, (op, n)
    sg.team_destroy(team)


@pytest.mark.parametrize("tile", [0, 1024, 2048])
def test_batch_plans_over_ragged_teams(sg, heapf, orc, tile):
    """The per-team plan (0) and uniform tiles: lengths at the ends of vectors, chunks and
    tiles, codes on and off their alignments, teams of 1 to 33 members."""
    world, H = 33, 2 << 20
    h = heapf(world, H)
    sizes = [1, 3, 4, 5, 127, 513, 1023, 1024, 1027, 4095, 4096, 5125]
    kinds = ["i64", "f32", "bf16", "e4m3"]
    descs, teams = [], []
    tmp = h.malloc(4 * 6000)
    x = W.normals_np(8, world * 6000).astype(np.float32).reshape(world, 6000)
    for p in range(world):
        h.view(tmp, p, torch.float32, 6000).copy_(torch.from_numpy(x[p]))
    for k, n in enumerate(sizes):
        for j, kind in enumerate(kinds):
            P = (1, 2, 7, 16, 33)[(k + j) % 5]
            start = (k * 5 + j) % (world - P + 1)
            shift = (0, 0, 1, 4)[(k + j) % 4]      # elements the source starts off its object
            qs = {"i64": 8, "f32": 4, "bf16": 2, "e4m3": 1}[kind]
            src, dst = h.malloc(qs * (n + 8)), h.malloc(8 * (n + 8))
            so, do = src.offset + shift * qs, dst.offset + (8 if kind == "i64" else 4) * (shift & 1)
            sc = h.malloc(4 * ((n + 127) // 128))
            for p in range(world):
                if kind == "i64":
                    v = W.uniform_ints_np(k, np.arange(n, dtype=np.uint64) + np.uint64(p * n), -(1 << 40), 1 << 40)
                    h.view(h.sym(so), p, torch.int64, n).copy_(torch.from_numpy(v))
                elif kind == "f32":
                    h.view(h.sym(so), p, torch.float32, n).copy_(torch.from_numpy(x[p, :n]))
            if qs < 4:
                sg.quantize(sg.TEAM_WORLD, h.base + so, sc, tmp, 0 if kind == "bf16" else 1, n)
            fmt = {"bf16": 0, "e4m3": 1}.get(kind, -1)
            descs.append(sg.CollDesc(start, P, sg.INT64 if kind == "i64" else sg.FLOAT, fmt, n, h.base + do, h.base + so,
                                     sc.ptr if fmt >= 0 else None))
            teams.append((kind, (start, 1, P), do, so, sc.offset, fmt, n))
    torch.cuda.synchronize()
    init = download(h)
    b = sg.Batch(descs, sg.Tune(tile, 0, 0, 0) if tile else None)
    b.launch()
    got = download(h)
    b.destroy()
    ref = orc.Heap(world, H, init)
    for kind, team, do, so, sco, fmt, n in teams:
        if fmt >= 0:
            ref.qsum_reduce(team, do, so, sco, fmt, n)
        else:
            ref.reduce(team, do, so, n, W.DT_INT64 if kind == "i64" else W.DT_FLOAT, W.RED_SUM)
    assert first_diff(got, ref.mem) is None


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("n,qshift", [(128 * 96, 0), (128 * 95 + 77, 1)])
def test_quantize_near_the_midpoints(sg, heapf, orc, fmt, n, qshift):
    """Quotients within a few units of the last place of the formats' midpoints, where the
    codes turn; scales over binary32's whole range, zeros, the smallest numbers."""
    rng = np.random.RandomState(3 + fmt)
    if fmt == 1:
        codes = np.array([orc.e4m3_decode(q) for q in range(127)])
    else:
        codes = np.array([orc.bf16_decode(q) for q in range(0x3C00, 0x3F81)])
    mids = (codes[1:] + codes[:-1]) / 2
    x = np.zeros((2, 96 * 128), np.float32)
    for p in range(2):
        for b in range(96):
            amax = np.float32(np.ldexp(1 + rng.rand(), rng.randint(-149, 127) if b % 3 == 0 else rng.randint(-20, 20)))
            s = np.float32(amax / np.float32(448.0)) if fmt == 1 else amax
            m = mids[rng.randint(0, len(mids), 128)] * rng.choice([-1.0, 1.0], 128)
            v = (m * np.float64(s) * (1 + rng.randint(-6, 7, 128) * 2.0 ** -25)).astype(np.float32)
            v[np.abs(v) > amax] = amax
            v[rng.randint(1, 128, 6)] = [0.0, -0.0, 1e-45, -1e-45, 1.1754944e-38, -amax]
            v[0] = amax
            x[p, 128 * b:128 * b + 128] = v
        x[p, 128 * 7:128 * 8] = 0.0
    qs = 1 if fmt == 1 else 2
    h = heapf(2, 1 << 18)
    src, sc = h.malloc(4 * n), h.malloc(4 * 96)
    q = h.malloc(qs * (n + 8))
    for p in range(2):
        h.view(src, p, torch.float32, n).copy_(torch.from_numpy(x[p, :n]))
    sg.quantize(sg.TEAM_WORLD, q.ptr + qs * qshift, sc, src, fmt, n)
    torch.cuda.synchronize()
    for p in range(2):
        wq, ws = orc.quantize(x[p, :n], fmt)
        gs = h.view(sc, p, torch.float32, len(ws)).cpu().numpy()
        gq = h.view(h.sym(q.offset + qs * qshift), p, torch.uint8, qs * n).cpu().numpy()
        assert np.array_equal(gs.view(np.uint32), np.asarray(ws, np.float32).view(np.uint32))
        assert np.array_equal(gq, np.asarray(wq).view(np.uint8).reshape(-1))


def test_autotune_keeps_the_batch_s_own_plan_where_it_is_the_fastest(sg, heapf):
    """Four teams of 128 PEs x 8192 int64: the uniform tiles leave most of the GPU idle (three times the
    per-team plan's time)."""
    P, n = 128, 8192
    h = heapf(P, 8 * 8 * n + 65536)
    objs = [(h.malloc(8 * n), h.malloc(8 * n)) for _ in range(4)]
    x = torch.arange(n, device="cuda")
    for k, (_, src) in enumerate(objs):
        for p in range(P):
            h.view(src, p, torch.int64, n).copy_(x * (k + 1) + p)
    b = sg.Batch([sg.CollDesc(0, P, sg.INT64, -1, n, dst.ptr, src.ptr, None) for dst, src in objs], None)
    assert b.autotune().tile_elems == 0
    for dst, _ in objs:
        for p in range(P):
            h.view(dst, p, torch.int64, n).zero_()
    b.launch()
    for k, (dst, _) in enumerate(objs):
        for p in (0, 77, P - 1):
            assert torch.equal(h.view(dst, p, torch.int64, n), x * (k + 1) * P + P * (P - 1) // 2)
    b.destroy()


@pytest.mark.parametrize("n,qshift", [(128 * 96, 0), (128 * 95 + 77, 1)])
def test_quantize_bf16_below_the_normal_range(sg, heapf, orc, n, qshift):
    """Quotients near the midpoints of bf16's subnormal codes, which binary32 holds with few bits: the
    code is the division's."""
    rng = np.random.RandomState(17)
    x = np.zeros((2, 96 * 128), np.float32)
    for p in range(2):
        for b in range(96):
            amax = np.float32(np.ldexp(1 + rng.rand(), rng.randint(-3, 101)))
            q = (rng.randint(0, 0x101, 128) + 0.5 + rng.randint(-3, 4, 128) * 2.0 ** -16) * 2.0 ** -133
            with np.errstate(under="ignore"):
                v = (q * rng.choice([-1.0, 1.0], 128) * np.float64(amax)).astype(np.float32)
            v[0] = amax
            x[p, 128 * b:128 * b + 128] = v
    # pairs whose product with the reciprocal lies on the other side
    x[0, 0:2] = np.array([0x3f81f780, 0x000fbcf8], np.uint32).view(np.float32)
    x[0, 2:128] = 0.0
    x[0, 128:130] = [float.fromhex("0x1.25a05cp+85"), float.fromhex("0x1.4a548cp-46")]
    h = heapf(2, 1 << 18)
    src, sc, q = h.malloc(4 * n), h.malloc(4 * 96), h.malloc(2 * (n + 8))
    for p in range(2):
        h.view(src, p, torch.float32, n).copy_(torch.from_numpy(x[p, :n]))
    sg.quantize(sg.TEAM_WORLD, q.ptr + 2 * qshift, sc, src, 0, n)
    torch.cuda.synchronize()
    for p in range(2):
        wq, ws = orc.quantize(x[p, :n], 0)
        gs = h.view(sc, p, torch.float32, len(ws)).cpu().numpy()
        gq = h.view(h.sym(q.offset + 2 * qshift), p, torch.uint16, n).cpu().numpy()
        assert np.array_equal(gs.view(np.uint32), np.asarray(ws, np.float32).view(np.uint32))
        assert np.array_equal(gq, np.asarray(wq).view(np.uint16).reshape(-1))


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("P,n,shift", [(1, 1, 0), (3, 1023, 0), (8, 1024, 0), (17, 5121, 0), (5, 2000, 1), (2, 2 * 608 * 2048 + 1029, 0)])
def test_qsum_chunk_forms(sg, heapf, orc, fmt, P, n, shift):
    """Chunks of 4 and 8 elements per thread, their tails, codes off their alignment."""
    qs = 1 if fmt == 1 else 2
    nb = (n + 127) // 128
    H = ((qs + 4) * (n + 512) + 4 * nb + 65536 + 4 * (n + 512)) // 4096 * 4096 + 4096
    h = heapf(P, H)
    src, q, sc, dst = h.malloc(4 * n), h.malloc(qs * (n + 8)), h.malloc(4 * nb), h.malloc(4 * n)
    x = W.normals_np(6, P * n).astype(np.float32).reshape(P, n)
    for p in range(P):
        h.view(src, p, torch.float32, n).copy_(torch.from_numpy(x[p]))
    sg.quantize(sg.TEAM_WORLD, q.ptr + qs * shift, sc, src, fmt, n)
    torch.cuda.synchronize()
    init = download(h)
    sg.qsum_reduce(sg.TEAM_WORLD, dst, q.ptr + qs * shift, sc, fmt, n)
    ref = orc.Heap(P, H, init)
    ref.qsum_reduce((0, 1, P), dst.offset, q.offset + qs * shift, sc.offset, fmt, n)
    assert first_diff(download(h), ref.mem) is None


@pytest.mark.parametrize("dt,op", [("int32", 0), ("int64", 1), ("int64", 0), ("float", 0), ("float", 1), ("float", 2)])
@pytest.mark.parametrize("P,start,stride", [(1, 0, 1), (7, 3, 2), (8, 0, 1), (24, 1, 2), (33, 2, 1), (50, 0, 1), (64, 0, 1)])
def test_reduce_ragged_lengths(sg, heapf, orc, dt, op, P, start, stride):
    """Partial last vectors in every form -- several threads per vector, one, the bulk ring --
    in place and not: nothing past the object changes."""
    es = 8 if dt == "int64" else 4
    sizes = [1, 3, 5, 1023, 4099] + ([32771] if P in (24, 50) else []) + ([300001] if P == 8 else [])
    npes, n_max = 64, max(sizes)
    H = (2 * es * (n_max + 64) + 4095) // 4096 * 4096
    h = heapf(npes, H)
    team = sg.team_split_strided(sg.TEAM_WORLD, start, stride, P)
    code = {"int32": sg.INT32, "int64": sg.INT64, "float": sg.FLOAT}[dt]
    for k, n in enumerate(sizes):
        init = random_heap(npes, H, 40 + k)
        if dt == "float":
            init = W.normals_np(9 + k, npes * H // 4).astype(np.float32).view(np.uint8).copy()
        src, dst = 256, (256 if k % 2 else 256 + (es * n + 271) // 16 * 16)
        upload(h, init)
        sg.reduce(team, h.base + dst, h.base + src, n, code, op)
        ref = orc.Heap(npes, H, init)
        ref.reduce((start, stride, P), dst, src, n, {"int32": W.DT_INT32, "int64": W.DT_INT64, "float": W.DT_FLOAT}[dt],
                   (W.RED_SUM, W.RED_MAX, W.RED_MIN)[op])
        assert first_diff(download(h), ref.mem) is None, n
    sg.team_destroy(team)


@pytest.mark.parametrize("op", [1, 2])
@pytest.mark.parametrize("P", [7, 8, 24, 41, 64])
def test_reduce_float_extrema_of_special_values(sg, heapf, op, P):
    """NaN, infinities and signed zeros: a member's value replaces the running one only where
    it compares greater (less), members in rank order, whatever threads share a vector."""
    n = 2000
    h = heapf(64, 1 << 16)
    rng = np.random.RandomState(P)
    x = rng.choice(np.array([0.0, -0.0, np.nan, np.inf, -np.inf, 1.5, -2.0], np.float32), (64, n))
    src, dst = h.malloc(4 * n), h.malloc(4 * n)
    for p in range(64):
        h.view(src, p, torch.float32, n).copy_(torch.from_numpy(x[p]))
    team = sg.team_split_strided(sg.TEAM_WORLD, 0, 1, P)
    sg.reduce(team, dst, src, n, sg.FLOAT, op)
    want = x[0].copy()
    with np.errstate(invalid="ignore"):
        for p in range(1, P):
            take = x[p] > want if op == 1 else x[p] < want
            want[take] = x[p][take]
    for p in (0, P - 1):
        got = h.view(dst, p, torch.float32, n).cpu().numpy()
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
    sg.team_destroy(team)


@pytest.mark.parametrize("mode,cd", [(0, 1), (1, 2)])
@pytest.mark.parametrize("span,biggest,seed", [(256, 64, 1), (4096, 3000, 2), (300000, 200000, 3)])
def test_script_ops_of_one_pe_keep_their_order(sg, heapf, orc, mode, cd, span, biggest, seed):
    """Puts, gets and AMOs of one PE over a few bytes, read after write, written after read and
    twice written in every order: the result is the list's, whichever of them overlap in time."""
    npes, H, nops = 3, (span + 4095) // 4096 * 4096 + 4096, 333
    rng = np.random.RandomState(seed)
    ops = np.zeros(nops, W.OP_DTYPE)
    for i in range(nops):
        o = ops[i]
        o["issuer"], o["pe"] = 0, rng.randint(0, npes)
        if rng.rand() < 0.3:
            o["kind"], o["dtype"] = rng.choice([W.OP_FADD, W.OP_CSWAP, W.OP_FXOR]), W.DT_INT64
            o["dst"], o["operand"], o["cond"] = 8 * rng.randint(0, span // 8), rng.randint(1, 1 << 40), 0
            continue
        n = int(np.exp(rng.rand() * np.log(biggest)))
        if rng.rand() < 0.5:
            n = max(16, n // 16 * 16)
        a = 16 if n % 16 == 0 and rng.rand() < 0.7 else 1
        o["kind"], o["n"] = rng.choice([W.OP_PUT, W.OP_GET]), n
        o["dst"], o["src"] = rng.randint(0, (span - n) // a + 1) * a, rng.randint(0, (span - n) // a + 1) * a
        if o["pe"] == 0 and o["dst"] < o["src"] + n and o["src"] < o["dst"] + n:
            o["pe"] = 1                                   # (a copy onto itself is undefined)
    h = heapf(npes, H, pe_mode=mode, cluster_dim=cd)
    init = random_heap(npes, H, seed)
    upload(h, init)
    fetched = torch.zeros(nops, dtype=torch.int64, device="cuda")
    sg.run_script(torch.from_numpy(ops.view(np.uint8).copy()).cuda(), nops, fetched)
    torch.cuda.synchronize()
    assert sg.get_status()[0] == 0
    ref = orc.Heap(npes, H, init)
    want = ref.run_script(ops)
    assert first_diff(download(h), ref.mem) is None
    amo = np.isin(ops["kind"], [W.OP_FADD, W.OP_CSWAP, W.OP_FXOR])
    if want is not None:
        assert np.array_equal(fetched.cpu().numpy()[amo], np.asarray(want)[amo])


@pytest.mark.parametrize("mode,cd", [(0, 1), (1, 2)])
@pytest.mark.parametrize("n", [8, 4096, 131072])
@pytest.mark.parametrize("at", [126, 127, 128, 255])
def test_script_op_alone_in_its_batch_sees_the_one_before(sg, heapf, orc, mode, cd, n, at):
    """PE 0 has two ops, at the end of one batch of the list and alone in the next (or beside it): a
    put, and a get of what it wrote."""
    npes, H = 3, 1 << 19
    ops = np.zeros(at + 2, W.OP_DTYPE)
    ops["kind"], ops["dtype"], ops["issuer"], ops["pe"] = W.OP_FADD, W.DT_INT64, 2, 2
    ops["dst"], ops["operand"] = 8 * (np.arange(at + 2) % 16), 3
    for i, kind, dst, src in ((at, W.OP_PUT, 1 << 17, 0), (at + 1, W.OP_GET, 2 << 17, 1 << 17)):
        ops[i] = np.zeros(1, W.OP_DTYPE)[0]
        ops[i]["kind"], ops[i]["issuer"], ops[i]["pe"], ops[i]["n"], ops[i]["dst"], ops[i]["src"] = kind, 0, 1, n, dst, src
    h = heapf(npes, H, pe_mode=mode, cluster_dim=cd)
    init = random_heap(npes, H, at)
    upload(h, init)
    fetched = torch.zeros(len(ops), dtype=torch.int64, device="cuda")
    sg.run_script(torch.from_numpy(ops.view(np.uint8).copy()).cuda(), len(ops), fetched)
    torch.cuda.synchronize()
    assert sg.get_status()[0] == 0
    ref = orc.Heap(npes, H, init)
    ref.run_script(ops)
    assert first_diff(download(h), ref.mem) is None


@pytest.mark.parametrize("npes", [1, 2, 5, 64])
def test_barriers_back_to_back(sg, heapf, orc, npes):
    """Consecutive barriers, in which PEs arrive at the next before the last has been folded:
    every PE's word goes round the ring one place per barrier."""
    rounds, H = 200, 8192
    h = heapf(npes, H)
    ops = []
    for r in range(rounds):
        for p in range(npes):
            o = np.zeros(1, W.OP_DTYPE)[0]
            o["kind"], o["issuer"], o["pe"], o["n"] = W.OP_PUT, p, (p + 1) % npes, 8
            o["src"], o["dst"] = 16 * (r % 2), 16 * ((r + 1) % 2)
            ops.append(o)
        for _ in range(1 + r % 3):
            o = np.zeros(1, W.OP_DTYPE)[0]
            o["kind"], o["issuer"] = W.OP_BARRIER_ALL, -1
            ops.append(o)
    ops = np.array(ops, W.OP_DTYPE)
    init = random_heap(npes, H, 5)
    upload(h, init)
    fetched = torch.zeros(len(ops), dtype=torch.int64, device="cuda")
    sg.run_script(torch.from_numpy(ops.view(np.uint8).copy()).cuda(), len(ops), fetched)
    torch.cuda.synchronize()
    assert sg.get_status()[0] == 0
    ref = orc.Heap(npes, H, init)
    ref.run_script(ops)
    assert first_diff(download(h), ref.mem) is None


@pytest.mark.parametrize("npes,arena_pages,inflight,count", [(4, 3, 1, 60), (8, 70, 5, 400), (33, 130, 64, 1000), (90, 4096, 1024, 1500)])
def test_serving_page_and_slot_reuse(sg, heapf, npes, arena_pages, inflight, count):
    """Few slots and pages reused many times, runs of pages across bitmap words, queues shorter and
    longer than the workers' window: every result equals the plain path's.
    (90 PEs x 4096 pages: bitmaps too large for the admitter's shared memory.)"""
    page = 256
    arena = arena_pages * page
    H = (arena + 8 * 64 + 4095) // 4096 * 4096
    h = heapf(npes, H)
    lay_amo = arena
    h.partitions().zero_()
    rng = np.random.RandomState(count)
    q = np.zeros(count, sg.REQ_DTYPE)
    for i in range(count):
        r = q[i]
        r["word"], r["flags"] = rng.randint(1, 1 << 60), 1
        u = rng.rand()
        if u < 0.6:
            r["kind"], r["pe"], r["issuer"] = rng.choice([W.OP_PUT, W.OP_GET]), rng.randint(npes), rng.randint(npes)
            r["n"] = 8 * rng.randint(1, max(2, arena // 2 // 8))
            r["n"] = min(int(r["n"]), arena // 2 // 16 * 16)
        elif u < 0.8:
            r["kind"], r["dtype"], r["flags"], r["word"], r["operand"] = W.OP_FADD, W.DT_INT64, 0, i % 64, 3
        else:
            P = rng.randint(1, npes + 1)
            r["kind"], r["dtype"], r["fmt"], r["issuer"], r["pe"] = W.OP_REDUCE, W.DT_FLOAT, 0xFF, P, rng.randint(npes - P + 1)
            r["n"] = 4 * rng.randint(1, max(2, arena // 16))
    cfg = sg.ServerCfg(page_bytes=page, max_inflight=inflight, ring_slots=256, arena_offset=0, arena_bytes=arena, amo_offset=lay_amo, amo_words=64)
    rec = torch.zeros(sg.COMPLETION_DTYPE.itemsize, dtype=torch.uint8).pin_memory()
    want = np.zeros(count, np.uint64)
    for i in range(count):
        if q[i]["kind"] == W.OP_FADD:
            continue
        sg.request_run(q[i:i + 1], cfg, rec.data_ptr())
        torch.cuda.synchronize()
        want[i] = rec.numpy().view(sg.COMPLETION_DTYPE)[0]["result"]
    s = torch.cuda.Stream()
    srv = sg.Server(cfg, s)
    recs, got, sent = np.zeros(count, sg.COMPLETION_DTYPE), 0, 0
    import time
    end = time.monotonic() + 30
    try:
        while got < count and time.monotonic() < end:
            while sent < count and srv.submit(sg.Req.from_buffer_copy(q[sent].tobytes())) is not None:
                sent += 1
            got += srv.poll(recs[got:])
    finally:
        srv.stop()
    assert got == count and not recs["status"].any()
    order = np.argsort(recs["ticket"], kind="stable")
    res = recs["result"][order]
    amo = q["kind"] == W.OP_FADD
    assert np.array_equal(res[~amo], want[~amo])
    final = h.view(h.sym(lay_amo), 0, torch.int64, 64).cpu().numpy()
    for w in range(64):
        k = np.nonzero(amo & (q["word"] == w))[0]
        assert sorted(res[k].tolist()) == [3 * j for j in range(len(k))] and final[w] == 3 * len(k)


@pytest.mark.parametrize("px,py,nx,ny,iters", [(2, 2, 64, 64, 1), (2, 2, 64, 64, 2), (2, 2, 64, 64, 3), (2, 2, 256, 256, 4), (2, 2, 256, 256, 5),
                                                (3, 1, 132, 61, 7), (1, 1, 2048, 61, 6), (2, 1, 520, 600, 3), (2, 1, 520, 600, 4)])
def test_halo_other_tile_holds_the_sweep_before(sg, heapf, orc, px, py, nx, ny, iters):
    """Both tiles after a run -- a second run with odd `iters` starts from what is left in tile 0."""
    hs, n = sg.halo_stride(nx, ny), nx * ny
    h = heapf(px * py, (8 * n + 8 * hs + 64 + 4095) // 4096 * 4096)
    tiles, halos, sigs = h.sym(0, 8 * n), h.sym(8 * n, 8 * hs), h.sym(8 * n + 8 * hs, 32)
    h.partitions().zero_()
    grid = W.normals_np(4, px * py * n).astype(np.float32).reshape(py * ny, px * nx)
    cut = lambda g, p: np.ascontiguousarray(g[p // px * ny:(p // px + 1) * ny, p % px * nx:(p % px + 1) * nx]).reshape(-1)
    for p in range(px * py):
        h.view(tiles, p, torch.float32, n).copy_(torch.from_numpy(cut(grid, p)))
    for run in range(2):
        sg.halo_jacobi(tiles, halos, sigs, px, py, nx, ny, iters)
        torch.cuda.synchronize()
        assert sg.get_status()[0] == 0
        last, prev = orc.halo_jacobi(grid, iters), orc.halo_jacobi(grid, iters - 1)
        for p in range(px * py):
            got = h.view(tiles, p, torch.float32, 2 * n).cpu().numpy().reshape(2, n)
            assert np.array_equal(got[iters & 1].view(np.uint32), cut(last, p).view(np.uint32))
            assert np.array_equal(got[(iters & 1) ^ 1].view(np.uint32), cut(prev, p).view(np.uint32))
        grid = prev if iters & 1 else last

def test_host_calls_captured_after_joins_and_fills(sg, heapf):
    """Host-issued calls in a captured stream: after a fill, after a join with another stream, and
    one after the other; replays give what the calls give."""
    npes, n = 8, 5003
    h = heapf(npes, 1 << 17)
    src, dst, tot, sig = h.malloc(4 * n), h.malloc(4 * n), h.malloc(4 * n), h.malloc(8)
    x = torch.zeros(n, device="cuda")
    side = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        x.add_(1.0)
        h.view(src, 3, torch.float32, n).copy_(x)
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            sg.broadcastmem(sg.TEAM_WORLD, dst, src, 4 * n, 3)
        torch.cuda.current_stream().wait_stream(side)
        sg.reduce(sg.TEAM_WORLD, tot, dst, n, sg.FLOAT, sg.SUM)
        sg.putmem_signal(src, tot, 4 * n, sig, 1, sg.SIGNAL_ADD, 5, 2)
        sg.atomic("fetch_add", sg.INT64, sig, 10, 5)
    h.partitions().zero_()
    torch.cuda.synchronize()
    for k in range(1, 4):
        g.replay()
        torch.cuda.synchronize()
        assert sg.get_status()[0] == 0
        for p in range(npes):
            assert torch.all(h.view(dst, p, torch.float32, n) == float(k))
            assert torch.all(h.view(tot, p, torch.float32, n) == float(k * npes))
        assert torch.all(h.view(src, 5, torch.float32, n) == float(k * npes))
        assert h.view(sig, 5, torch.int64, 1).item() == 11 * k


def test_host_calls_chained_on_two_streams(sg, heapf):
    """A long chain of dependent small calls, handed from one stream to another by events: each
    sees the whole result of the one before it."""
    npes = 4
    h = heapf(npes, 1 << 18)
    a = h.malloc(40000)
    h.partitions().zero_()
    h.view(a, 0, torch.int64, 5000).copy_(torch.arange(5000))
    s = [torch.cuda.Stream(), torch.cuda.Stream()]
    for q in s:
        q.wait_stream(torch.cuda.current_stream())
    for k in range(200):
        cur = s[k // 7 % 2]
        if k % 7 == 0:
            cur.wait_stream(s[(k // 7 + 1) % 2])
        if k % 3 == 2:
            sg.reduce(sg.TEAM_WORLD, a, a, 5000, sg.INT64, sg.MAX, stream=cur)
        else:
            sg.putmem(a, a, 40000 - 3 * (k % 2), (k + 1) % npes, k % npes, stream=cur)
    for q in s:
        torch.cuda.current_stream().wait_stream(q)
    sg.reduce(sg.TEAM_WORLD, a, a, 5000, sg.INT64, sg.MAX)
    want = torch.arange(5000, device="cuda")
    for p in range(npes):
        assert torch.equal(h.view(a, p, torch.int64, 5000), want)
