"""GPU parity where a call's work is cut differently from its PEs or vectors: ends of
ranges, remainders, the smallest and largest sizes of each form."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_amo_quant_batch import _check_stream, _table_heap
from test_gpu_halo import _run as _run_halo

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
