"""GPU parity where a call's work is cut differently from its PEs or vectors: ends of
ranges, remainders, the smallest and largest sizes of each form."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_amo_quant_batch import _check_stream, _table_heap

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("agg", [0, 1])
@pytest.mark.parametrize("npes,wpp,nops", [(1, 2048, 1), (3, 1000, 255), (3, 1000, 257), (1, 2048, 513), (64, 32, 152 * 3 * 256 * 2 + 1)])
def test_amo_stream_ranges_of_the_grid(sg, heapf, orc, agg, npes, wpp, nops):
    """The stream is cut into ranges of 256-op blocks over the resident CTAs, whatever the
    PE count: one op, a block less or more one op, one op past a full round of the GPU."""
    h, init = _table_heap(heapf, npes, wpp, 11)
    _check_stream(sg, orc, h, init, W.amo_stream_np(5, nops, 11), wpp, 21, 11, agg)
