"""Weighted ranks of a forest take no more workspace than their layout uses, on both
sides of the size from which the records are kept in the walk words. Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_1002_4482_gb300 as lrcc
from tests.test_scan_records_gpu import _dev, _forest

pytestmark = pytest.mark.gpu
NEAR = 1 << 22


@pytest.mark.parametrize("n,per_element", [(NEAR, 30), (NEAR + 1, 21.5), (10_000_019, 21.5)])
@pytest.mark.parametrize("lists", [3, 400_000])
def test_bytes_held(n, per_element, lists):
    succ = _forest(n, lists, n)
    val = np.random.default_rng(n).integers(-(2**31), 2**31, n).astype(np.int32)
    stream = torch.cuda.Stream()
    args = _dev(succ), _dev(val)
    torch.cuda.synchronize()
    with lrcc.Context(0) as ctx:
        ctx.reserve(stream, 0)
        got = lrcc.lr_scan_forest(*args, stream=stream)
        assert ctx.last_status(stream) == lrcc.OK
        assert ctx.bytes() <= per_element * n
    assert np.array_equal(got.cpu().numpy(), oracle.lr_scan_forest(succ, val))


def test_every_element_a_head():
    for n in (NEAR, NEAR + 1):
        val = np.arange(n, dtype=np.int32)
        got = lrcc.lr_scan_forest(_dev(np.full(n, -1, np.int32)), _dev(val))
        lrcc.check()
        assert np.array_equal(got.cpu().numpy(), val)
