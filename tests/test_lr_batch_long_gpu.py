"""Batches of more than 2^24 elements with a long list among short ones, and on both
sides of the limits that decide how they are ranked. Exact."""
import numpy as np
import pytest

import gen
from tests.test_lr_batch_modes_gpu import _check

import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
M = 1 << 20


@pytest.mark.parametrize("sizes", [
    [256] * 5000 + [16 * M],                  # short on average, one list as long as the rest is small
    [24_576] + [1500] * 11_500,               # all short enough for single blocks
    [24_577] + [1500] * 11_500,               # one element too long for one
    [1500] * 11_200 + [0] * 5,
    [8 * M] * 2,                              # 2^24 in all
    [8 * M + 1, 0, 8 * M],
    [8 * M] * 3,                              # long on average
    [3 * M] * 6,
], ids=str)
@pytest.mark.parametrize("in_place", [False, True])
def test_size_mixes_above_2_24(sizes, in_place):
    _check(*gen.list_batch(np.asarray(sizes, np.int64), len(sizes)), in_place=in_place)


@pytest.mark.parametrize("sizes", [[24_576] + [1500] * 11_500, [24_577] + [1500] * 11_500, [8 * M] * 3])
def test_queried_workspace_is_enough(sizes):
    import torch

    succ, off, heads = gen.list_batch(np.asarray(sizes, np.int64), 9)
    stream = torch.cuda.Stream()
    with lrcc.Context(0) as ctx, torch.cuda.stream(stream):
        ctx.reserve(stream, lrcc.workspace_query(lrcc.KIND_LR_BATCH, len(succ), len(sizes)))
        held = ctx.bytes()
        args = [torch.from_numpy(a).to("cuda:0") for a in (succ.astype(np.int32), off.astype(np.int64), heads.astype(np.int32))]
        lrcc.lr_rank_batched(*args, stream=stream)
        assert ctx.last_status(stream) == lrcc.OK and ctx.bytes() == held
