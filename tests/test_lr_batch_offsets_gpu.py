"""Batched lists whose offsets do not describe the arrays of the call: every mode
keeps to the arrays and reports what it cannot rank."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
M = 1 << 20

# the mean and the total decide the mode: one block per list (in shared memory or
# not), together with records in the rank array, together by the read-only first level
MIXES = {"blocks": [300] * 50, "blocks_long": [30_000] + [100] * 9, "together": [40_000, 60_000, 70_000],
         "together_large": [2 * M] * 9, "read_only": [17 * M, 17 * M]}


def _call(succ, off, heads, out=None):
    rank = lrcc.lr_rank_batched(torch.from_numpy(np.ascontiguousarray(succ, np.int32)).to(DEV),
                                torch.from_numpy(np.asarray(off, np.int64)).to(DEV),
                                torch.from_numpy(np.asarray(heads, np.int32)).to(DEV), out=out)
    return lrcc.last_status(), rank.cpu().numpy()


@pytest.mark.parametrize("mix", MIXES)
@pytest.mark.parametrize("case", ["decreasing", "past_the_end", "first_not_zero", "negative"])
def test_offsets_that_name_no_lists(mix, case):
    succ, off, heads = gen.list_batch(np.asarray(MIXES[mix], np.int64), 3)
    bad = off.copy()
    if case == "decreasing":
        bad[1] = off[2] + 7
    elif case == "past_the_end":
        bad[-1] = off[-1] + 100_000
    elif case == "first_not_zero":
        bad[0] = 5
    else:
        bad[1] = -4096
    status, _ = _call(succ, bad, heads)
    assert status == lrcc.ERR_INVALID_INPUT
    status, rank = _call(succ, off, heads)
    assert status == lrcc.OK and np.array_equal(rank, oracle.lr_rank_batched(succ, off, heads))


@pytest.mark.parametrize("mix", ["together_large", "read_only"])
@pytest.mark.parametrize("pad", [1, 300_000])
def test_large_totals_beyond_the_last_list_are_reported(mix, pad):
    succ, off, heads = gen.list_batch(np.asarray(MIXES[mix], np.int64), 4)
    status, _ = _call(np.concatenate([succ, np.zeros(pad, np.int32)]), off, heads)
    assert status == lrcc.ERR_INVALID_INPUT
