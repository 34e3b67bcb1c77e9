"""Batched list ranking in each of its modes: one block per list (both sizes of
block), all lists together with records in the rank array, and the limits
between them. Exact."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc
from tests.test_direct_level0_gpu import SEED, _splitters

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _check(succ, off, heads, shift=0, in_place=False):
    buf = torch.zeros(len(succ) + shift, dtype=torch.int32, device=DEV)
    buf[shift:] = torch.from_numpy(np.ascontiguousarray(succ, np.int32)).to(DEV)
    s = buf[shift:]
    out = s if in_place else torch.empty(len(succ) + shift, dtype=torch.int32, device=DEV)[shift:]
    lrcc.lr_rank_batched(s, torch.from_numpy(np.asarray(off, np.int64)).to(DEV),
                         torch.from_numpy(np.asarray(heads, np.int32)).to(DEV), out=out)
    lrcc.check()
    assert np.array_equal(out.cpu().numpy(), oracle.lr_rank_batched(succ, off, heads))


@pytest.mark.parametrize("sizes", [
    [8192, 8193, 8191, 1, 0, 24575, 24576, 24577, 100],         # one block per list, every limit of the two kernels
    [16384, 2, 0, 50_000],
    [40_000, 0, 60_000, 1, 0, 31_071, 3, 0],                    # 2^17 + 3 elements: together
    [1 << 17],
    [1 << 17, 1],
    [0, 0, (1 << 20) + 5, 0, 77, 300_001, 0],
    [4096] * 31 + [4095],                                       # just under the limits
    [4096] * 32,
])
@pytest.mark.parametrize("shift", [0, 1])
def test_size_mixes(sizes, shift):
    succ, off, heads = gen.list_batch(np.asarray(sizes, np.int64), 11 + len(sizes))
    succ = succ.copy()
    for k in range(0, len(sizes), 2):                            # every second list ends in a self-loop
        b, e = off[k], off[k + 1]
        if e > b:
            tail = b + int(np.flatnonzero(succ[b:e] == -1)[0])
            succ[tail] = tail - b
    _check(succ, off, heads, shift)
    _check(succ, off, heads, shift, in_place=True)


@pytest.mark.parametrize("total_log", [21, 24, 26])
def test_log_uniform_lists(total_log):
    sizes = gen.loguniform_sizes(1 << (total_log - 16), 8, 19, total_log)
    _check(*gen.list_batch(sizes, total_log))


def test_ordered_lists_and_long_sublists():
    # one list whose elements that are no splitters come in one run, longer than the
    # records' position bits, between two ordered lists
    n, pre = 1 << 20, 70_000
    lrcc.set_plan(lrcc.KIND_LR, 0, 32, rs_spacing0=4, rs_spacing=4, seed=SEED)
    try:
        rng = np.random.default_rng(5)
        total = pre + n + 9
        head0 = 17
        # splitters of the whole id range, those of the middle list by local id
        spl = _splitters(total, 4, head0)
        spl = spl[(spl >= pre) & (spl < pre + n)] - pre
        rest = rng.permutation(np.setdiff1d(np.arange(n), spl))
        order = np.concatenate([rng.permutation(spl), rest])
        mid = np.full(n, -1, np.int32)
        mid[order[:-1]] = order[1:]
        first = np.concatenate([np.arange(1, pre), [-1]])
        first = np.roll(first, 0).astype(np.int32)
        # the first list starts at its element 17: 17 .. pre-1, then 0 .. 16
        first[pre - 1], first[16] = 0, -1
        last = np.concatenate([np.arange(1, 9), [-1]]).astype(np.int32)
        _check(np.concatenate([first, mid, last]), [0, pre, pre + n, total], [head0, int(order[0]), 0])
    finally:
        lrcc.reset_plans()


@pytest.mark.parametrize("case", ["cycle", "two_lists", "head_out_of_range", "succ_out_of_range"])
def test_invalid_lists_are_reported(case):
    sizes = [100, 200_000, 0, 50, 90_000]
    succ, off, heads = gen.list_batch(np.asarray(sizes, np.int64), 40)
    succ, heads = succ.copy(), heads.copy()
    b, e = off[1], off[2]
    tail = b + int(np.flatnonzero(succ[b:e] == -1)[0])
    if case == "cycle":
        succ[tail] = heads[1]
    elif case == "two_lists":
        succ[b + heads[1]] = -1
    elif case == "head_out_of_range":
        heads[4] = sizes[4]
    else:
        succ[tail] = sizes[1]
    lrcc.lr_rank_batched(torch.from_numpy(succ).to(DEV), torch.from_numpy(off).to(DEV), torch.from_numpy(heads).to(DEV))
    assert lrcc.last_status() == lrcc.ERR_INVALID_INPUT
    _check(*gen.list_batch(np.asarray(sizes, np.int64), 41))
