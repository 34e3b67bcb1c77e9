"""The first level that keeps its records in the rank array (in-place plan, lists
of at most 2^24 elements): sizes around its limits, layouts that run a sublist
past the record's position bits, and inputs that are not lists. Exact."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SEED = 0x5EED


def _mix32(h):
    h = h.astype(np.uint64)
    for mul, sh in ((0x85EBCA6B, 16), (0xC2B2AE35, 13), (None, 16)):
        h ^= h >> np.uint64(sh)
        if mul is not None:
            h = (h * np.uint64(mul)) & np.uint64(0xFFFFFFFF)
    return h


def _splitters(n, D, head):
    """The stratified splitter of every block of D ids (the head in its block)."""
    b = np.arange((n + D - 1) // D, dtype=np.uint64)
    size = np.minimum(D, n - b.astype(np.int64) * D).astype(np.uint64)
    h = _mix32((b * np.uint64(0x9E3779B1) + np.uint64(SEED)) & np.uint64(0xFFFFFFFF))
    spl = (b * np.uint64(D) + ((h * size) >> np.uint64(32))).astype(np.int64)
    spl[head // D] = head
    return spl


def _list(order):
    succ = np.full(len(order), -1, np.int32)
    succ[order[:-1]] = order[1:]
    return succ, int(order[0])


@pytest.fixture
def spacing4():
    lrcc.set_plan(lrcc.KIND_LR, 0, 32, rs_level0=1, rs_spacing0=4, rs_spacing=4, seed=SEED)
    yield
    lrcc.reset_plans()


@pytest.mark.parametrize("n", [16385, 65539, 300_007, (1 << 20) + 3, (1 << 24) - 1, 1 << 24, (1 << 24) + 1])
def test_sizes_and_layouts(spacing4, n):
    succ, head, perm = gen.list_random(n, 7, with_perm=True)
    rank = lrcc.lr_rank(torch.from_numpy(succ).to(DEV), head)
    lrcc.check()
    assert np.array_equal(rank.cpu().numpy()[perm], np.arange(n - 1, -1, -1, dtype=np.int32))
    succ, head = gen.list_ordered(n)
    rank = lrcc.lr_rank(torch.from_numpy(succ).to(DEV), head)
    lrcc.check()
    assert np.array_equal(rank.cpu().numpy(), np.arange(n - 1, -1, -1, dtype=np.int32))


@pytest.mark.parametrize("n", [(1 << 17) + 5, 1 << 20])
@pytest.mark.parametrize("first", ["splitter", "plain"])
def test_one_sublist_longer_than_the_position_bits(spacing4, n, first):
    # every element that is no splitter comes in one run, as the first sublist or the last
    rng = np.random.default_rng(n)
    head = 1 if first == "splitter" else 2
    spl = rng.permutation(_splitters(n, 4, head))
    rest = rng.permutation(np.setdiff1d(np.arange(n), spl))
    spl = np.concatenate([[head], spl[spl != head]])
    order = np.concatenate([spl, rest]) if first == "splitter" else np.concatenate([spl[:1], rest, spl[1:]])
    succ, head = _list(order)
    rank = lrcc.lr_rank(torch.from_numpy(succ).to(DEV), head)
    lrcc.check()
    assert np.array_equal(rank.cpu().numpy()[order], np.arange(n - 1, -1, -1, dtype=np.int32))


def test_inputs_that_are_not_one_list(spacing4):
    n = 100_003
    succ, head, perm = gen.list_random(n, 9, with_perm=True)
    plain = np.setdiff1d(np.arange(n), _splitters(n, 4, head))
    loop = succ.copy()                      # two elements that name each other, neither a splitter
    loop[plain[0]], loop[plain[1]] = plain[1], plain[0]
    two = succ.copy()
    two[perm[n // 3]] = -1
    back = succ.copy()
    back[perm[-1]] = perm[n // 2]
    far = succ.copy()
    far[perm[5]] = n
    for bad in (loop, two, back, far):
        lrcc.lr_rank(torch.from_numpy(bad).to(DEV), head)
        assert lrcc.last_status() == lrcc.ERR_INVALID_INPUT
    t = torch.from_numpy(succ).to(DEV)
    assert np.array_equal(lrcc.lr_rank(t, head, out=t).cpu().numpy(), oracle.lr_rank(succ, head))   # out = succ
    lrcc.check()
