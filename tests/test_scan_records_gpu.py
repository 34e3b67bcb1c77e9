"""Weighted ranks whose records are kept apart from the walk words (and, above
2^23 elements, in them): one list and forests around the limits. Exact."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _dev(a, shift=0):
    buf = torch.empty(len(a) + shift, dtype=torch.int32, device=DEV)
    buf[shift:] = torch.from_numpy(np.ascontiguousarray(a, np.int32)).to(DEV)
    return buf[shift:]


def _forest(n, lists, seed):
    """`lists` random lists over a permutation of n ids, self-loop tails on every other one."""
    rng = np.random.default_rng(seed)
    order = gen.permutation(n, seed)
    ends = np.unique(np.concatenate([rng.choice(np.arange(1, n), lists - 1, replace=False), [n]])) if lists > 1 else [n]
    succ = np.empty(n, np.int32)
    succ[order[:-1]] = order[1:]
    tails = order[np.asarray(ends) - 1]
    succ[tails] = -1
    succ[tails[::2]] = tails[::2]
    return succ


@pytest.mark.parametrize("n", [16385, 100_003, (1 << 23) - 1, 1 << 23, (1 << 23) + 1])
@pytest.mark.parametrize("shift", [0, 1])
def test_one_list(n, shift):
    succ, head = gen.list_random(n, n)
    val = (np.arange(n) % 11).astype(np.int32)
    got = lrcc.lr_scan(_dev(succ, shift), _dev(val, shift), head)
    lrcc.check()
    assert np.array_equal(got.cpu().numpy(), oracle.lr_scan(succ, val, head))


@pytest.mark.parametrize("n,lists", [(1, 1), (2, 2), (7, 3), (1000, 1000), (33_000, 1), (33_000, 33_000), (200_003, 4096),
                                     (1 << 23, 100), ((1 << 23) + 1, 5000)])
def test_forests(n, lists):
    succ = _forest(n, lists, n)
    val = np.random.default_rng(n).integers(-(2**31), 2**31, n).astype(np.int32)
    got = lrcc.lr_scan_forest(_dev(succ, 1), _dev(val, 1))
    lrcc.check()
    assert np.array_equal(got.cpu().numpy(), oracle.lr_scan_forest(succ, val))


def test_ordered_forest_and_a_list_longer_than_its_splitters_rounds():
    n = 1 << 20
    succ = np.arange(1, n + 1, dtype=np.int32)
    succ[-1] = -1
    succ[::1000] = -1
    val = np.ones(n, np.int32)
    for s in (succ, np.arange(-1, n - 1, dtype=np.int32)):
        got = lrcc.lr_scan_forest(_dev(s), _dev(val))
        lrcc.check()
        assert np.array_equal(got.cpu().numpy(), oracle.lr_scan_forest(s, val))


@pytest.mark.parametrize("case", ["named_twice", "cycle", "two_cycle", "self_far", "out_of_range"])
@pytest.mark.parametrize("n", [20_000, 300_000])
def test_invalid_forests(case, n):
    succ = _forest(n, 5, 3)
    tail = int(np.flatnonzero((succ == -1) | (succ == np.arange(n)))[0])
    inner = np.flatnonzero((succ != -1) & (succ != np.arange(n)))
    if case == "named_twice":
        succ[inner[0]] = succ[inner[1]]
    elif case == "cycle":                                # the whole list of that tail becomes a cycle
        x = tail
        pred = np.full(n, -1, np.int64)
        pred[succ[inner]] = inner
        while pred[x] >= 0:
            x = pred[x]
        succ[tail] = x
        if x == tail:
            pytest.skip("a list of one element")
    elif case == "two_cycle":                            # two elements that name each other
        a = int(inner[2])
        b = int(succ[a])
        c = succ[b]
        prev = np.flatnonzero(succ == a)
        if len(prev):
            succ[prev[0]] = -1 if c in (-1, b) else c
        succ[b] = a
    elif case == "self_far":
        succ[inner[3]] = n
    else:
        succ[inner[3]] = -2
    lrcc.lr_scan_forest(_dev(succ), _dev(np.ones(n, np.int32)))
    assert lrcc.last_status() == lrcc.ERR_INVALID_INPUT


@pytest.mark.parametrize("n", [20_000, 300_000])
def test_scan_of_a_list_with_a_detached_cycle(n):
    # the list is whole from head to tail but for a cycle of two elements cut out of it
    succ, head = gen.list_random(n, 4)
    a = int(succ[succ[head]])
    b = int(succ[a])
    succ[succ[head]] = succ[b]
    succ[b] = a
    lrcc.lr_scan(_dev(succ), _dev(np.ones(n, np.int32)), head)
    assert lrcc.last_status() == lrcc.ERR_INVALID_INPUT


@pytest.mark.parametrize("n,lists", [((1 << 24) - 32, 1), ((1 << 24) - 16, 1), (1 << 24, 3), ((1 << 24) + 5, 1),
                                     ((1 << 24) + 5, 20_000), (1_500_000, 1_500_000), (1_500_000, 1_200_000)])
def test_forests_whose_splitters_jump_by_rulers(n, lists):
    """Around 2^20 splitters (stratified ones and heads), from where one word of four jumps and the others walk to it."""
    succ = _forest(n, lists, n + lists)
    val = np.random.default_rng(n).integers(-(2**31), 2**31, n).astype(np.int32)
    got = lrcc.lr_scan_forest(_dev(succ), _dev(val))
    lrcc.check()
    assert np.array_equal(got.cpu().numpy(), oracle.lr_scan_forest(succ, val))


@pytest.mark.parametrize("length", [12_000_000, 64, 40, 24, 9])
def test_cycles_among_the_rulers_words(length):
    """A cycle of many splitters, or of a few of which some or none are rulers."""
    n = 1 << 24
    order = gen.permutation(n, length)
    succ = np.empty(n, np.int32)
    succ[order[:-1]] = order[1:]
    succ[order[-1]] = -1
    for start in range(0, 1 if length > 1000 else 64 * length, length):   # many short ones, or one long one
        succ[order[start + length - 1]] = order[start]
    lrcc.lr_scan_forest(_dev(succ), _dev(np.ones(n, np.int32)))
    assert lrcc.last_status() == lrcc.ERR_INVALID_INPUT
