"""Components of one graph in one launch (hook rule 1): the one-block and gang
kernels at their size limits, with and without a sample, with each membership
table, on graphs with hot roots, deep chains and unaligned arrays. Exact."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
BITS_MAX_N = 130 * 1024 * 8


def _dev(a, shift=0):
    buf = torch.empty(len(a) + shift, dtype=torch.int32, device=DEV)
    buf[shift:] = torch.from_numpy(np.ascontiguousarray(a, np.int32)).to(DEV)
    return buf[shift:]


def _check(src, dst, n, shift=0):
    got = lrcc.cc_label(_dev(src, shift), _dev(dst, shift), n)
    lrcc.check()
    assert np.array_equal(got.cpu().numpy(), oracle.cc_uf(src, dst, n))


@pytest.mark.parametrize("n,m", [(2, 1), (1023, 1024), (49152, 24576), (49153, 24576), (49152, 24577), (20_000, 24_575),
                                 (50_001, 0), (70_001, 70_003), (262_144, 524_287), (262_144, 524_288),
                                 (300_007, 600_013)])
@pytest.mark.parametrize("shift", [0, 1])
def test_uniform_graphs_around_the_limits(n, m, shift):
    _check(*gen.er(n, m, n + m), n, shift)


@pytest.mark.parametrize("n", [BITS_MAX_N - 1, BITS_MAX_N, BITS_MAX_N + 1])
def test_membership_tables(n):
    _check(*gen.er(n, 2 * n + 3, 5), n)                    # bit map up to BITS_MAX_N, none above (uniform)
    src, dst = gen.rmat(21, 9 << 20, 0.57, 0.19, 0.19, 6)    # skewed: cache of members above BITS_MAX_N
    _check(src % n, dst % n, n, 1)


def test_skewed_graph_of_long_passes():
    src, dst = gen.rmat(21, 16 << 21, 0.57, 0.19, 0.19, 7)   # one pass over the sample, every edge filtered
    _check(src, dst, 1 << 21)


@pytest.mark.parametrize("n", [40_000, 400_000])
def test_stars_and_hot_roots(n):
    rng = np.random.default_rng(n)
    ids = rng.permutation(n)
    leaves = ids[1:]
    _check(np.full(n - 1, ids[0]), leaves, n)                                   # one star
    hubs = rng.choice(ids[:3], n - 3)                                           # three stars, then joined
    _check(np.concatenate([hubs, ids[:2]]), np.concatenate([ids[3:], ids[1:3]]), n)
    # a large component without the smallest ids, then one edge from each of them into it
    low = n // 8
    s, d = rng.integers(low, n, 4 * n), rng.integers(low, n, 4 * n)
    _check(np.concatenate([s, np.arange(low)]), np.concatenate([d, rng.integers(low, n, low)]), n)


@pytest.mark.parametrize("n", [30_000, 200_000, 3_000_000])
def test_consecutive_ids_in_both_edge_orders(n):
    e = np.arange(n - 1)
    _check(e, e + 1, n)
    _check(e[::-1] + 1, e[::-1], n)
    _check(e // 2, e + 1, n)                                                    # a binary heap
    _check(np.repeat(e[: n // 4], 3), np.repeat(e[: n // 4] + 1, 3), n)         # repeated edges, isolated vertices


def test_ids_out_of_range_are_reported():
    for n, m in ((1000, 2000), (300_000, 700_000)):
        src, dst = gen.er(n, m, 3)
        for bad in (n, -1):
            wrong = src.copy()
            wrong[m // 2] = bad
            lrcc.cc_label(_dev(wrong), _dev(dst), n)
            assert lrcc.last_status() == lrcc.ERR_INVALID_INPUT
        _check(src, dst, n)


@pytest.mark.parametrize("sample", [2, 3, 7])
def test_sample_given_by_the_plan(sample):
    lrcc.set_cc_plan(0, 32, cc_sample=sample)
    try:
        src, dst, n = gen.list_graph(5, 50_000, 8)      # the sample holds whole paths and a piece of one
        _check(src, dst, n)
        _check(*gen.er(1 << 17, 1 << 19, 9), 1 << 17, 1)
    finally:
        lrcc.reset_plans()


@pytest.mark.slow
def test_more_pairs_than_the_buffer_holds():
    # 10^8 edges of a sparse graph keep more than 2^26 pairs after the first passes:
    # the warps read their ranges of the edge list again
    lrcc.set_cc_plan(0, 32, cc_hook=1, cc_sample=1)
    try:
        n = 1 << 26
        _check(*gen.er(n, 100_000_000, 10), n)
    finally:
        lrcc.reset_plans()


def test_calls_on_several_streams_at_once():
    graphs = [(n, *gen.er(n, m, k)) for k, (n, m) in enumerate([(1000, 1500), (200_000, 500_000), (1 << 20, 1 << 22)])]
    on_dev = [(n, _dev(s), _dev(d), oracle.cc_uf(s, d, n)) for n, s, d in graphs]
    streams = [torch.cuda.Stream() for _ in range(4)]
    torch.cuda.synchronize()
    out = []
    for rep in range(6):
        for k, st in enumerate(streams):
            n, s, d, want = on_dev[(rep + k) % len(on_dev)]
            with torch.cuda.stream(st):
                out.append((lrcc.cc_label(s, d, n, stream=st), want))
    for st in streams:
        lrcc.check(st)
    for got, want in out:
        assert np.array_equal(got.cpu().numpy(), want)
    for st in streams:
        lrcc.release(st)
