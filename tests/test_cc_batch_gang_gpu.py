"""Batched components, hook rule 1: graphs on both sides of the one-block limit,
sampled and not, in batches that make one gang or many. Exact."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _run(graphs):
    voff = np.cumsum([0] + [n for n, _, _ in graphs])
    eoff = np.cumsum([0] + [len(s) for _, s, _ in graphs])
    src = np.concatenate([s for _, s, _ in graphs]).astype(np.int32)
    dst = np.concatenate([d for _, _, d in graphs]).astype(np.int32)
    a, b, eo, vo = (torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in (src, dst, eoff, voff))
    lab = lrcc.cc_label_batched(a, b, eo, vo, n_total=int(voff[-1]))
    return lab.cpu().numpy(), [oracle.cc_uf(s, d, n) if n else np.zeros(0, np.int32) for n, s, d in graphs]


def _er(n, m, seed):
    return (n, *gen.er(n, m, seed))


def _check(graphs):
    got, want = _run(graphs)
    lrcc.check()
    assert np.array_equal(got, np.concatenate(want))


@pytest.mark.parametrize("n,m", [(16384, 65536), (16385, 65536), (16384, 65537), (16385, 0), (30_000, 59_999),
                                 (30_000, 60_000), (70_001, 140_003), (1 << 20, 3 << 20)])
def test_one_graph_alone_and_between_small_ones(n, m):
    small = [_er(5, 3, 1), (0, np.zeros(0, np.int32), np.zeros(0, np.int32)), _er(1, 2, 2), _er(1000, 999, 3)]
    _check([_er(n, m, 4)])
    _check(small[:2] + [_er(n, m, 5)] + small[2:])


def test_many_sizes_and_families():
    rng = np.random.default_rng(3)
    graphs = []
    for k in range(60):
        n = int(2 ** rng.uniform(3, 18))
        kind = k % 5
        if kind == 0:
            graphs.append(_er(n, 2 * n, k))
        elif kind == 1:
            graphs.append(_er(n, n // 2 + 1, k))
        elif kind == 2:                       # a path of consecutive ids
            graphs.append((n, np.arange(n - 1), np.arange(1, n)))
        elif kind == 3:                       # a star with a random centre
            c = int(rng.integers(n))
            graphs.append((n, np.full(n, c), np.arange(n)))
        else:                                 # dense
            graphs.append(_er(n, 8 * n, k))
    _check(graphs)
    _check([g for g in graphs if g[0] > 16384] * 3)


def test_bad_ids_are_reported_and_others_labelled():
    graphs = [_er(20_000, 50_000, 1), _er(300, 500, 2), _er(40_000, 90_000, 3)]
    for bad in range(3):
        broken = [(n, s.copy(), d.copy()) for n, s, d in graphs]
        broken[bad][1][7] = broken[bad][0]
        voff = np.cumsum([0] + [n for n, _, _ in broken])
        broken_ok = [(n, s, d) for n, s, d in broken]
        args = [np.concatenate([s for _, s, _ in broken_ok]), np.concatenate([d for _, _, d in broken_ok]),
                np.cumsum([0] + [len(s) for _, s, _ in broken_ok]), voff]
        a, b, eo, vo = (torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in args)
        lab = lrcc.cc_label_batched(a, b, eo, vo, n_total=int(voff[-1])).cpu().numpy()
        assert lrcc.last_status() == lrcc.ERR_INVALID_INPUT
        for k, (n, s, d) in enumerate(graphs):
            if k != bad:
                assert np.array_equal(lab[voff[k]:voff[k + 1]], oracle.cc_uf(s, d, n))
    _check(graphs)
