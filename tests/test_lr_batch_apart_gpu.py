"""Batched lists that cannot all be ranked together, in totals of at most 2^24
elements: a list that is none spoils only its own ranks, and elements behind the
last list are left alone. Exact."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
M = 1 << 20
MIXES = {"blocks": [300, 9000, 24_577, 0, 77], "together": [40_000, 0, 24_576, 60_000, 1, 24_577, 30_000],
         "limit": [4 * M - 1, 4 * M, 1, 8 * M]}


def _call(succ, off, heads, shift=0):
    buf = torch.empty(len(succ) + shift, dtype=torch.int32, device=DEV)
    buf[shift:] = torch.from_numpy(succ).to(DEV)
    out = torch.full((len(succ) + shift,), -7, dtype=torch.int32, device=DEV)[shift:]
    lrcc.lr_rank_batched(buf[shift:], torch.from_numpy(off).to(DEV), torch.from_numpy(heads).to(DEV), out=out)
    return lrcc.last_status(), out.cpu().numpy()


def _batch(mix):
    succ, off, heads = gen.list_batch(np.asarray(MIXES[mix], np.int64), len(mix))
    return succ.astype(np.int32), off.astype(np.int64), heads.astype(np.int32)


@pytest.mark.parametrize("mix", MIXES)
@pytest.mark.parametrize("case", ["cycle", "two_lists", "named_twice", "succ_out_of_range", "head_out_of_range"])
def test_one_bad_list(mix, case):
    succ, off, heads = _batch(mix)
    want = oracle.lr_rank_batched(succ, off, heads)
    k = 1 if MIXES[mix][1] > 2 else 3
    b, e = int(off[k]), int(off[k + 1])
    tail = b + int(np.flatnonzero(succ[b:e] == -1)[0])
    if case == "cycle":
        succ[tail] = heads[k]
    elif case == "two_lists":
        succ[b + heads[k]] = -1
    elif case == "named_twice":
        succ[tail] = succ[b + heads[k]]          # a cycle with the head leading into it
    elif case == "succ_out_of_range":
        succ[tail] = e - b
    else:
        heads[k] = e - b
    status, got = _call(succ, off, heads)
    assert status == lrcc.ERR_INVALID_INPUT
    assert np.array_equal(got[:b], want[:b]) and np.array_equal(got[e:], want[e:])


@pytest.mark.parametrize("mix", MIXES)
@pytest.mark.parametrize("pad", [1, 4097, 200_000])
@pytest.mark.parametrize("shift", [0, 1])
def test_elements_behind_the_last_list(mix, pad, shift):
    succ, off, heads = _batch(mix)
    total = int(off[-1])
    if total + pad > 1 << 24:
        off = off[:-1]                            # without its last list: up to 2^24 elements with the others
        heads, succ, total = heads[:-1], succ[:off[-1]], int(off[-1])
    status, got = _call(np.concatenate([succ, np.full(pad, 5, np.int32)]), off, heads, shift)
    assert status == lrcc.OK
    assert np.array_equal(got[:total], oracle.lr_rank_batched(succ, off, heads))
    assert (got[total:] == -7).all()


@pytest.mark.parametrize("sizes,k", [([300, 9000, 24_577, 77, 500, 30_000, 900] + [100] * 5, 3),  # one block per list
                                     ([40_000, 24_576, 60_000, 24_577, 30_000, 50_000], 2)])      # together
@pytest.mark.parametrize("case", ["decreasing", "overlapping", "past_the_end", "first_not_zero", "negative"])
def test_one_bad_offset(sizes, k, case):
    succ, off, heads = (a.astype(t) for a, t in zip(gen.list_batch(np.asarray(sizes, np.int64), 8),
                                                    (np.int32, np.int64, np.int32)))
    want, good = oracle.lr_rank_batched(succ, off, heads), off.copy()
    touched = {k - 1, k}                          # the lists that the offset bounds
    if case == "decreasing":
        off[k] = good[k - 1] - 9                  # list k also runs over the end of list k - 2
        touched.add(k - 2)
    elif case == "overlapping":
        off[k] = good[k + 1] + 5                  # list k - 1 runs into list k + 1
        touched.add(k + 1)
    elif case == "past_the_end":
        off[k] = good[-1] + 1000
    elif case == "first_not_zero":
        off[0] = 2
        touched = {0}
    else:
        off[k] = -5
    status, got = _call(succ, off, heads)
    assert status == lrcc.ERR_INVALID_INPUT
    for i in set(range(len(sizes))) - touched:
        assert np.array_equal(got[good[i]:good[i + 1]], want[good[i]:good[i + 1]]), i
