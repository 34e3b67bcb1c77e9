"""Batched components (hook rule 1) whose offsets do not describe the arrays of the
call: reported, and the next call is sound."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SIZES = [70_001, 300, 60_000, 40_000]


def _call(src, dst, eoff, voff):
    a, b, eo, vo = (torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in (src, dst, eoff, voff))
    lab = lrcc.cc_label_batched(a, b, eo, vo, n_total=sum(SIZES))
    return lrcc.last_status(), lab.cpu().numpy()


@pytest.mark.parametrize("case", ["vertices_decrease", "edges_decrease", "first_vertex", "first_edge", "edges_past_the_end"])
def test_offsets_that_name_no_graphs(case):
    src, dst, eoff, voff = gen.er_batch(np.asarray(SIZES, np.int64), 3, 1, 6)
    e, v = eoff.copy(), voff.copy()
    if case == "vertices_decrease":
        v[1] = voff[2] + 9
    elif case == "edges_decrease":
        e[2] = eoff[1] - 9
    elif case == "first_vertex":
        v[0] = 3
    elif case == "first_edge":
        e[0] = 3
    else:
        e[-1] = eoff[-1] + 50_000
    status, _ = _call(src, dst, e, v)
    assert status == lrcc.ERR_INVALID_INPUT
    # sound offsets, and edges behind the last graph's that belong to none
    more = np.zeros(1000, src.dtype)
    status, lab = _call(np.concatenate([src, more]), np.concatenate([dst, more]), eoff, voff)
    assert status == lrcc.OK
    for k, n in enumerate(SIZES):
        s, d = src[eoff[k]:eoff[k + 1]], dst[eoff[k]:eoff[k + 1]]
        assert np.array_equal(lab[voff[k]:voff[k + 1]], oracle.cc_uf(s, d, n))


@pytest.mark.parametrize("case", ["vertices_decrease", "edges_decrease", "edges_past_the_end"])
def test_the_other_graphs_are_labelled(case):
    sizes = [70_001, 300, 60_000, 40_000, 50, 30_000]
    src, dst, eoff, voff = gen.er_batch(np.asarray(sizes, np.int64), 3, 1, 6)
    e, v = eoff.copy(), voff.copy()
    touched = {1, 2}                              # bounded by offset 2
    if case == "vertices_decrease":
        v[2] = voff[3] + 9                        # graph 1 runs over graph 2 into graph 3
        touched.add(3)
    elif case == "edges_decrease":
        e[2] = eoff[1] - 9
    else:
        e[2] = eoff[-1] + 50_000
    a, b, eo, vo = (torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in (src, dst, e, v))
    lab = lrcc.cc_label_batched(a, b, eo, vo, n_total=sum(sizes)).cpu().numpy()
    assert lrcc.last_status() == lrcc.ERR_INVALID_INPUT
    for k in set(range(len(sizes))) - touched:
        s, d = src[eoff[k]:eoff[k + 1]], dst[eoff[k]:eoff[k + 1]]
        assert np.array_equal(lab[voff[k]:voff[k + 1]], oracle.cc_uf(s, d, sizes[k])), k
