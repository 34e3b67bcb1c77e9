"""Components within the queried workspace (about 2 bytes per edge), on a reserved stream
and where a larger one cannot be had. Exact."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
GRAPHS = {"sparse": (1 << 22, 1 << 22), "sparse_small": (60_000, 60_000), "two": (300_007, 600_013), "four": (1 << 20, 1 << 22)}


@pytest.mark.parametrize("graph", GRAPHS)
@pytest.mark.parametrize("how", ["reserved", "no_room"])
def test_labels_with_the_least_room(graph, how):
    n, m = GRAPHS[graph]
    src, dst = gen.er(n, m, n)
    a, b = (torch.from_numpy(x).to(DEV) for x in (src, dst))
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    need = lrcc.workspace_query(lrcc.KIND_CC, n, m)
    assert need <= 2 * m + (6 << 20)          # (at least one iteration of pairs for every warp)
    if how == "reserved":
        with lrcc.Context(0) as ctx:
            ctx.reserve(stream, need)
            held = ctx.bytes()
            label = lrcc.cc_label(a, b, n, stream=stream)
            lrcc.check(stream)
            assert ctx.bytes() == held
    else:
        lrcc.last_status(stream)                  # the stream's status word is allocated
        lrcc.debug_fail_allocs(1)
        try:
            label = lrcc.cc_label(a, b, n, stream=stream)
            lrcc.check(stream)
        finally:
            lrcc.debug_fail_allocs(0)
            lrcc.release(stream)
    assert np.array_equal(label.cpu().numpy(), oracle.cc_uf(src, dst, n))
