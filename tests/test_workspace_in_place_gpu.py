"""The queried workspace covers every call of its kind and size: ranks written over
the successors, and splitters given by the caller, as well as ranks of their own."""
import numpy as np
import pytest
import torch

import gen
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n", [16_385, 100_003, 1 << 20, 1 << 24, (1 << 24) + 1])
@pytest.mark.parametrize("how", ["apart", "in_place", "overlapping", "splitters"])
def test_reserved_stream_does_not_grow(n, how):
    succ, head, perm = gen.list_random(n, 5, with_perm=True)
    stream = torch.cuda.Stream()
    with lrcc.Context(0) as ctx, torch.cuda.stream(stream):
        ctx.reserve(stream, lrcc.workspace_query(lrcc.KIND_LR, n))
        held = ctx.bytes()
        buf = torch.empty(n + 1, dtype=torch.int32, device=DEV)
        src = buf[:n]
        src.copy_(torch.from_numpy(succ))
        out = {"apart": torch.empty_like(src), "in_place": src, "overlapping": buf[1:]}.get(how)
        if how == "splitters":
            spl = torch.from_numpy(np.ascontiguousarray(perm[::16])).to(DEV)
            out = lrcc.lr_rank_splitters(src, head, spl, stream=stream)
        else:
            lrcc.lr_rank(src, head, out=out, stream=stream)
        assert ctx.last_status(stream) == lrcc.OK
        assert ctx.bytes() == held
        assert np.array_equal(out.cpu().numpy()[perm], np.arange(n - 1, -1, -1, dtype=np.int32))
