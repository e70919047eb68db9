"""Gradients of padding rows, which warps of their own zero: sequences that are nearly all padding, with more chunks of 64 padding
rows than CTAs, and chunks and rows left over.  The memory that the gradients get holds NaN before."""
import numpy as np
import pytest
import torch

from tests import helpers as hp
from workloads import tables

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,N,sat", [(4, 4, 5000, False), (1, 2, 193, False), (2, 2, 3001, True), (3, 12, 1063, False)])
def test_mostly_padding(B, H, N, sat):
    import paper_2109_04312_b200 as m
    P, cells = 5, [(r, c, 2) for r in range(1, 13) for c in range(1, 6)]
    rows, cols = (np.repeat(x, B, axis=0) for x in tables.custom_structure(P, cells, N))
    r, c = torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda()
    plan = m.mate_plan_sat(r, c, P, H) if sat else m.mate_plan(r, c, P, [h % 2 for h in range(H)], 12, 5)
    g = torch.Generator(device="cuda").manual_seed(N)
    Q, K, V, dO = ((torch.randn((B, H, N, 64), device="cuda", generator=g) * 0.5).to(torch.bfloat16) for _ in range(4))
    O, LSE = m.mate_attn_fwd(plan, Q, K, V, None, m.IMPL_TCGEN05)
    ref = m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO, None, m.IMPL_SIMT)
    dirty = [torch.full_like(Q, float("nan")) for _ in range(6)]
    del dirty  # (the allocator hands the same memory out again)
    got = m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO, None, m.IMPL_TCGEN05)
    torch.cuda.synchronize()
    plan.status()
    pad = torch.from_numpy(rows < 0).cuda()[:, None, :, None].expand_as(Q)
    atol, rtol = hp.tol("bf16")  # of either side against exact values: twice that between them
    for name, a, b in zip(("dQ", "dK", "dV"), got, ref):
        assert torch.all(a[pad] == 0), name
        hp.assert_close(hp.to_np(a), hp.to_np(b), 2 * atol, 2 * rtol, name)
    plan.destroy()
