"""The joined work-lists of row-or-column plans: one launch does the three passes, so a part of a split unit, its counters
and its partial results, padding and empty halves of every pass share one list.  On sizes where the passes' lists differ
most, against the fp32 kernels' three launches (the same plan, no work-lists); and with several items per CTA, those of two tiles, of
one and without a tile behind one another, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from tests import helpers as hp
from tests.test_gpu_parity import custom_case
from workloads import tables

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["split units", "single tokens", "padding only", "column longer than a tile"])
def test_one_launch_equals_three(what):
    import paper_2109_04312_b200 as m
    if what == "split units":       # one example, few heads: the long global rows are cut into parts in several passes
        case = custom_case(300, [(r, c, 5) for r in range(1, 121) for c in range(1, 7)], 300 + 5 * 720)
    elif what == "single tokens":   # every cell one token: no pass has two tokens of a cell
        case = custom_case(3, [(r, c, 1) for r in range(1, 14) for c in range(1, 12)], 160)
    elif what == "padding only":    # an example without a valid table token
        case = custom_case(1, [], 130)
    else:                           # own rows of a column pass meet several tiles in front and behind
        case = custom_case(17, [(r, 1, 33) for r in range(1, 20)], 17 + 33 * 19 + 1)
    cfg, rows, cols, vals = case
    plan = m.mate_plan_sat(torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda(), cfg.P, cfg.H)
    Q, K, V, dO = (hp.to_dev(vals[n], "bf16") for n in ("Q", "K", "V", "dO"))
    got = {}
    for impl in (m.IMPL_TCGEN05, m.IMPL_SIMT):
        for i in range(2):          # the counters of the split units are back at zero after a launch
            O, LSE = m.mate_attn_fwd(plan, Q, K, V, None, impl)
            outs = (O, LSE) + tuple(m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO, None, impl))
            assert i == 0 or all(torch.equal(a, b) for a, b in zip(got[impl], outs))
            got[impl] = outs
    torch.cuda.synchronize()
    plan.status()
    atol, rtol = hp.tol("bf16")     # of either side against exact values: twice that between them
    for name, a, b in zip(("O", "LSE", "dQ", "dK", "dV"), got[m.IMPL_TCGEN05], got[m.IMPL_SIMT]):
        a, b = (x.float().cpu().numpy().astype(np.float64) for x in (a, b))
        on = np.isfinite(b)
        assert np.array_equal(on, np.isfinite(a)), name
        hp.assert_close(a[on], b[on], 2 * atol, 2 * rtol, name)
    plan.destroy()


def small_table(e, P):
    n = 60 + 11 * e % 120       # table tokens of an ordinary one
    if e % 4 == 0:              # two tokens per cell
        return [(r, c, 2) for r in range(1, 2 + n // 10) for c in range(1, 6)]
    if e % 4 == 1:              # one row: nothing in front of or behind a cell, in any column
        return [(1, c, 9) for c in range(1, 2 + n // 9)]
    if e % 4 == 2:              # one cell
        return [(1, 1, n)]
    return [(r, 1, 1) for r in range(1, 129 - P)] + [(200, 2, 1 + n // 3)]   # the last half is one cell


def test_many_small_examples():
    import paper_2109_04312_b200 as m
    B, H, P, N = 32, 12, 10, 256
    parts = [tables.custom_structure(P, small_table(e, P), N) for e in range(B)]
    rows, cols = (np.concatenate([p[i] for p in parts]) for i in (0, 1))
    cfg = tables.TableConfig("custom", B, H, H // 2, 64, N, P, 0, 0, "uniform", 1, 1, "bf16", 0.5)
    vals = tables.make_values(cfg, N, 3)
    hv, scale = np.full(H, 2, np.uint8), 0.125
    plan = m.mate_plan_sat(torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda(), P, H)
    Q, K, V, dO = (hp.to_dev(vals[n], "bf16") for n in ("Q", "K", "V", "dO"))
    first = None
    for _ in range(20):
        O, LSE = m.mate_attn_fwd(plan, Q, K, V, scale, m.IMPL_TCGEN05)
        got = (O, LSE) + tuple(m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO, scale, m.IMPL_TCGEN05))
        first = first or got
        for name, a, b in zip(("O", "LSE", "dQ", "dK", "dV"), first, got):
            assert torch.equal(a, b), name
    plan.status()
    want = oracle.fwd(vals["Q"], vals["K"], vals["V"], rows, cols, P, hv, scale) + \
        tuple(oracle.bwd(vals["Q"], vals["K"], vals["V"], vals["dO"], rows, cols, P, hv, scale))
    atol, rtol = hp.tol("bf16")
    for name, g, o in zip(("O", "LSE", "dQ", "dK", "dV"), first, want):
        g, on = hp.to_np(g), np.isfinite(o)
        assert np.array_equal(on, np.isfinite(g)), name
        hp.assert_close(g[on], o[on], atol, rtol, name)
    plan.destroy()
