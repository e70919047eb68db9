"""The joined work-lists of row-or-column plans: one launch does the three passes, so a part of a split unit, its counters
and its partial results, padding and empty halves of every pass share one list.  Against the fp32 kernels' three launches
(the same plan, no work-lists) on sizes where the passes' lists differ most."""
import numpy as np
import pytest
import torch

from tests import helpers as hp
from tests.test_gpu_parity import custom_case

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
        for _ in range(2):          # the counters of the split units are back at zero after a launch
            O, LSE = m.mate_attn_fwd(plan, Q, K, V, None, impl)
            got[impl] = (O, LSE) + tuple(m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO, None, impl))
    torch.cuda.synchronize()
    plan.status()
    atol, rtol = hp.tol("bf16")     # of either side against exact values: twice that between them
    for name, a, b in zip(("O", "LSE", "dQ", "dK", "dV"), got[m.IMPL_TCGEN05], got[m.IMPL_SIMT]):
        a, b = (x.float().cpu().numpy().astype(np.float64) for x in (a, b))
        on = np.isfinite(b)
        assert np.array_equal(on, np.isfinite(a)), name
        hp.assert_close(a[on], b[on], 2 * atol, 2 * rtol, name)
    plan.destroy()
