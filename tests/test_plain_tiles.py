"""Edges of the tiles of the kernels without tensor cores (32 rows, 64 columns, two groups that take the tiles in turn,
columns that a warp leaves out): forward and backward in fp32 against the oracle."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


# prefix, rows, cols, tokens per cell, padding: no second tile; one column more than a tile; rows of 2 / 17 / 70 tokens, so that
# a warp's columns begin and end in every group of 16; prefixes of 63, 64, 65 and 129; an odd and an even number of tiles
@pytest.mark.parametrize("d", [8, 40, 64, 128])
@pytest.mark.parametrize("P,rows,cols,cell,pad", [
    (1, 3, 2, 1, 0), (8, 8, 7, 1, 1), (9, 8, 7, 1, 0), (63, 30, 2, 1, 5), (64, 7, 17, 1, 0), (65, 3, 35, 2, 3), (129, 40, 5, 1, 31)])
def test_tile_edges(P, rows, cols, cell, pad, d):
    import paper_2109_04312_b200 as mate
    N, B, H = P + rows * cols * cell + pad, 2, 2
    ids = np.full((2, B, N), -1, np.int32)
    ids[:, :, :P] = 0
    ids[0, :, P:N - pad] = np.repeat(np.arange(1, rows + 1), cols * cell)
    ids[1, :, P:N - pad] = np.tile(np.repeat(np.arange(1, cols + 1), cell), rows)
    rng = np.random.default_rng(N + d)
    Q, K, V, dO = (rng.standard_normal((B, H, N, d)).astype(np.float32) * 0.5 for _ in range(4))
    scale, hv = 1.0 / np.sqrt(d), [0, 1]
    plan = mate.mate_plan(torch.from_numpy(ids[0]).cuda(), torch.from_numpy(ids[1]).cuda(), P, hv, rows, cols)
    q, k, v, do = (torch.from_numpy(x).cuda() for x in (Q, K, V, dO))
    O, LSE = mate.mate_attn_fwd(plan, q, k, v, scale)
    got = (O,) + tuple(mate.mate_attn_bwd(plan, q, k, v, O, LSE, do, scale))
    oO, _ = oracle.fwd(Q, K, V, ids[0], ids[1], P, hv, scale)
    ref = (oO,) + tuple(oracle.bwd(Q, K, V, dO, ids[0], ids[1], P, hv, scale))
    # fp32 sums of at most 300 terms of order one and below: 300 x 2^-24 x 0.5 is 9e-6 if all roundings went one way
    for g, r, name in zip(got, ref, ("O", "dQ", "dK", "dV")):
        err = np.abs(g.cpu().numpy().astype(np.float64) - r)
        assert np.all(err <= 1e-5 + 1e-5 * np.abs(r)), (name, err.max())
