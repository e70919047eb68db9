"""Sizes at which the kernels take another branch or a tile is partly filled: work units of the tensor-core
kernels (global block in front of the own keys, halves filled up with table rows, units cut along their
tiles), the tiled fp32 kernels, the cell mean's buffers, plan memory reused between streams; what must not
reach a result: values at padding and of a packed neighbour, and the time of the kernel before."""
import numpy as np
import pytest
import torch

import oracle
from tests import helpers as hp
from workloads import tables

pytestmark = pytest.mark.gpu


def _check(rows, cols, P, hv, d, dtype, seed, pad=0):
    import paper_2109_04312_b200 as m
    if pad:
        rows, cols = (np.concatenate([x, np.full((x.shape[0], pad), -1, np.int32)], 1) for x in (rows, cols))
    B, N = rows.shape
    rng = np.random.default_rng(seed)
    vals = {n: (rng.standard_normal((B, len(hv), N, d)) * 0.5).astype(np.float32) for n in ("Q", "K", "V", "dO")}
    if dtype == "bf16":
        vals = {n: tables.round_to_bf16(v) for n, v in vals.items()}
    plan = m.mate_plan(torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda(), P, hv)
    Q, K, V, dO = (hp.to_dev(vals[n], dtype) for n in ("Q", "K", "V", "dO"))
    scale = 1.0 / np.sqrt(d)
    O, LSE = m.mate_attn_fwd(plan, Q, K, V)
    grads = m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO)
    torch.cuda.synchronize()
    plan.status()
    hv = np.asarray(hv, np.uint8)
    oO, oL = oracle.fwd(vals["Q"], vals["K"], vals["V"], rows, cols, P, hv, scale)
    og = oracle.bwd(vals["Q"], vals["K"], vals["V"], vals["dO"], rows, cols, P, hv, scale)
    assert np.array_equal(plan.useful_pairs(), oracle.useful_pairs(rows, cols, P, hv))
    atol, rtol = hp.tol(dtype)
    valid = np.broadcast_to((rows >= 0)[:, None, :], oL.shape)
    hp.assert_close(hp.to_np(O), oO, atol, rtol, "O")
    hp.assert_close(hp.to_np(LSE)[valid], oL[valid], atol, rtol, "LSE")
    for name, g, o in zip(("dQ", "dK", "dV"), grads, og):
        hp.assert_close(hp.to_np(g), o, atol, rtol, name)


def _structure(P, n_table, row_len, n_cols, seed):
    """P prefix tokens, then n_table table tokens: rows of about row_len tokens, columns drawn at random."""
    rng = np.random.default_rng(seed)
    r = np.concatenate([np.zeros(P, np.int32), 1 + np.arange(n_table, dtype=np.int32) // row_len])
    c = np.concatenate([np.zeros(P, np.int32), rng.integers(1, n_cols + 1, n_table).astype(np.int32)])
    return r[None, :].astype(np.int32), c[None, :].astype(np.int32)


@pytest.mark.parametrize("P,n_table,row_len,n_cols,pad", [
    (1, 0, 1, 1, 0), (0, 1, 1, 1, 3), (20, 107, 9, 4, 1), (20, 108, 9, 4, 0), (20, 109, 9, 4, 0),   # around 128 positions
    (100, 155, 40, 3, 0), (100, 156, 40, 3, 0), (100, 157, 40, 3, 0),                                # around 256
    (64, 300, 64, 2, 5), (116, 400, 12, 5, 0), (127, 260, 130, 2, 0), (128, 256, 128, 2, 0), (129, 255, 17, 2, 0),
    (383, 129, 33, 3, 0), (384, 200, 33, 3, 0), (16, 2500, 700, 2, 0)])
def test_tensor_core_unit_edges(P, n_table, row_len, n_cols, pad):
    rows, cols = _structure(P, n_table, row_len, n_cols, P + n_table)
    _check(rows, cols, P, [0, 1, 1], 64, "bf16", 7, pad)


def test_tensor_core_units_that_are_cut_and_a_busy_grid():
    rows, cols = _structure(130, 2900, 40, 3, 5)    # few heads: the global rows' units are cut along their tiles
    _check(rows, cols, 130, [0, 1], 64, "bf16", 8)
    rows, cols = _structure(70, 330, 25, 4, 6)      # many heads: halves of the global block filled up with table rows
    rows, cols = np.repeat(rows, 3, 0), np.repeat(cols, 3, 0)
    _check(rows, cols, 70, [0, 1] * 26, 64, "bf16", 9)


# x 37 positions: around one and two rows per thread on 148 SMs, with six and with eight blocks to an SM
@pytest.mark.parametrize("H", [768, 769, 1024, 1025, 1536, 1537, 2048, 2049])
def test_row_dots_of_every_size(H):
    rows, cols = _structure(5, 31, 4, 3, 11)
    _check(rows, cols, 5, [0, 1, 0] * (H // 3) + [1] * (H % 3), 64, "bf16", 12, 1)


# On both sides of where the tensor-core backward stops dividing by the scale, and the scales in use.  Q and K are scaled by powers of two so
# that the scores stay what they are, and the gradients are compared by 2-norm, so that those of a tiny scale count as much.
# Bound: P, dS (or O in D) and the result rounded to bf16, 2^-9 each and independent of one another; row or column: two more, the
# gradients of the passes and their sum.
@pytest.mark.parametrize("kind", ["exact", "sat"])
@pytest.mark.parametrize("scale", [0.0, 2.0 ** -120, 2.0 ** -101, 2.0 ** -99, -2.0 ** -101, -0.125, 1.5, 2.0 ** 99, 2.0 ** 101])
def test_backward_takes_every_scale(scale, kind):
    import paper_2109_04312_b200 as m
    rows, cols = _structure(20, 300, 30, 4, 13)
    hv, rng = np.array([2, 2] if kind == "sat" else [0, 1], np.uint8), np.random.default_rng(14)
    vals = {n: tables.round_to_bf16((rng.standard_normal((1, 2, 320, 64)) * 0.5).astype(np.float32)) for n in ("Q", "K", "V", "dO")}
    e = -3 - int(np.floor(np.log2(abs(scale)))) if scale else 0
    vals["Q"], vals["K"] = np.ldexp(vals["Q"], e // 2), np.ldexp(vals["K"], e - e // 2)
    r, c = torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda()
    plan = m.mate_plan_sat(r, c, 20, 2) if kind == "sat" else m.mate_plan(r, c, 20, hv)
    Q, K, V, dO = (hp.to_dev(vals[n], "bf16") for n in ("Q", "K", "V", "dO"))
    O, LSE = m.mate_attn_fwd(plan, Q, K, V, scale)
    auto, forced, simt = (m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO, scale, i) for i in (m.IMPL_AUTO, m.IMPL_TCGEN05, m.IMPL_SIMT))
    plan.status()
    want = oracle.bwd(vals["Q"], vals["K"], vals["V"], vals["dO"], rows, cols, 20, hv, scale)
    bound = (5 if kind == "sat" else 3) ** 0.5 * 2.0 ** -9
    for name, a, f, s, w in zip(("dQ", "dK", "dV"), auto, forced, simt, want):
        assert torch.equal(a, f), name
        for g in (f, s):
            assert np.linalg.norm(hp.to_np(g) - w) <= bound * np.linalg.norm(w), name
        # P and dS are rounded on the tensor cores only: the implementation that was asked for has run
        assert not np.any(w) or not torch.equal(f, s), name


@pytest.mark.parametrize("q0,v0", [(0.0, 0.0), (8192.0, 0.0), (0.0, 64.0), (8192.0, 64.0)])
@pytest.mark.parametrize("P,n_table,row_len", [(20, 300, 30), (130, 254, 254)])
def test_key_side_keeps_the_low_bits_of_lse_and_d(P, n_table, row_len, q0, v0):
    # A component of its own takes LSE / scale to 8192 (LSE to 1024) or D to 4096 in front of scores and differences dP - D of a few
    # units.  dK and dV against 64 bits given the same O and LSE: 2.3e-3 to 2.4e-3 of their norm, 1.3e-2 to 2.3e-2 where the last 8 of the
    # 24 bits of either are left out.  Bound: P (or dS) and the result rounded to bf16, 2^-9 each, and as much for S and dP, whose
    # last bits are 2^-10 in fp32.
    import paper_2109_04312_b200 as m
    rows, cols = _structure(P, n_table, row_len, 4, 16)
    r, c = torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda()
    plan, scale, n = m.mate_plan(r, c, P, [0, 1]), 0.125, P + n_table
    gen = torch.Generator(device="cuda").manual_seed(17)
    Q, K, V, dO = ((torch.randn(1, 2, n, 64, device="cuda", generator=gen) * 0.5).bfloat16() for _ in range(4))
    if q0:
        Q[..., 0], K[..., 0] = q0, 1.0
    if v0:
        V[..., 0], dO[..., 0] = v0, v0
    O, LSE = m.mate_attn_fwd(plan, Q, K, V, scale, m.IMPL_TCGEN05)
    _, dK, dV = m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO, scale, m.IMPL_TCGEN05)
    plan.status()
    ids, pre = torch.stack([r[0], c[0]]), torch.arange(n, device="cuda") < P
    on = pre[:, None] | pre[None, :] | (ids[:, :, None] == ids[:, None, :])
    Q, K, V, dO, O = (x[0].double() for x in (Q, K, V, dO, O))
    p = torch.exp(scale * Q @ K.transpose(1, 2) - LSE[0].double()[..., None]) * on
    ds = p * (dO @ V.transpose(1, 2) - (dO * O).sum(-1, keepdim=True))
    for name, g, w in (("dK", dK, scale * ds.transpose(1, 2) @ Q), ("dV", dV, p.transpose(1, 2) @ dO)):
        g, w = g[0, :, :, 1:].double(), w[:, :, 1:]  # (without the component that is as large as that)
        assert (g - w).norm() <= 3.0 ** 0.5 * 2.0 ** -9 * w.norm(), (name, float((g - w).norm() / w.norm()))


@pytest.mark.parametrize("at", [[130], [5, 130]])  # a row of the table; one of the prefix too, which every other row meets
@pytest.mark.parametrize("kind", ["exact", "sat"])
def test_a_query_without_a_finite_score(kind, at):
    # All scores of some valid queries are -inf (products of -2^200), so their LSE is -inf as well: their weights are not numbers
    # on either side of the backward, whichever kernels run.  A row that is padding has that LSE too, and reaches nothing.
    import paper_2109_04312_b200 as m
    rows, cols = (np.concatenate([x, np.full((1, 40), -1, np.int32)], 1) for x in _structure(20, 300, 30, 4, 13))
    r, c = torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda()
    plan = m.mate_plan_sat(r, c, 20, 2) if kind == "sat" else m.mate_plan(r, c, 20, [0, 1])
    gen = torch.Generator(device="cuda").manual_seed(15)
    Q, K, V, dO = ((torch.randn(1, 2, 360, 64, device="cuda", generator=gen) * 0.5).bfloat16() for _ in range(4))
    Q[..., 0], K[..., 0] = 0.0, -2.0 ** 100
    Q[:, :, at, 0] = 2.0 ** 100
    mask = {}
    for impl in (m.IMPL_TCGEN05, m.IMPL_SIMT):
        O, LSE = m.mate_attn_fwd(plan, Q, K, V, None, impl)
        assert torch.equal(torch.isneginf(LSE[0, 0]).nonzero().flatten().cpu(), torch.tensor(at + list(range(320, 360))))
        mask[impl] = [torch.isnan(x) for x in m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO, None, impl)]
    plan.status()
    ids = [rows[0, :320], cols[0, :320]]
    for name, tc, simt in zip(("dQ", "dK", "dV"), mask[m.IMPL_TCGEN05], mask[m.IMPL_SIMT]):
        assert torch.equal(tc, simt), name
        for h in range(2):
            met = np.zeros(360, bool)
            for k in at:
                same = (ids[0] == ids[0][k]) | (ids[1] == ids[1][k]) if kind == "sat" else ids[h] == ids[h][k]
                met[:320] |= same | (np.arange(320) < 20) | (k < 20)
            if name == "dQ":
                met = np.isin(np.arange(360), at)
            assert np.array_equal(tc[0, h].any(-1).cpu().numpy(), met), (name, h)


def _poisoned(t, where):
    """A copy of t whose rows `where` (a mask over its rows) hold NaN, Inf and -Inf in turn."""
    x = t.clone().view(-1, t.shape[-1])
    i = torch.nonzero(where.reshape(-1)).flatten()
    x[i] = torch.tensor([float("nan"), float("inf"), -float("inf")], dtype=t.dtype, device=t.device)[i % 3][:, None]
    return x.view(t.shape)


def _fwd_bwd(m, plan, impl, Q, K, V, dO):
    O, LSE = m.mate_attn_fwd(plan, Q, K, V, None, impl)
    return (O, LSE) + m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO, None, impl)


# The order's rows lie in place in the row view (bulk copies) and not in the column view (gathers); the valid
# positions end inside a group of 16 (the unit of the matrix instructions), with a whole box of padding behind.
@pytest.mark.parametrize("kind", ["exact", "bucketed", "sat"])
@pytest.mark.parametrize("P,n_table,row_len,n_cols", [(64, 136, 150, 2), (20, 301, 9, 4), (100, 157, 40, 3), (128, 259, 259, 1),
                                                      (31, 0, 1, 1), (130, 1000, 17, 3)])
def test_values_at_padding_are_ignored(kind, P, n_table, row_len, n_cols):
    import paper_2109_04312_b200 as m
    rows, cols = _structure(P, n_table, row_len, n_cols, P + n_table)
    nv = rows.shape[1]
    assert nv % 16 != 0
    rows, cols = (np.concatenate([np.concatenate([x, np.full((1, 160), -1, np.int32)], 1)] * 2) for x in (rows, cols))
    r, c = torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda()
    if kind == "sat":
        plan = m.mate_plan_sat(r, c, P, 3)
    else:
        plan = m.mate_plan(r, c, P, [0, 1, 0], radius=24 if kind == "bucketed" else 0)
    gen = torch.Generator(device="cuda").manual_seed(P)
    clean = [(torch.randn(2, 3, nv + 160, 64, device="cuda", generator=gen) * 0.5).bfloat16() for _ in range(4)]
    pad = (r < 0)[:, None, :].expand(2, 3, nv + 160)
    dirty = [_poisoned(x, pad) for x in clean]
    for impl in (m.IMPL_TCGEN05, m.IMPL_SIMT):
        want, got = _fwd_bwd(m, plan, impl, *clean), _fwd_bwd(m, plan, impl, *dirty)
        for name, w, g in zip(("O", "LSE", "dQ", "dK", "dV"), want, got):
            assert torch.equal(w, g), (name, impl)
            assert torch.isfinite(g[~pad]).all(), (name, impl)
    if kind != "sat":  # in view order every whole box inside the tensors may come by bulk copy
        perm = torch.from_numpy(np.stack([plan.get(v)[0] for v in (0, 1, 0)], 1).astype(np.int64)).cuda()
        a, b = ([x.gather(2, perm[..., None].expand(x.shape)) for x in t[:3]] for t in (clean, dirty))
        flags = m.IMPL_TCGEN05 | m.FLAG_VIEW_ORDER
        for w, g in zip(m.mate_attn_fwd(plan, *a, None, flags), m.mate_attn_fwd(plan, *b, None, flags)):
            assert torch.equal(w, g)
    plan.status()


def test_a_packed_example_does_not_reach_its_neighbours():
    import paper_2109_04312_b200 as m
    rng = np.random.default_rng(11)
    prefix, lengths = [64, 20, 40, 7], [200, 421, 61, 333]
    rows, cols = zip(*((np.concatenate([np.zeros(P, np.int32), 1 + np.arange(L - P, dtype=np.int32) // 90]),
                        np.concatenate([np.zeros(P, np.int32), rng.integers(1, 4, L - P).astype(np.int32)]))
                       for P, L in zip(prefix, lengths)))
    cu = np.concatenate([[0], np.cumsum(lengths)])
    r, c = (torch.from_numpy(np.concatenate(x)).cuda() for x in (rows, cols))
    plan = m.mate_plan_packed(r, c, cu, prefix, [0, 1, 0])
    gen = torch.Generator(device="cuda").manual_seed(3)
    clean = [(torch.randn(3, int(cu[-1]), 64, device="cuda", generator=gen) * 0.5).bfloat16() for _ in range(4)]
    for bad in range(4):
        where = torch.zeros(3, int(cu[-1]), dtype=torch.bool, device="cuda")
        where[:, cu[bad]:cu[bad + 1]] = True
        dirty = [_poisoned(x, where) for x in clean]
        for impl in (m.IMPL_TCGEN05, m.IMPL_SIMT):
            for name, w, g in zip(("O", "LSE", "dQ", "dK", "dV"), _fwd_bwd(m, plan, impl, *clean), _fwd_bwd(m, plan, impl, *dirty)):
                assert torch.isfinite(w).all() and torch.equal(w[~where], g[~where]), (name, impl, bad)
    plan.status()


@pytest.mark.parametrize("d,dtype", [(8, "f32"), (16, "f32"), (24, "bf16"), (40, "f32"), (64, "f32"), (72, "bf16"), (128, "f32")])
@pytest.mark.parametrize("P,n_table", [(0, 33), (31, 66), (64, 129), (65, 31)])
def test_tiled_fp32_kernels(P, n_table, d, dtype):
    rows, cols = _structure(P, n_table, 11, 3, d)
    _check(rows, cols, P, [0, 1], d, dtype, d, pad=2)


@pytest.mark.parametrize("row_len,n_cols", [(1, 1), (1023, 5), (1025, 129), (2100, 300)])
def test_cell_mean_buffers(row_len, n_cols):
    import paper_2109_04312_b200 as m
    rows, cols = _structure(7, 2 * row_len + 3, row_len, n_cols, row_len)
    x = np.random.default_rng(3).standard_normal(rows.shape).astype(np.float32)
    r, c = torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda()
    plan = m.mate_plan(r, c, 7, [0, 1])
    mean, count = m.mate_cell_mean(plan, torch.from_numpy(x).cuda(), c)
    n = np.zeros(tuple(mean.shape[1:]), np.int64)
    s = np.zeros(n.shape)
    np.add.at(n, (rows[0, 7:], cols[0, 7:]), 1)
    np.add.at(s, (rows[0, 7:], cols[0, 7:]), x[0, 7:])
    assert np.array_equal(count[0].cpu().numpy(), n)
    hp.assert_close(mean[0].cpu().numpy(), s / np.maximum(n, 1), 1e-5, 1e-5, "mean")


def test_plan_memory_is_reused_safely_across_streams_and_in_graphs():
    import paper_2109_04312_b200 as m
    rows, cols = _structure(40, 700, 21, 4, 2)
    r, c = torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda()
    Q, K, V = ((torch.randn(1, 2, 740, 64, device="cuda") * 0.5).bfloat16() for _ in range(3))
    torch.cuda.synchronize()
    want = m.mate_attn_fwd(m.mate_plan(r, c, 40, [0, 1]), Q, K, V)
    streams = [torch.cuda.Stream() for _ in range(3)]
    got = []
    for i in range(12):                       # plans made on one stream, used on the next, dropped while in flight
        with torch.cuda.stream(streams[i % 3]):
            plan = m.mate_plan(r, c, 40, [0, 1])
        with torch.cuda.stream(streams[(i + 1 + i // 6) % 3]):
            got.append(m.mate_attn_fwd(plan, Q, K, V))
        del plan
    torch.cuda.synchronize()
    plan = m.mate_plan(r, c, 40, [0, 1])      # captured before anything else has used it
    ws = torch.empty(max(m.mate_attn_workspace_bytes(plan, 64, 0)[0], 256), dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got.append(m.mate_attn_fwd(plan, Q, K, V, workspace=ws))
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for O, LSE in got:
        assert torch.equal(O, want[0]) and torch.equal(LSE, want[1])
    plan.status()


def test_the_kernel_before_does_not_count_against_the_bounded_waits():
    # A kernel that lets its successor start at once and then keeps one SM busy for about 75 ms: the attention
    # kernels are resident all that time, several times as long as one of their waits may take.
    import paper_2109_04312_b200 as m
    hold = torch.cuda._compile_kernel("""extern "C" __global__ void hold(int kclocks) {
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        const long long t0 = clock64();
        while (clock64() - t0 < 1000ll * kclocks) {}
    }""", "hold")
    rows, cols = _structure(40, 700, 21, 4, 2)
    plan = m.mate_plan(torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda(), 40, [0, 1])
    Q, K, V, dO = ((torch.randn(1, 2, 740, 64, device="cuda") * 0.5).bfloat16() for _ in range(4))
    fwd = lambda: m.mate_attn_fwd(plan, Q, K, V)  # noqa: E731
    O, LSE = fwd()
    bwd = lambda: m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO)  # noqa: E731
    for call in (fwd, bwd):
        want = call()
        torch.cuda.synchronize()
        begin, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        begin.record()
        hold(grid=(1, 1, 1), block=(1, 1, 1), args=[150000])
        got = call()
        end.record()
        torch.cuda.synchronize()
        plan.status()
        assert begin.elapsed_time(end) > 60
        for w, g in zip(want, got):
            assert torch.equal(w, g)
