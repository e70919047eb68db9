"""The native binding of the per-layer calls: what it lets other threads do, and what it refuses."""
import ctypes
import threading
import time

import pytest
import torch


@pytest.mark.gpu
def test_other_threads_run_while_a_call_waits():
    # libc's usleep stands in for the three entry points that may wait: their first argument, the plan's address, is
    # what it takes for its microseconds, and it returns 0 (MATE_OK)
    import paper_2109_04312_b200 as m
    lib = m.api._load()
    from paper_2109_04312_b200 import _native
    address = lambda f: ctypes.cast(f, ctypes.c_void_p).value  # noqa: E731
    nothing = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_uint, ctypes.c_void_p,
                               ctypes.c_void_p)(lambda *a: 0)
    usleep = address(ctypes.CDLL(None).usleep)
    info = _native.plan_info(200000, 1, 16, 2, -1, 1, 1, torch.cuda.current_device())
    t, lse = torch.zeros(1, 2, 16, 64, device="cuda"), torch.zeros(1, 2, 16, device="cuda")
    logits, ids = torch.zeros(1, 16, device="cuda"), torch.zeros(1, 16, dtype=torch.int32, device="cuda")
    ticks, stop = [0], threading.Event()

    def tick():
        while not stop.is_set():
            time.sleep(0.001)
            ticks[0] += 1

    thread = threading.Thread(target=tick)
    _native.bind(address(nothing), usleep, usleep, usleep, m.MateError)
    try:
        thread.start()
        for call in (lambda: _native.attn_fwd(info, t, t, t, None, 0, None, None, None),
                     lambda: _native.attn_fwd(info, t, t, t, None, 0, t, lse, None),
                     lambda: _native.attn_bwd(info, t, t, t, t, lse, t, None, 0, None),
                     lambda: _native.cell_mean(info, logits, ids, True, None, None),
                     lambda: _native.cell_mean(info, logits, ids, False, logits, None)):
            before, begin = ticks[0], time.monotonic()
            call()
            assert time.monotonic() - begin > 0.19
            assert ticks[0] - before > 20
    finally:
        stop.set()
        thread.join()
        _native.bind(*(address(f) for f in (lib.mate_attn_workspace_bytes, lib.mate_attn_fwd, lib.mate_attn_bwd,
                                            lib.mate_cell_mean)), m.MateError)


@pytest.mark.gpu
def test_a_plans_workspace_outlives_it_on_every_stream():
    # The workspace is allocated by the first call and used by one on another stream, which is still to run when
    # the plan goes: the memory must not be handed out on the first stream until then.
    import paper_2109_04312_b200 as m
    ids = torch.ones(1, 4096, dtype=torch.int32, device="cuda")
    Q, K, V, dO = ((torch.randn(1, 2, 4096, 64, device="cuda") * 0.5).bfloat16() for _ in range(4))
    plan = m.mate_plan(ids, ids, 0, [0, 1])
    need = m.mate_attn_workspace_bytes(plan, 64, 0)
    assert min(need) > 0                              # (few heads: units are cut, and their parts go through it)
    O, LSE = m.mate_attn_fwd(plan, Q, K, V)
    want = (O, LSE) + m.mate_attn_bwd(plan, Q, K, V, O, LSE, dO)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(50_000_000)
        o, l = m.mate_attn_fwd(plan, Q, K, V)
        got = (o, l) + m.mate_attn_bwd(plan, Q, K, V, o, l, dO)
    plan.destroy()
    junk = [torch.full((n,), 255, dtype=torch.uint8, device="cuda") for n in need * 4]   # NaN, whatever is read there
    torch.cuda.synchronize()
    for w, g in zip(want, got):
        assert torch.equal(w, g)
    del junk


def test_types_and_sizes_are_checked_before_anything_is_launched():
    # host tensors: what is refused here is refused for its type or size; what passes stops at the next check,
    # that the tensors are on a GPU
    import paper_2109_04312_b200 as m
    m.api._load()
    from paper_2109_04312_b200 import _native
    info = _native.plan_info(0, 1, 16, 2, -1, 3, 5, 0)
    q, h = torch.zeros(1, 2, 16, 64), torch.zeros(1, 2, 16, 64, dtype=torch.bfloat16)
    stat, ids = torch.zeros(1, 2, 16), torch.zeros(1, 16, dtype=torch.int32)

    def fwd(k=q, v=q, out=None, lse=None):
        _native.attn_fwd(info, q, k, v, None, 0, out, lse, None)

    def bwd(lse):
        _native.attn_bwd(info, q, q, q, q, lse, q, None, 0, None)

    def cells(mean, count):
        _native.cell_mean(info, torch.zeros(1, 16), ids, True, mean, count)

    def noalloc(lse):
        plan = m.Plan.__new__(m.Plan)
        plan._h, plan.B, plan.H, plan.N, plan.T = None, 1, 2, 16, None
        m.mate_attn_bwd_noalloc(plan, q, q, q, q, lse, q, q, q, q)

    for what, call in (("K and V", lambda: fwd(k=h)), ("K and V", lambda: fwd(v=h)), ("O", lambda: fwd(out=h)),
                       ("O", lambda: fwd(out=q[..., :32])), ("LSE", lambda: fwd(lse=stat.bfloat16())),
                       ("LSE", lambda: fwd(lse=stat[..., 1:])), ("LSE", lambda: bwd(stat.bfloat16())), ("LSE", lambda: bwd(stat[..., 1:])),
                       ("mean", lambda: cells(torch.zeros(1, 3, 5).half(), torch.zeros(1, 3, 5, dtype=torch.int32))),
                       ("mean", lambda: cells(torch.zeros(1, 3, 4), torch.zeros(1, 3, 5, dtype=torch.int32))),
                       ("count", lambda: cells(torch.zeros(1, 3, 5), torch.zeros(1, 3, 5, dtype=torch.int16))),
                       ("LSE", lambda: noalloc(stat.bfloat16())), ("LSE", lambda: noalloc(stat[..., 1:]))):
        with pytest.raises(ValueError, match="^%s must (match|be a )(?!contiguous)" % what):
            call()
    for call in (lambda: fwd(out=q, lse=stat), lambda: fwd(out=q.flatten(), lse=torch.zeros(40)), lambda: bwd(stat),
                 lambda: cells(torch.zeros(1, 3, 5), torch.zeros(1, 3, 5, dtype=torch.int32))):
        with pytest.raises(ValueError, match="contiguous CUDA tensor"):
            call()
