"""Products of one and of two shared-memory stages launched by several host threads at
once: the launches take different amounts of shared memory of the same kernels."""
import ctypes
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu

CALLS = 20000


@pytest.mark.parametrize("rows", [8, 16])
def test_threads_launch_products_of_one_and_two_stages(rows):
    """Two threads with each number of stages: the forward product of 8 rows (16 and 17
    input blocks) and the weight gradient of 16 (8 and 9); every call succeeds and every
    word is the same as alone."""
    from paper_2403_11166_gb300 import he
    dual = rows == 16
    ctx = he.Context(12, 2, 54, 41)
    jobs = []
    for k in ((8, 9) if dual else (16, 17)) * 2:   # the most input blocks of one stage, the least of two
        layer = he.Layer(he.FC, k, rows, 16) if dual else he.Layer(he.FC, rows, k, 16)
        plan = he.Plan(ctx, layer, he.ROLE_WGRAD if dual else he.ROLE_FWD, (1, 1, 1, 1, 1, 1, 1))
        s = plan.sizes
        ct_in, ct_out = plan.new_ct(s.ct_in).zero_(), plan.new_ct(s.ct_out)
        pt, ct_k = plan.new_pt(s.pt).zero_(), plan.new_ct(s.pt).zero_()
        x0 = torch.zeros(rows * k, dtype=torch.int64, device="cuda")
        g0 = torch.zeros(16 * k, dtype=torch.int64, device="cuda")
        y0 = torch.empty(s.out_elems, dtype=torch.int64, device="cuda")
        ws = plan.new_ws(max(s.ws_forward, s.ws_backward))
        stream = torch.cuda.Stream()
        p, nb, st = he._ptr, ctypes.c_size_t(ws.numel() * 8), he._stream(stream)
        seed = ctypes.c_uint64(9)
        # arguments converted once: a thread then spends its time inside the library
        if dual:
            fn = he.lib.he_linear_backward
            args = (ctx.h, None, plan.h, None, None, p(ct_in), p(ct_k), p(g0), p(x0), seed, seed, None, None,
                    p(ct_out), p(y0), p(ws), nb, st)
        else:
            he.he_linear_forward(ctx, plan, ct_in, pt, x0, None, 9, ct_out, y0, ws)
            fn = he.lib.he_linear_forward_apply
            args = (ctx.h, plan.h, p(ct_in), p(pt), p(ct_out), p(ws), nb, st)
        torch.cuda.synchronize()
        assert fn(*args) == 0
        torch.cuda.synchronize()
        jobs.append((fn, args, ct_out, ct_out.clone(), (plan, ct_in, pt, ct_k, x0, g0, y0, ws, stream)))
    codes = []
    start = threading.Barrier(len(jobs))

    def run(fn, args):
        start.wait()
        for _ in range(CALLS // (8 if dual else 1)):
            rc = fn(*args)
            if rc:
                codes.append(rc)

    threads = [threading.Thread(target=run, args=j[:2]) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not codes
    for _, _, out, want, _ in jobs:
        assert torch.equal(out, want)


def test_threads_launch_staged_products_of_different_shapes():
    """The same for the shared-memory staged kernel (columns 0), whose stage depends on the
    number of output columns: 1 (the largest) and 8 (the smallest)."""
    from paper_2403_11166_gb300 import he
    ctx = he.Context(12, 2, 60, 41)
    ctx.tune(he.TUNE_MAC_COLUMNS, 0)
    jobs = []
    for nc in (1, 8) * 2:
        plan = he.Plan(ctx, he.Layer(he.FC, 8, 2, nc), he.ROLE_FWD, (1, 1, 1, 1, 1, 1, 1))
        s = plan.sizes
        ct_in, ct_out, pt = plan.new_ct(s.ct_in).zero_(), plan.new_ct(s.ct_out), plan.new_pt(s.pt).zero_()
        x0 = torch.zeros(16, dtype=torch.int64, device="cuda")
        y0 = torch.empty(s.out_elems, dtype=torch.int64, device="cuda")
        ws, stream = plan.new_ws(s.ws_forward), torch.cuda.Stream()
        he.he_linear_forward(ctx, plan, ct_in, pt, x0, None, 9, ct_out, y0, ws)
        torch.cuda.synchronize()
        args = (ctx.h, plan.h, he._ptr(ct_in), he._ptr(pt), he._ptr(ct_out), he._ptr(ws),
                ctypes.c_size_t(ws.numel() * 8), he._stream(stream))
        jobs.append((args, ct_out, ct_out.clone(), (plan, ct_in, pt, ws, stream)))
    codes = []
    start = threading.Barrier(len(jobs))

    def run(args):
        start.wait()
        for _ in range(CALLS):
            rc = he.lib.he_linear_forward_apply(*args)
            if rc:
                codes.append(rc)

    threads = [threading.Thread(target=run, args=(j[0],)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not codes
    for _, out, want, _ in jobs:
        assert torch.equal(out, want)
