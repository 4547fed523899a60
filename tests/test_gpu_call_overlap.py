"""Calls enqueued one after the other overlap: one of them costs less than a call that is waited for.

A kernel that starts its CTAs while the one before drains can be placed badly (several CTAs on the SMs that
are free first, the others idle), which shows only when the call's kernels are all enqueued: 20 positions of
32 x 32 with 16 slices took 142 us each in a row and 106 us waited for, against 92 and 106 well placed.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_in_a_row_costs_no_more():
    import torch
    from paper_2012_12686_gb300.adorym import Engine
    N, L, B, S = 32, 16, 20, 90
    p = dict(N=N, L=L, M=1, B=B, Lz=L, Ly=S, Lx=S, kdz=1.0, lambda_dz_over_px2=0.3, farfield=1, nf=[], loss="lsq",
             eps=1e-6)
    g = torch.Generator("cuda").manual_seed(1)
    d = torch.rand((L, S, S), device="cuda", generator=g) * 1e-3
    b = 0.1 * d
    probe = torch.view_as_complex(torch.randn((1, N, N, 2), device="cuda", generator=g))
    pos = torch.rand((B, 2), device="cuda", generator=g) * (S - N)
    meas = torch.rand((B, N, N), device="cuda", generator=g) + 0.5
    eng = Engine(0)
    oid = eng.register_object(d, b)
    out = [torch.zeros((), dtype=torch.float64, device="cuda"), torch.zeros_like(d), torch.zeros_like(b),
           torch.zeros_like(probe), torch.zeros_like(pos)]

    def elapsed(calls):
        t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        t0.record()
        for _ in range(calls):
            eng.loss_grad(p, oid, probe, pos, meas, *out)
        t1.record()
        torch.cuda.synchronize()
        return t0.elapsed_time(t1) / calls

    elapsed(30)
    in_a_row = float(np.median([elapsed(40) for _ in range(9)]))
    waited_for = float(np.median([elapsed(1) for _ in range(41)]))
    eng.close()
    assert in_a_row < waited_for
