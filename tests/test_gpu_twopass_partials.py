"""Two-pass path: position-gradient partials of a batch whose partials outgrow the probe-transform
buffer that they share, and the slice-gap sum over many partials.

Each position's gradient is the same sum whatever the batch, scaled by the batch's pixel count, so a
batch of 1400 agrees with two of 700 to the FP32 rounding of the result (1e-6); the object gradient
is summed in FP64.
"""
import numpy as np
import pytest

from tests import _cases as C

pytestmark = pytest.mark.gpu


def test_large_batch_matches_halves():
    import torch
    from paper_2012_12686_gb300.adorym import Engine
    B = 1400
    case = C.small_case(N=256, L=2, M=1, B=B, loss="lsq", seed=3)
    p = dict(case["problem"], gaps=[0.4])
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    d, b, probe, pos = t(case["delta"]), t(case["beta"]), t(case["probe"].astype(np.complex64)), t(case["pos"])
    eng = Engine(0)
    oid = eng.register_object(d, b)
    Im = torch.zeros((B, 256, 256), device="cuda")
    eng.forward(p, oid, probe, pos, Im)
    Im = 0.9 * Im + 0.5

    def call(lo, hi):
        q = dict(p, B=hi - lo)
        out = dict(g_delta=torch.zeros_like(d), g_beta=torch.zeros_like(b), g_probe=torch.zeros_like(probe),
                   g_pos=torch.zeros_like(pos[lo:hi]), g_gaps=torch.zeros(1, device="cuda"))
        eng.loss_grad_ext(q, oid, probe, pos[lo:hi].contiguous(), Im[lo:hi].contiguous(), **out)
        torch.cuda.synchronize()
        return {k: v.cpu().numpy().astype(np.complex128 if v.is_complex() else np.float64) for k, v in out.items()}

    whole, parts = call(0, B), [call(0, B // 2), call(B // 2, B)]
    assert C.rel(whole["g_pos"], 0.5 * np.concatenate([q["g_pos"] for q in parts])) <= 1e-6
    for k in ("g_delta", "g_beta", "g_probe", "g_gaps"):
        assert C.rel(whole[k], 0.5 * (parts[0][k] + parts[1][k])) <= 1e-6, k
    eng.close()
