"""The fused kernels' shared-memory layouts and warp-level hand-overs at N = 64 and N = 128: forms that
reach every pass (single slice, several modes, near field with several distances, variable spacing,
batches of one, of the pipelined form and of more CTAs than SMs), against the FP64 oracle at the
parity bars."""
import numpy as np
import pytest

from tests import _cases as C
from tests.test_gpu_parity import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L,M,B,loss,cp", [
    (128, 1, 1, 1, "lsq", 0),
    (128, 3, 2, 2, "poisson", 2),
    (128, 4, 1, 80, "lsq", 2),      # above half the SM count: recompute helpers
    (64, 2, 3, 2, "poisson", 0),
    (64, 1, 2, 160, "lsq", 0),      # more positions than SMs
])
def test_far(N, L, M, B, loss, cp):
    _compare(C.small_case(N=N, L=L, M=M, B=B, loss=loss, cp=cp, seed=N + L + B), workers=min(B, 8))


@pytest.mark.parametrize("N,L,M,B,nd", [(128, 2, 1, 1, 3), (128, 3, 2, 1, 1), (64, 2, 2, 2, 2)])
def test_near(N, L, M, B, nd):
    _compare(C.small_case(N=N, L=L, M=M, B=B, loss="lsq", far=False, n_dist=nd, seed=2 + N + L))


@pytest.mark.parametrize("N,L,M,cp", [(128, 4, 1, 0), (128, 3, 2, 1), (64, 5, 2, 0)])
def test_variable_spacing(N, L, M, cp):
    """The variable-spacing instantiation: intensities, object and slice-gap gradients."""
    import torch
    import oracle
    from paper_2012_12686_gb300.adorym import Engine
    case = C.small_case(N=N, L=L, M=M, B=2, loss="lsq", cp=cp, seed=31 + N + L)
    p = dict(case["problem"], gaps=[0.2 + 0.3 * j for j in range(L - 1)])
    Im = C.measured(dict(case, problem=p)).astype(np.float32)
    ref = oracle.loss_grad(p, case["delta"], case["beta"], case["probe"], case["pos"], Im, want_gaps=True)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    d, b = t(case["delta"]), t(case["beta"])
    eng = Engine(0)
    oid = eng.register_object(d, b)
    gd, gb = torch.zeros_like(d), torch.zeros_like(b)
    gg, I = torch.zeros(L - 1, device="cuda"), torch.zeros(Im.shape, device="cuda")
    eng.loss_grad_ext(p, oid, t(case["probe"].astype(np.complex64)), t(case["pos"]), t(Im), g_delta=gd, g_beta=gb,
                      g_gaps=gg, I_out=I)
    torch.cuda.synchronize()
    assert C.rel(I.cpu().numpy(), oracle.forward(p, case["delta"], case["beta"], case["probe"], case["pos"])) <= C.TOL_I
    for x, y in ((gd, ref[1]), (gb, ref[2]), (gg, ref[-1])):
        assert C.rel(x.cpu().numpy(), y) <= C.TOL_G
    eng.close()
