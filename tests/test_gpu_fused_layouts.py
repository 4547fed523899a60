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


@pytest.mark.parametrize("N", [64, 128])
def test_equal_gaps_match_uniform(N):
    """Equal gaps take the variable-spacing kernel: same stages, same FP64-built tables, so the same
    values up to the order of the FP64 object-gradient sums."""
    import torch
    from paper_2012_12686_gb300.adorym import Engine
    L = 5
    case = C.small_case(N=N, L=L, M=1, B=3, loss="poisson", seed=N)
    p = case["problem"]
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    d, b, probe, pos = t(case["delta"]), t(case["beta"]), t(case["probe"].astype(np.complex64)), t(case["pos"])
    eng = Engine(0)
    oid = eng.register_object(d, b)
    Im = torch.zeros((3, N, N), device="cuda")
    eng.forward(p, oid, probe, pos, Im)
    Im = 0.9 * Im + 0.5

    def call(problem):
        out = [torch.zeros((), dtype=torch.float64, device="cuda"), torch.zeros_like(d), torch.zeros_like(b),
               torch.zeros_like(probe), torch.zeros_like(pos)]
        eng.loss_grad(problem, oid, probe, pos, Im, *out)
        torch.cuda.synchronize()
        return [x.cpu().numpy() for x in out]

    for x, y in zip(call(p), call(dict(p, gaps=[p["lambda_dz_over_px2"]] * (L - 1)))):
        assert C.rel(x, y) <= 1e-6
    eng.close()
