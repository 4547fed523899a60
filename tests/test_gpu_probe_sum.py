"""Probe-gradient sum over a batch of at most eight: as accurate as an FP64 sum rounded once, element by
element (a norm would not see the elements whose terms cancel).

Near field, so that the sum itself is the result: problem b of a batch of B gives 1 / B of the gradient
that it gives alone, an exact scaling for a power of two.  Bound: half an ulp of the result for the one
rounding, and 2^-53 of the sum of magnitudes per FP64 addition, here and in the sum compared with.
"""
import numpy as np
import pytest

from tests import _cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,M", [(2, 1), (4, 2), (8, 1), (8, 2)])
def test_sum_rounds_once(B, M):
    import torch
    from paper_2012_12686_gb300.adorym import Engine
    case = C.small_case(N=256, L=1, M=M, B=B, loss="lsq", far=False, n_dist=2, seed=40 + B)
    p = case["problem"]
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    d, b, probe, pos = t(case["delta"]), t(case["beta"]), t(case["probe"]), t(case["pos"])
    meas = torch.rand((B, 2, 256, 256), generator=torch.Generator("cuda").manual_seed(B), device="cuda") * 2
    eng = Engine(0)

    def g_probe(lo, hi):
        q = dict(p, B=hi - lo, Lz=hi - lo)
        oid = eng.register_object(d[lo:hi].contiguous(), b[lo:hi].contiguous())
        g = torch.zeros_like(probe)
        eng.loss_grad(q, oid, probe, pos[lo:hi].contiguous(), meas[lo:hi].contiguous(), g_probe=g)
        torch.cuda.synchronize()
        eng.unregister_object(oid)
        return torch.view_as_real(g).cpu().numpy()

    terms = np.stack([g_probe(k, k + 1) for k in range(B)]).astype(np.float64) / B
    ref, got = terms.sum(0), g_probe(0, B)
    ulp = np.spacing(np.maximum(np.abs(got), np.abs(ref.astype(np.float32)))).astype(np.float64)
    bound = 0.5 * ulp + 2 * B * 2.0 ** -53 * np.abs(terms).sum(0)
    assert (np.abs(got - ref) <= bound).all(), float((np.abs(got - ref) > bound).mean())
    eng.close()
