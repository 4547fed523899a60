"""Kernels of consecutive calls that overlap their starts: each kernel of a call has to read what the one
before it wrote, not what an earlier call left at the same place.

One context runs different problems in turn (other tile, batch, object, scan region and, through them, other
workspace layouts), each call's results compared with the same problem in a context of its own.  The
object gradient is summed in FP64 in any order, everything else in a fixed one, hence 1e-6.
"""
import numpy as np
import pytest

from tests import _cases as C

pytestmark = pytest.mark.gpu


def _problem(**kw):
    import torch
    case = C.small_case(**kw)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    p = case["problem"]
    nd = () if p["farfield"] else (len(p["nf"]),)
    meas = 0.5 + torch.rand((p["B"], *nd, p["N"], p["N"]), generator=torch.Generator("cuda").manual_seed(kw["N"]),
                            device="cuda") * 4
    return p, t(case["delta"]), t(case["beta"]), t(case["probe"].astype(np.complex64)), t(case["pos"]), meas


def _run(eng, q, oid):
    import torch
    p, d, b, probe, pos, meas = q
    out = [torch.zeros((), dtype=torch.float64, device="cuda"), torch.zeros_like(d), torch.zeros_like(b),
           torch.zeros_like(probe), torch.zeros_like(pos), torch.zeros_like(meas)]
    eng.loss_grad(p, oid, probe, pos, meas, *out)
    return out


def test_alternating_problems():
    import torch
    from paper_2012_12686_gb300.adorym import Engine
    problems = [_problem(N=32, L=2, M=1, B=5, loss="lsq", seed=1),
                _problem(N=128, L=3, M=1, B=9, loss="poisson", seed=2, Ly=401, Lx=390),   # side-stream form
                _problem(N=16, L=4, M=2, B=30, loss="poisson", seed=3),
                _problem(N=64, L=17, M=1, B=4, loss="lsq", tomo=True, theta=0.7, seed=4),
                _problem(N=256, L=2, M=1, B=3, loss="poisson", seed=5),
                _problem(N=256, L=1, M=1, B=2, loss="lsq", far=False, n_dist=2, seed=6),
                _problem(N=64, L=1, M=1, B=200, loss="lsq", seed=7)]
    ref = []
    for q in problems:
        eng = Engine(0)
        oid = eng.register_object(q[1], q[2])
        ref.append([x.cpu().numpy() for x in _run(eng, q, oid)])
        torch.cuda.synchronize()
        eng.close()
    eng = Engine(0)
    oids = [eng.register_object(q[1], q[2]) for q in problems]
    rng = np.random.default_rng(8)
    for _ in range(12):
        order = rng.permutation(len(problems))
        got = [(k, _run(eng, problems[k], oids[k])) for k in order]   # back to back, no synchronisation
        torch.cuda.synchronize()
        for k, out in got:
            for x, y in zip(out, ref[k]):
                assert C.rel(x.cpu().numpy(), y) <= 1e-6, k
    eng.close()
