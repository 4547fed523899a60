"""Regularizer and l1-weight kernels at the edges of their tiles (32 x 8 columns and a few planes; 128-bit
groups where Lx % 4 == 0), against the FP64 oracle.

Tolerances: a gradient value is a sum of at most seven FP32 terms scaled once, so 8 x 2^-24 < 1e-6
of its size; the value is Kahan-compensated; a weight takes one addition and one division.
"""
import numpy as np
import pytest

from tests import _cases as C

pytestmark = pytest.mark.gpu


def _volume(shape, seed):
    g = np.random.default_rng(seed)
    return (g.uniform(-1e-5, 1e-5, shape).astype(np.float32), g.uniform(-1e-6, 1e-6, shape).astype(np.float32))


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 8, 128), (2, 9, 132), (3, 7, 31), (17, 8, 33), (33, 16, 64), (5, 1, 260)])
@pytest.mark.parametrize("gamma", [0.0, 0.7])
def test_tile_edges(shape, gamma):
    import torch
    from oracle import regularizers as R
    from paper_2012_12686_gb300.adorym import Engine
    d, b = _volume(shape, sum(shape))
    eng = Engine(0)
    td, tb = torch.from_numpy(d).cuda(), torch.from_numpy(b).cuda()
    oid = eng.register_object(td, tb)
    wd, wb = torch.empty_like(td), torch.empty_like(tb)
    eng.l1_weights(oid, 1e-7, wd, wb)
    rw = R.l1_weights(d, 1e-7), R.l1_weights(b, 1e-7)
    assert C.rel(wd.cpu().numpy(), rw[0]) < 3e-7 and C.rel(wb.cpu().numpy(), rw[1]) < 3e-7
    kw = dict(alpha_delta=0.3, alpha_beta=2.0, gamma_tv=gamma)
    ref = R.regularize(d, b, w_delta=rw[0], w_beta=rw[1], **kw)
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    gd, gb = torch.ones_like(td), torch.ones_like(tb)
    gd.zero_(), gb.zero_()
    eng.regularize(oid, w_delta=wd, w_beta=wb, loss_out=loss, g_delta=gd, g_beta=gb, **kw)
    assert abs(loss.item() - ref[0]) <= 1e-6 * abs(ref[0])
    assert C.rel(gd.cpu().numpy(), ref[1]) <= 1e-6 and C.rel(gb.cpu().numpy(), ref[2]) <= 1e-6
    eng.close()


@pytest.mark.parametrize("n", [64, 63])
def test_one_buffer_for_both_weights(n):
    """Both weight arrays the same memory: the weights of beta, as from one volume after the other."""
    import torch
    from paper_2012_12686_gb300.adorym import Engine
    d, b = _volume((2, 3, n), n)
    eng = Engine(0)
    td, tb = torch.from_numpy(d).cuda(), torch.from_numpy(b).cuda()
    oid = eng.register_object(td, tb)
    w, wd, wb = (torch.empty_like(td) for _ in range(3))
    eng.l1_weights(oid, 1e-7, w, w)
    eng.l1_weights(oid, 1e-7, wd, wb)
    assert torch.equal(w, wb) and not torch.equal(w, wd)
    eng.close()
