"""Regularizer and l1-weight kernels on volumes where a CTA has more to do than one short tile: many planes
per tile, more tiles than CTAs, several rounds of loads per thread.

Planes per tile are halved from 16 until there are 1216 tiles, and 1216 is also the number of CTAs; the
weight kernels take 608 CTAs of 256 threads with four loads each, of four values where the volume allows
it.  Tolerances as in the tests at the tile edges: seven FP32 terms scaled once for a gradient (1e-6), a
compensated sum for the value, one addition and one division for a weight.  The largest magnitudes stand at the
end, so that a tail left out changes every weight.
"""
import numpy as np
import pytest

from tests import _cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [
    (33, 509, 511),   # 16 planes a tile, the last of one; 3072 tiles; 14 rounds of single weight loads
    (29, 157, 509),   # 8 planes, the last tile of 5; 1280 tiles
    (14, 157, 509),   # 4 planes, the last tile of 2; 1280 tiles
    (21, 512, 508),   # whole rows of 128-bit groups: the flat form; three rounds of 128-bit weight loads
    (21, 511, 512),
])
def test_long_walk(shape):
    import torch
    from oracle import regularizers as R
    from paper_2012_12686_gb300.adorym import Engine
    g = np.random.default_rng(sum(shape))
    d = g.uniform(-1e-5, 1e-5, shape).astype(np.float32)
    b = g.uniform(-1e-6, 1e-6, shape).astype(np.float32)
    d.flat[-1], b.flat[-2] = -2e-5, 3e-6
    eng = Engine(0)
    td, tb = torch.from_numpy(d).cuda(), torch.from_numpy(b).cuda()
    oid = eng.register_object(td, tb)
    wd, wb = torch.empty_like(td), torch.empty_like(tb)
    eng.l1_weights(oid, 1e-7, wd, wb)
    rw = R.l1_weights(d, 1e-7), R.l1_weights(b, 1e-7)
    for w, r in zip((wd, wb), rw):
        assert (np.abs(w.cpu().numpy() - r) <= 3e-7 * r).all()
    kw = dict(alpha_delta=0.3, alpha_beta=2.0, gamma_tv=0.7)
    ref = R.regularize(d, b, w_delta=rw[0], w_beta=rw[1], **kw)
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    gd, gb = torch.zeros_like(td), torch.zeros_like(tb)
    eng.regularize(oid, w_delta=wd, w_beta=wb, loss_out=loss, g_delta=gd, g_beta=gb, **kw)
    assert abs(loss.item() - ref[0]) <= 1e-6 * abs(ref[0])
    assert C.rel(gd.cpu().numpy(), ref[1]) <= 1e-6 and C.rel(gb.cpu().numpy(), ref[2]) <= 1e-6
    eng.close()
