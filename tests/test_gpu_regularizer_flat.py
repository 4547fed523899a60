"""Regularizer on volumes of few rows or of one plane, whose tiles have fewer rows and walk along the longer
axis: against the FP64 oracle, and no slower than the same volume with the axes named otherwise.

Tolerances as at the tile edges (tests/test_gpu_regularizer_tiles.py): at most seven FP32 terms scaled once for a
gradient, a compensated sum for the value.
"""
import numpy as np
import pytest

from tests import _cases as C

pytestmark = pytest.mark.gpu


def _setup(shape):
    import torch
    from paper_2012_12686_gb300.adorym import Engine
    g = np.random.default_rng(sum(shape))
    d = g.uniform(-1e-5, 1e-5, shape).astype(np.float32)
    b = g.uniform(-1e-6, 1e-6, shape).astype(np.float32)
    eng = Engine(0)
    td, tb = torch.from_numpy(d).cuda(), torch.from_numpy(b).cuda()
    return eng, eng.register_object(td, tb), d, b, td, tb


@pytest.mark.parametrize("shape", [
    (37, 1, 33), (16, 1, 1), (300, 1, 65), (19, 2, 31), (35, 6, 33), (9, 4, 127), (70, 4, 5), (18, 3, 33), (33, 5, 63),
    (16, 7, 34), (1, 9, 33), (1, 100, 70), (1, 1, 97), (1, 300, 31), (1, 31, 1),
])
@pytest.mark.parametrize("gamma", [0.0, 0.7])
def test_few_rows_or_planes(shape, gamma):
    import torch
    from oracle import regularizers as R
    eng, oid, d, b, td, tb = _setup(shape)
    g = np.random.default_rng(3)
    w = [g.uniform(0.5, 2.0, shape).astype(np.float32) for _ in range(2)]
    kw = dict(alpha_delta=0.3, alpha_beta=2.0, gamma_tv=gamma)
    ref = R.regularize(d, b, w_delta=w[0], w_beta=w[1], **kw)
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    gd, gb = torch.zeros_like(td), torch.zeros_like(tb)
    tw = [torch.from_numpy(x).cuda() for x in w]
    eng.regularize(oid, w_delta=tw[0], w_beta=tw[1], loss_out=loss, g_delta=gd, g_beta=gb, **kw)
    assert abs(loss.item() - ref[0]) <= 1e-6 * abs(ref[0])
    assert C.rel(gd.cpu().numpy(), ref[1]) <= 1e-6 and C.rel(gb.cpu().numpy(), ref[2]) <= 1e-6
    eng.close()


def _us(shape):
    import torch
    eng, oid, d, b, td, tb = _setup(shape)
    out = [torch.zeros((), dtype=torch.float64, device="cuda"), torch.zeros_like(td), torch.zeros_like(tb)]

    def elapsed():
        t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t0.record()
        for _ in range(30):
            eng.regularize(oid, alpha_delta=0.3, alpha_beta=2.0, gamma_tv=0.7, loss_out=out[0], g_delta=out[1],
                           g_beta=out[2])
        t1.record()
        torch.cuda.synchronize()
        return t0.elapsed_time(t1) / 30 * 1e3

    elapsed()
    best = min(elapsed() for _ in range(7))
    eng.close()
    return best


def test_one_row_takes_the_time_of_one_plane():
    """The same numbers in the same order in memory: 92 against 34 us with one row per tile, 28 and 28 now."""
    assert _us((4096, 1, 511)) <= 1.5 * _us((1, 4096, 511))
