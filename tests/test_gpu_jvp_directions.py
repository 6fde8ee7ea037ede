"""The JVP's direction counts around its passes: launches of 16 directions in two passes of eight, so a
partial first or second pass, a full one, and a second launch; blocks of 32 modes with a partial last
one, propagating and grazing modes.  Each direction by itself, against the oracle: dxi by its relative
L2 (1e-10 FS_FP64, 1e-5 FS_MIXED), Phi-dot, a sum of signed terms, by the size of those terms,
2 ||g|| ||F dW|| + 2 |lnalpha-dot| ||g||^2 (the same figures: a term is rounded to its own size)."""
import numpy as np
import pytest

from _cases import geometry
from oracle import adjoint, forward
from synth import random_gaussians

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision, tol", [("fp64", 1e-10), ("mixed", 1e-5)])
@pytest.mark.parametrize("n, m, m1, nd", [(12, 9, 5, 7), (12, 9, 5, 8), (12, 9, 5, 9), (16, 17, 9, 15), (12, 5, 3, 16), (8, 9, 2, 17),
                                          (12, 7, 3, 25)])
def test_each_direction(n, m, m1, nd, precision, tol):
    import torch
    from paper_1911_10487_gb300 import Geometry, Reconstructor
    from paper_1911_10487_gb300.diff import DiffPlan
    g = geometry(n, m, m1)
    rng = np.random.default_rng(1000 * n + nd)
    om = np.pi * np.array([3.0, 4.4])  # 3 pi: grazing modes
    W, _ = forward.make_data(random_gaussians(rng, n, m, g.z1, g.z2, 2, (0.15, 0.3), 0.05), list(om), g, method="born")
    W = W + 0.01 * np.sqrt(np.mean(np.abs(W) ** 2)) * (rng.standard_normal(W.shape) + 1j * rng.standard_normal(W.shape))
    la = np.array([np.log(3e-2 * np.max(np.linalg.svd(o ** 2 * adjoint.data_matrices(o, g), compute_uv=False)[..., 0] ** 2))
                   for o in om])
    t = adjoint.forward(W, om, g, la)
    dW = rng.standard_normal((nd,) + W.shape) + 1j * rng.standard_normal((nd,) + W.shape)
    dla = rng.standard_normal((nd, len(om)))
    rc = Reconstructor(0)
    plan = DiffPlan(rc, Geometry(g.n, g.m, g.z1, g.z2, tuple(g.zy), g.period), om, precision)
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)
    _, _, _, tape = plan.forward(dev(W, plan.cdt), dev(la, torch.float64))
    dxi, dphi = plan.jvp(tape, dev(dW, plan.cdt), dev(dla, torch.float64))
    dxi, dphi = dxi.cpu().numpy(), dphi.cpu().numpy()
    plan.close()
    rc.close()
    ex = ep = 0.0
    for d in range(nd):
        rx, rp = adjoint.jvp(t, dW[d], dla[d])
        ex = max(ex, np.linalg.norm(dxi[d] - rx) / np.linalg.norm(rx))
        fd = np.linalg.norm(np.fft.fft2(dW[d]).reshape(len(om), -1), axis=1)
        size = 2 * np.sqrt(t.phi) * fd + 2 * np.abs(dla[d]) * t.phi
        ep = max(ep, np.max(np.abs(dphi[d] - rp) / size))
    print(n, nd, precision, f"dxi {ex:.1e} dphi {ep:.1e}")
    assert ex <= tol and ep <= tol
