"""Derivatives at fixed alpha at the edges of the per-mode kernels' split: 32 modes per block
(N = 8: two blocks, N = 12: a last block of 16 modes), X planes in blocks of 8 (M below, at
and past a block, and the limit 64), data planes dealt over 8 warps (M1 = 1 .. 32), grazing
and underflowing modes, and direction counts around the four of one pass.  Forward, VJP and
JVP against the oracle's SVD-based derivatives, relative L2: FS_FP64 1e-10, FS_MIXED 1e-5
(FP32 transforms and step 3), as for every result of this map."""
import functools

import numpy as np
import pytest

from _cases import geometry
from oracle import adjoint, forward
from synth import random_gaussians

pytestmark = pytest.mark.gpu

SHAPES = [(8, 1, 1, 1, 1), (12, 7, 2, 2, 3), (8, 8, 8, 1, 4), (12, 9, 9, 1, 5), (24, 17, 31, 2, 2), (16, 64, 32, 1, 17)]


@functools.lru_cache(maxsize=None)
def tape(shape):
    n, m, m1, n_om, nd = shape
    g = geometry(n, m, m1)
    rng = np.random.default_rng(sum(1000 ** i * v for i, v in enumerate(shape)))
    om = np.pi * np.array([3.0, 4.4])[:n_om]  # 3 pi: the modes (+-3, 0), (0, +-3) are grazing
    W, _ = forward.make_data(random_gaussians(rng, n, m, g.z1, g.z2, 2, (0.15, 0.3), 0.05), list(om), g, method="born")
    W = W + 0.01 * np.sqrt(np.mean(np.abs(W) ** 2)) * (rng.standard_normal(W.shape) + 1j * rng.standard_normal(W.shape))
    la = np.array([np.log(3e-2 * np.max(np.linalg.svd(o ** 2 * adjoint.data_matrices(o, g), compute_uv=False)[..., 0] ** 2))
                   for o in om])
    t = adjoint.forward(W, om, g, la)
    gxi, gphi = rng.standard_normal(t.xi.shape), rng.standard_normal(n_om) / t.phi
    dW = rng.standard_normal((nd,) + W.shape) + 1j * rng.standard_normal((nd,) + W.shape)
    dla = rng.standard_normal((nd, n_om))
    return g, om, W, la, t, gxi, gphi, dW, dla


def _rel(a, b):
    a = a.cpu().numpy()
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


@pytest.mark.parametrize("precision, tol", [("fp64", 1e-10), ("mixed", 1e-5)])
@pytest.mark.parametrize("shape", SHAPES)
def test_derivatives_at_the_edges_of_the_split(shape, precision, tol):
    import torch
    from paper_1911_10487_gb300 import Geometry, Reconstructor
    from paper_1911_10487_gb300.diff import DiffPlan
    g, om, W, la, t, gxi, gphi, dW, dla = tape(shape)
    rc = Reconstructor(0)
    plan = DiffPlan(rc, Geometry(g.n, g.m, g.z1, g.z2, tuple(g.zy), g.period), om, precision)
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)
    xi, _, phi, tp = plan.forward(dev(W, plan.cdt), dev(la, torch.float64))
    gW, gla = plan.vjp(tp, dev(gxi, plan.rdt), dev(gphi, torch.float64))
    gW0, _ = plan.vjp(tp, dev(gxi, plan.rdt), None)
    dxi, dphi = plan.jvp(tp, dev(dW, plan.cdt), dev(dla, torch.float64))
    rW, ra = adjoint.vjp(t, gxi, gphi)
    rW0, _ = adjoint.vjp(t, gxi, np.zeros(len(om)))
    err = {"xi": _rel(xi, t.xi), "phi": _rel(phi, t.phi), "gW": _rel(gW, rW), "gW0": _rel(gW0, rW0), "gla": _rel(gla, ra)}
    ref = [adjoint.jvp(t, dW[d], dla[d]) for d in range(dW.shape[0])]
    # over all directions together: one direction's Phi-dot is a sum that may cancel
    err["dxi"], err["dphi"] = _rel(dxi, np.stack([r[0] for r in ref])), _rel(dphi, np.stack([r[1] for r in ref]))
    plan.close()
    rc.close()
    print(shape, precision, {k: f"{v:.1e}" for k, v in err.items()})
    assert all(v <= tol for v in err.values()), err
