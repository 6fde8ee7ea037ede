"""Single-scattering data at the edges of the kernels' splits, against the oracle (relative L2;
FS_FP64 1e-12, the transforms' and exponentials' rounding; FS_MIXED 2e-6, a few FP32 roundings
through two transforms): X planes around the blocks of 8 and an odd count (pairs of real planes),
data planes uniform (at least 8) and not, frequencies around the four of one block, grazing
modes, and a given incident field, whose data with the plane wave given must equal the packed
path's.  One step of Algorithm 1 from the same field covers the interior kernel's chunks."""
import numpy as np
import pytest

from oracle import forward
from oracle.grid import Geometry as OGeom, layer_planes
from synth import random_gaussians

pytestmark = pytest.mark.gpu

SHAPES = [(8, 1, 1, 1, "uniform"), (12, 7, 8, 2, "uniform"), (16, 8, 9, 4, "ragged"), (24, 9, 17, 5, "uniform"),
          (32, 17, 33, 3, "ragged"), (12, 40, 40, 1, "uniform"), (8, 65, 5, 1, "uniform"), (8, 128, 128, 5, "uniform")]


@pytest.mark.parametrize("precision, tol", [("fp64", 1e-12), ("mixed", 2e-6)])
@pytest.mark.parametrize("shape", SHAPES)
def test_born_data(shape, precision, tol):
    import torch
    from paper_1911_10487_gb300 import Geometry, Reconstructor
    n, m, m1, n_om, planes = shape
    rng = np.random.default_rng(n * 1000 + m * 10 + m1)
    zy = np.asarray(layer_planes(1.2, 1.6, m1)) if planes == "uniform" else np.sort(rng.uniform(1.2, 1.6, m1))
    g = OGeom(n, m, 0.2, 1.0, tuple(zy))
    om = np.pi * np.array([3.0, 2.2, 3.4, 2.6, 1.7])[:n_om]  # 3 pi: grazing modes
    xi = random_gaussians(rng, n, m, g.z1, g.z2, 2, (0.15, 0.3), 0.05)
    ref, _ = forward.make_data(xi, list(om), g, method="born")
    rc = Reconstructor(0)
    geom = Geometry(n, m, g.z1, g.z2, tuple(zy), g.period)
    x = torch.from_numpy(xi).to("cuda", torch.float64 if precision == "fp64" else torch.float32)
    W = rc.forward_born(x, list(om), geom, precision=precision)
    u0 = np.stack([np.broadcast_to(forward.incident_plane_wave(o, g), (m, n, n)) for o in om])
    u0 = torch.from_numpy(np.ascontiguousarray(u0)).to("cuda", W.dtype)
    Wi = rc.forward_born(x, list(om), geom, precision=precision, incident=u0)
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)
    e, ei = rel(W.cpu().numpy(), ref), rel(Wi.cpu().numpy(), ref)
    print(shape, precision, f"{e:.1e} {ei:.1e}")
    assert e <= tol and ei <= tol
    if m <= 64:  # to convergence: the interior kernel at this plane count
        full, _ = forward.make_data(xi, list(om), g, method="fixed_point")
        Wf, _, _ = rc.forward(x, list(om), geom, precision=precision)
        ef = rel(Wf.cpu().numpy(), full)
        print(f"   full {ef:.1e}")
        assert ef <= (1e-11 if precision == "fp64" else 1e-5)  # stopping at 1e-13 / 1e-6 of ||U~0||, W ~ xi u0 below it
    rc.close()
