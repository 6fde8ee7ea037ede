"""Algorithm 1 over every transform length, against the oracle's own iteration (relative L2;
FS_FP64 1e-11: it stops at 1e-13 of ||U~0||, and W ~ xi u0 lies below u0; FS_MIXED 1e-5: stops at
1e-6).  The row kernel around the product with xi keeps it in registers (N = 8, 16 whole lines; 32,
64, 128, 256) or takes it through the tile (12-point plans), with row blocks that the planes do not
fill; plane wave and given field."""
import numpy as np
import pytest

from oracle import forward
from oracle.grid import Geometry as OGeom, layer_planes
from synth import random_gaussians

pytestmark = pytest.mark.gpu

SHAPES = [(8, 1, 2), (8, 9, 3), (12, 3, 2), (16, 5, 2), (24, 3, 2), (32, 3, 2), (48, 5, 2), (64, 3, 2), (96, 3, 2),
          (128, 3, 2), (192, 2, 1), (256, 2, 1)]


@pytest.mark.parametrize("precision, tol", [("fp64", 1e-11), ("mixed", 1e-5)])
@pytest.mark.parametrize("shape", SHAPES)
def test_fixed_point_lengths(shape, precision, tol):
    import torch
    from paper_1911_10487_gb300 import Geometry, Reconstructor
    n, m, n_om = shape
    rng = np.random.default_rng(n * 100 + m)
    g = OGeom(n, m, 0.2, 1.0, tuple(layer_planes(1.2, 1.6, 3)))
    om = list(np.pi * np.array([3.0, 2.2])[:n_om])  # 3 pi: grazing modes
    xi = random_gaussians(rng, n, m, g.z1, g.z2, 2, (0.15, 0.3), 0.05)
    rc = Reconstructor(0)
    geom = Geometry(n, m, g.z1, g.z2, g.zy, g.period)
    x = torch.from_numpy(xi).to("cuda", torch.float64 if precision == "fp64" else torch.float32)
    ref, ur = forward.make_data(xi, om, g, method="fixed_point")
    W, u, _ = rc.forward(x, om, geom, precision=precision, want_u=True)
    u0 = np.stack([np.broadcast_to(forward.incident_plane_wave(o, g), (m, n, n)) for o in om])
    u0 = torch.from_numpy(np.ascontiguousarray(u0)).to("cuda", W.dtype)
    Wi, _, _ = rc.forward(x, om, geom, precision=precision, incident=u0)
    torch.cuda.synchronize()
    rel = lambda a, b: np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)
    e = rel(W, ref), rel(u, ur), rel(Wi, ref)
    print(shape, precision, *(f"{v:.1e}" for v in e))
    assert max(e) <= tol
    rc.close()
