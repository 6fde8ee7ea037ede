"""FS_MIXED recovery at N = 192 and 256: V and u of a voxel as packed pairs, against the general pass (the
small-tile form of the same transforms): xi to the rounding of two factorisations of the FP32
transforms (relative L2 2e-6), the same guarded voxels.  Plane wave and a given field, FP32 and FP64
sums, one frequency and several, columns within one sixteenth of the band, two, and beyond (the highest
frequency), with more columns than a block stages."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [(256, 1, (2.3,)), (256, 3, (2.3, 24.0, 70.0)), (192, 1, (3.1, 40.0)), (192, 2, (2.3,))]


@pytest.mark.parametrize("given, fp64_sums", [(False, 0), (True, 0), (False, 1), (True, 1)])
@pytest.mark.parametrize("n, m, k", CASES)
def test_pairs_match_the_general_pass(n, m, k, given, fp64_sums):
    import torch
    from oracle import forward
    from oracle.grid import Geometry as OGeom, layer_planes
    from paper_1911_10487_gb300 import Geometry, Reconstructor
    from synth import random_gaussians
    rng = np.random.default_rng(n + m)
    zy = tuple(layer_planes(1.2, 1.6, 9))
    geom, og = Geometry(n, m, 0.2, 1.0, zy), OGeom(n, m, 0.2, 1.0, zy)
    om = list(np.pi * np.array(k))
    rc = Reconstructor(0)
    xi = torch.from_numpy(random_gaussians(rng, n, m, 0.2, 1.0, 2, (0.1, 0.3), 0.05)).cuda()
    u0 = np.stack([np.broadcast_to(forward.incident_plane_wave(o, og), (m, n, n)) for o in om])
    u0 = torch.from_numpy(np.ascontiguousarray(u0)).cuda()
    W = rc.forward_born(xi, om, geom)
    e = torch.view_as_complex(torch.randn(tuple(W.shape) + (2,), dtype=torch.float64, device="cuda",
                                          generator=torch.Generator("cuda").manual_seed(3)))
    for j in range(len(om)):
        W[j] += 0.008 * torch.linalg.vector_norm(W[j]) / torch.linalg.vector_norm(e[j]) * e[j]
    W, u0 = W.to(torch.complex64), u0.to(torch.complex64)
    got = []
    for tile in (0, 1):
        x, _, _ = rc.reconstruct(W, om, geom, 0.01, precision="mixed", solve_form=1, fft_tile=tile,
                                 fp64_sums=fp64_sums, **({"incident": u0} if given else {}))
        got.append((x.double(), rc.report()))
    rc.close()
    (a, ra), (b, rb) = got
    err = float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))
    print(n, m, k, given, fp64_sums, f"{err:.1e}", ra["n_active"], ra["n_columns"])
    assert ra["n_active"] == rb["n_active"] > 0 and ra["n_u_guard"] == rb["n_u_guard"]
    assert err <= 2e-6
