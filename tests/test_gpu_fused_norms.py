"""FS_MIXED: the pass that transforms the data planes' columns and sums the norms at once, and
leaves W~ to a transform of the active columns, against the separate passes, which the
single-launch classification still takes: same active modes, and xi to the rounding of the two
orders of summation (relative L2 2e-6, the FP32 norms and sums).  Sizes: last tiles of 4 planes,
groups of one and several planes, the cap of 4 M groups (M = 1), from the 8 MB up at which it is
taken, a 3-smooth length, one frequency beside several, and the two-pass form at N = 128."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [(256, 2, 16, 1), (256, 5, 30, 3), (192, 1, 15, 2), (192, 6, 31, 1), (128, 2, 31, 3)]


@pytest.mark.parametrize("n, m, m1, n_om", CASES)
def test_fused_norms_match_the_separate_passes(n, m, m1, n_om):
    import torch
    from oracle.grid import layer_planes
    from paper_1911_10487_gb300 import Geometry, Reconstructor
    from synth import random_gaussians
    rng = np.random.default_rng(n + 100 * m + m1)
    geom = Geometry(n, m, 0.2, 1.0, tuple(layer_planes(1.2, 1.6, m1)))
    om = list(np.pi * np.array([2.3, 3.0, 4.1])[:n_om])
    rc = Reconstructor(0)
    xi = torch.from_numpy(random_gaussians(rng, n, m, 0.2, 1.0, 2, (0.1, 0.3), 0.05)).cuda()
    W = rc.forward_born(xi, om, geom)
    e = torch.view_as_complex(torch.randn(tuple(W.shape) + (2,), dtype=torch.float64, device="cuda",
                                          generator=torch.Generator("cuda").manual_seed(3)))
    for j in range(n_om):
        W[j] += 0.008 * torch.linalg.vector_norm(W[j]) / torch.linalg.vector_norm(e[j]) * e[j]
    W = W.to(torch.complex64)
    got = []
    for single in (0, 1):
        x, _, _ = rc.reconstruct(W, om, geom, 0.01, precision="mixed", solve_form=1, classify_single_pass=single,
                                 forward_single_pass=0)
        got.append((x.double(), rc.report()))
    rc.close()
    (a, ra), (b, rb) = got
    err = float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))
    print(n, m, m1, n_om, f"{err:.1e}", ra["n_active"])
    assert ra["n_active"] == rb["n_active"] > 0 and ra["n_columns"] == rb["n_columns"]
    assert err <= 2e-6
