"""fs_forward that does not converge returns FS_ENOCONV with nothing left running, so that the caller
may reuse or free xi: at the cap of the iterations, and where the iterate grows out of range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["fixed_point", "fixed_point_gmres"])
@pytest.mark.parametrize("strength, max_iter", [(0.3, 3), (1e6, 50)])
def test_stream_is_idle_after_enoconv(strength, max_iter, method):
    import torch
    from paper_1911_10487_gb300 import FlatLayerError, Geometry, Reconstructor
    geom = Geometry(128, 64, 0.2, 1.0, tuple(1.2 + 0.1 * k for k in range(4)))
    xi = torch.zeros((64, 128, 128), dtype=torch.float64, device="cuda")
    xi[10:50, 30:90, 30:90] = strength
    rc = Reconstructor(0)
    busy = 0
    for _ in range(3):
        with pytest.raises(FlatLayerError, match="FS_ENOCONV"):
            rc.forward(xi, [8 * np.pi], geom, max_iter=max_iter, method=method)
        busy += not rc.stream.query()
    torch.cuda.synchronize()
    rc.close()
    assert busy == 0


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_convergence_in_the_last_iteration_allowed(precision):
    """The same data, to the bit, whether more iterations were allowed or not."""
    import torch
    from paper_1911_10487_gb300 import Geometry, Reconstructor
    geom = Geometry(24, 5, 0.2, 1.0, (1.3, 1.5))
    xi = torch.zeros((5, 24, 24), dtype=torch.float64 if precision == "fp64" else torch.float32, device="cuda")
    xi[1:4, 8:16, 8:16] = 0.05
    om = [2.2 * np.pi, 3.4 * np.pi]
    rc = Reconstructor(0)
    W, u, its = rc.forward(xi, om, geom, precision=precision, want_u=True)
    for f in (0, 1):
        W1, u1, it1 = rc.forward(xi, om[f:f + 1], geom, precision=precision, max_iter=its[f], want_u=True)
        assert it1 == [its[f]] and torch.equal(W1[0], W[f]) and torch.equal(u1[0], u[f])
    rc.close()
