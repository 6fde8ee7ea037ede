"""Single-scattering data of a weak plane beside a strong one.  The data are linear in xi, and a strong
plane below, of wavenumbers that do not reach the data, must leave the weak plane's share what it is:
at modes nu whose field decays by q = e^{-|k_z| h_z} from plane to plane, the strong plane's rounding,
some eps A N a mode of its transform beside the weak plane's N^2 / 2, arrives as eps A q.  Held to
32 eps A q / N (ten butterfly stages, the differences taken here) + 8 eps max|W| over the share of one
of the weak plane's modes, on a layer of which only mode 0 propagates."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision, big, eps", [("fp64", 2.0 ** 40, 2.0 ** -52), ("mixed", 2.0 ** 15, 2.0 ** -23)])
@pytest.mark.parametrize("n, m", [(8, 2), (12, 3), (16, 4), (24, 2), (32, 9), (48, 3), (64, 2), (96, 3), (128, 2), (192, 2), (256, 2)])
def test_weak_plane_beside_a_strong_one(n, m, precision, big, eps):
    import torch
    from paper_1911_10487_gb300 import Geometry, Reconstructor
    rng = np.random.default_rng(n + m)
    hz, om = 2.0, 1.0
    geom = Geometry(n, m, 0.2, 0.2 + hz * m, (0.25 + hz * m, 0.3 + hz * m))
    x = np.arange(n) * (2 * np.pi / n)
    weak, strong = np.zeros((m, n, n)), np.zeros((m, n, n))
    weak[m - 1] = np.cos(2 * x)[None, :] + np.cos(2 * x + 0.4)[:, None]
    band = np.fft.fft2(rng.uniform(-1, 1, (n, n)))
    mi = np.abs(np.fft.fftfreq(n) * n)
    band[np.maximum(mi[:, None], mi[None, :]) < 3] = 0  # the highest wavenumbers only
    s = np.fft.ifft2(band).real
    dt, rdt = (torch.float64, np.float64) if precision == "fp64" else (torch.float32, np.float32)
    strong[m - 2] = (big * s / np.abs(s).max()).astype(rdt)
    rc = Reconstructor(0)
    W = [rc.forward_born(torch.from_numpy(a).to("cuda", dt), [om], geom, precision=precision).cpu().numpy()[0].astype(complex)
         for a in (weak + strong, strong, weak)]
    rc.close()
    F = [np.fft.fft2(w) for w in W]
    kz = np.sqrt((2 * np.pi) ** 2 - om ** 2)  # of the weak plane's modes (+-2, 0), (0, +-2)
    worst = 0.0
    for i, j in ((0, 2), (0, n - 2), (2, 0), (n - 2, 0)):
        got, ref = F[0][:, i, j] - F[1][:, i, j], F[2][:, i, j]
        tol = 32 * eps * big * np.exp(-kz * hz) / n + 8 * eps * n * n * max(np.abs(w).max() for w in W) / np.abs(ref)
        worst = max(worst, np.max(np.abs(got - ref) / np.abs(ref) / tol))
    print(f"N={n} M={m} {precision}: {worst:.2g} of the tolerance")
    assert worst <= 1
