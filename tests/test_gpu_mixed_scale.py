"""FS_MIXED on data far from unit size.  W and W 2^k differ in their exponents alone, and so do
||W||, the modes' norms and delta_nu: the same modes are active and alpha is the same (2e-6, a few
FP32 roundings) while the modes' own squares |W~|^2 stay in the FP32 range: from the size where those
of the threshold's modes are still normal, with W~ up to N^2 times W, to the other end.  Where a mode
at the threshold has a square of two units of the FP32 format's end, the noise modes' squares (6e-5 of
||W||^2) may be lost and no more: the same modes, alpha to 1e-2 (slopes of the discrepancy function of
0.02 and more).  The forward transform in one pass, in two, and in two with the norms joined to it."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, m1, n_om, single", [(32, 6, 2, 1), (32, 6, 2, 0), (128, 4, 1, 1), (128, 4, 1, 0), (128, 64, 2, 0),
                                                 (192, 20, 2, 0)])
def test_scaled_data(n, m1, n_om, single):
    import torch
    from paper_1911_10487_gb300 import Geometry, Reconstructor
    rng = np.random.default_rng(n + m1)
    m, om = 8, [2.3 * math.pi, 3.6 * math.pi][:n_om]
    geom = Geometry(n, m, 0.2, 1.0, tuple(1.2 + 0.4 * k / m1 for k in range(m1)))
    b = np.zeros((n_om, m1, n, n), complex)
    b[..., :5, :5] = rng.standard_normal((n_om, m1, 5, 5)) + 1j * rng.standard_normal((n_om, m1, 5, 5))
    W = np.fft.ifft2(b)
    noise = rng.standard_normal(W.shape) + 1j * rng.standard_normal(W.shape)
    W += 0.008 * np.linalg.norm(W) / np.linalg.norm(noise) * noise
    W = torch.from_numpy(W / np.abs(W).max()).to("cuda", torch.complex64)
    rms = float(torch.sqrt(torch.mean(torch.abs(W.double() if not W.is_complex() else W.to(torch.complex128)) ** 2)))
    rc = Reconstructor(0)
    run = lambda x: rc.reconstruct(x, om, geom, 0.01, precision="mixed", solve_form=1, forward_single_pass=single,
                                   want_alpha=True)[2].cpu()
    ref, rep = run(W), rc.report()
    # threshold: delta_nu^2 = 4e-4 ||W||^2 = 4e-4 rms^2 N^2 M1; normal above 2^-126, with 2^20 to spare
    size = math.log2(4e-4 * rms ** 2 * n * n * m1)
    lo, end = math.ceil(0.5 * (-126 + 20 - size)), math.ceil(0.5 * (-149 + 1 - size))
    hi = math.floor(0.5 * (127 - 4 - math.log2(m1 * float(n) ** 4)))
    for k in (lo, lo // 2, 20, hi, end):
        s = 2.0 ** (k // 2)
        got, r = run((W * s) * 2.0 ** (k - k // 2)), rc.report()
        act = torch.isfinite(ref)
        same = bool((torch.isfinite(got) == act).all())
        err = float((got[act] / ref[act] - 1).abs().max()) if same else math.inf
        print(f"N={n} single={single} 2^{k}: active {r['n_active']} of {rep['n_active']}, alpha {err:.1e}")
        assert same and r["n_active"] == rep["n_active"] and err <= (2e-6 if k > end else 1e-2)
    rc.close()
