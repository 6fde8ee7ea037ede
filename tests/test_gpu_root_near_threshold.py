"""Modes just above the discrepancy threshold, through the dense FP64 solve.  With ||b||^2 =
delta_nu^2 / (1 - e) the discrepancy function has slope g' = d log phi^2 / d log alpha ~ e at its root:
a residual of rounding size, a few eps, moves log alpha by a few eps / e.  Held to 100 eps / e + 1e-12
relative of the rank-one closed form in extended precision: eps = 2.2e-16 of the norms of b and W, of
the transform, of the tridiagonal model and of the residual, some ten each."""
import numpy as np
import pytest
import scipy.fft

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, m, m1, seed", [(32, 8, 6, 1), (32, 16, 12, 2), (24, 5, 2, 3)])
def test_alpha_of_modes_near_delta(n, m, m1, seed):
    import torch
    from paper_1911_10487_gb300 import Geometry, Reconstructor
    LD, CLD = np.longdouble, np.clongdouble
    rng = np.random.default_rng(seed)
    om = 2.3 * np.pi
    zy = tuple(1.2 + 0.4 * k / m1 for k in range(m1))
    geom = Geometry(n, m, 0.2, 1.0, zy)
    idx = [(i, j) for i in range(-4, 5) for j in range(-4, 5)]
    e = np.exp(rng.uniform(np.log(1e-5), np.log(1e-2), len(idx)))
    b = np.zeros((m1, n, n), complex)
    hz, pi = (LD(1.0) - LD(0.2)) / m, LD(np.pi) + LD(1.2246467991473532e-16)
    zc = LD(0.2) + (np.arange(m).astype(LD) + LD(0.5)) * hz
    E, sP = {}, {}
    for (i, j) in idx:
        qq = LD(om) ** 2 - pi ** 2 * (i * i + j * j)
        kz = CLD(np.sqrt(qq)) if qq > 0 else CLD(1j) * np.sqrt(-qq)
        E[i, j] = LD(om) ** 2 * hz * CLD(-0.5j) / kz * np.exp(CLD(1j) * kz * (np.array(zy, LD) - zc[-1]))
        sP[i, j] = (np.abs(np.exp(CLD(1j) * kz * (zc[-1] - zc))) ** 2).sum()
    for (i, j), t in zip(idx, e):  # along E and across it; ||b|| = 1 / sqrt(1 - e)
        u = (E[i, j] / np.sqrt((np.abs(E[i, j]) ** 2).sum())).astype(complex)
        v = u * np.exp(1j * rng.uniform(0, 6)) + 0.3 * (rng.standard_normal(m1) + 1j * rng.standard_normal(m1)) / np.sqrt(m1)
        b[:, i, j] = v / np.linalg.norm(v) / np.sqrt(1 - t)
    W = np.fft.ifft2(b)
    wn = np.sqrt((np.abs(W.astype(CLD)) ** 2).sum())
    delta = float(1 / (2 * wn))  # delta_nu = 2 delta ||W|| ~ 1
    dnu2 = (2 * LD(delta) * wn) ** 2
    rc = Reconstructor(0)
    _, _, alpha = rc.reconstruct(torch.from_numpy(W[None]).cuda(), [om], geom, delta, want_alpha=True)
    torch.cuda.synchronize()
    rep = rc.report()
    rc.close()
    alpha = alpha.cpu().numpy()[0]
    bt = scipy.fft.fft2(W.astype(CLD))
    worst = 0.0
    for (i, j) in idx:
        x, Em = bt[:, i, j], E[i, j]
        sE, bb = (np.abs(Em) ** 2).sum(), (np.abs(x) ** 2).sum()
        c = np.abs((Em.conj() * x).sum()) ** 2 / sE
        # phi^2 = k^2 c + bb - c = delta_nu^2, k = alpha / (tr + alpha)
        k2 = 1 - (bb - dnu2) / c
        k = np.sqrt(k2)
        ref = sE * sP[i, j] * k * (1 + k) / (1 - k2)
        t = float((bb - dnu2) / dnu2)
        got = abs(float(alpha[i, j] / ref) - 1)
        worst = max(worst, got / (100 * 2.2e-16 / t + 1e-12))
    print(f"N={n} M1={m1}: {worst:.2g} of the tolerance; capped {rep['n_root_capped']}, floor {rep['n_alpha_floor']}")
    assert worst <= 1
