"""The allocation-free entry point takes what fits its fixed scratch: the intermediates of
fs_reconstruct laid out one after another, each on a 256-byte boundary, then counters and twiddles.
Arrays that only one route of the classification needs lie inside those of another, so that the
accepted set is a function of these sizes alone.  Checked at the largest M accepted and the next one
over frequencies and data planes, on the CPU: a size that fits goes on to the device and fails there
(FS_ECUDA), one that does not is refused before (FS_EUNSUPPORTED)."""
import ctypes as C
import random

import pytest

SIZES = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256)


def up(v):
    return (v + 255) // 256 * 256


def scratch_bytes(n, m, m1, f, fp64):
    cx, n2 = 16 if fp64 else 8, n * n
    cb = f * ((n2 + 1023) // 1024)
    parts = [max(16 * f * m1 * n2, 2 * cx * f * m * n2), 2 * cx * f * m * n2,  # transforms, profiles
             8 * f * n2, 8 * f * ((n2 + 63) // 64), 4 * f * n2, 4 * f * n2,  # norms, their sums, slots, active modes
             128 * cb, 4 * cb, 4 * cb, 32 * cb,  # flags, counts, column masks per block
             4 * f * n, 4 * f, 4 * f, 8 * f, 4 * f]  # columns, their number, active, delta_nu, barriers
    b = sum(up(v) for v in parts)
    return up(up(up(b + 8 * 16) + (16 if fp64 else 8) * n) + 16 * n)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_accepted_sizes(prec):
    import torch
    if torch.cuda.is_available():
        pytest.skip("the fake addresses are for a machine without a GPU")
    from paper_1911_10487_gb300 import _abi as abi, build
    build.build()
    L, fp64 = abi.lib(), prec == "fp64"
    o = abi.make_options(solve_form=1)
    om = (C.c_double * 64)(*([1.0] * 64))

    def status(n, m, m1, f):
        g = abi.make_geometry(n, m, 0.2, 1.0, [1.2 + 0.01 * k for k in range(m1)])
        return L.fs_reconstruct_static(C.byref(g), abi.FS_FP64 if fp64 else abi.FS_MIXED, C.c_void_p(1 << 20), om, f,
                                       0.01, 1.0, C.byref(o), C.c_void_p(1 << 20), None, None)

    rng = random.Random(5)
    cases = [(24, 5, 34), (24, 5, 64), (8, 128, 64)] + [(rng.choice(SIZES), rng.randint(1, 128), rng.randint(1, 64))
                                                        for _ in range(1500)]
    edges = 0
    for n, m1, f in cases:
        fits = [m for m in range(1, 129) if scratch_bytes(n, m, m1, f, fp64) <= 32 << 20]
        m = max(fits, default=0)
        if m:
            assert status(n, m, m1, f) == 3, (n, m, m1, f)  # FS_ECUDA
        if m < 128:
            edges += 1
            assert status(n, m + 1, m1, f) == abi.FS_EUNSUPPORTED, (n, m + 1, m1, f)
    assert edges > 300


@pytest.mark.gpu
@pytest.mark.parametrize("shape, prec, form", [((24, 53, 5, 34), "mixed", 1), ((24, 53, 5, 34), "fp64", 0), ((8, 127, 128, 64), "fp64", 1),
                                               ((8, 128, 128, 64), "mixed", 1)])
def test_at_the_edge_equals_the_context_entry(shape, prec, form):
    """A size near the limit, or the most frequencies and planes: the same xi as fs_reconstruct to the
    parity tolerances (1e-10 FS_FP64, 1e-5 FS_MIXED), or refused where it does not fit."""
    import numpy as np
    import torch
    from paper_1911_10487_gb300 import FS_FP64, FS_MIXED, Geometry, Reconstructor, _abi as abi
    n, m, m1, f = shape
    fp64 = prec == "fp64"
    rng = np.random.default_rng(n + m + f)
    geom = Geometry(n, m, 0.2, 1.0, tuple(1.2 + 0.4 * k / m1 for k in range(m1)))
    om = [float(v) for v in np.linspace(3.1, 9.7, f)]
    modes = np.zeros((f, m1, n, n), complex)
    modes[..., :3, :3] = rng.standard_normal((f, m1, 3, 3)) + 1j * rng.standard_normal((f, m1, 3, 3))
    W = torch.from_numpy(np.fft.ifft2(modes)).to("cuda", torch.complex128 if fp64 else torch.complex64)
    rc = Reconstructor(0)
    ref, _, _ = rc.reconstruct(W, om, geom, 0.05, precision=prec, solve_form=form)
    xi = torch.full_like(ref, float("nan"))
    st = abi.fs_reconstruct_static(geom.c_struct(), FS_FP64 if fp64 else FS_MIXED, W.data_ptr(), om, 0.05, 1.0,
                                   abi.make_options(solve_form=form), xi.data_ptr(), None, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    rc.close()
    if scratch_bytes(n, m, m1, f, fp64) > 32 << 20:
        assert st == abi.FS_EUNSUPPORTED
        return
    assert st == abi.FS_OK
    err = float(torch.linalg.vector_norm((xi - ref).double()) / torch.linalg.vector_norm(ref.double()))
    print(shape, prec, f"{err:.1e}")
    assert err <= (1e-10 if fp64 else 1e-5)
