"""Workloads that stand for the use of this library: what a program has in hand (prepare), one
pass through the public entry points (run), the work it cannot do without (work) and the same
outputs by plain FP64 torch / numpy without the library (exact).

Geometries: "box" is X = [-1,1]^2 x [0.2,1.0] with data planes in [1.2,1.6], period 2;
"paper" is the layer of the paper's own experiment (Sec. 5): X = [-10,10]^2 x [-0.5,1.5], data in
[6.01,6.5], period 20, eleven point sources.  Frequencies are omega = k pi (box) or omega = k
(paper), k from k_lo to k_hi.  The data carry complex Gaussian noise of 0.8 delta ||W||.
"""
import math

import numpy as np
import torch

from paper_1911_10487_gb300 import FS_FP64, FS_MIXED, Geometry, KernelPlan, Reconstructor, fs_reconstruct_host, make_options
from paper_1911_10487_gb300.diff import DiffPlan, reconstruct_diff

SIZES = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256)
BATCH_GRIDS = ((64, 16), (128, 32), (192, 48), (256, 64))
TAU, DELTA_FLOOR, ALPHA_REL, EPS_U = 2.0, 1e-5, 1e-6, 1e-8  # the library's defaults


def _case(kind, n, m, m1, f, precision, k_lo, k_hi, name=None, **more):
    c = {"kind": kind, "n": n, "m": m, "m1": m1, "f": f, "precision": precision, "k_lo": k_lo, "k_hi": k_hi, **more}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: one frequency on a 32 x 32 grid, default options; latency and launches count
        _case("reconstruct", 32, 16, 8, 1, "fp64", 4.0, 4.0, "small32_fp64_dense", form="dense", delta=0.01, layer="box"),
        # an ordinary call with default options (the dense per-mode solve) in the mixed precision
        _case("reconstruct", 128, 64, 32, 1, "mixed", 8.0, 8.0, "rec128_mixed_dense", form="dense", delta=0.01, layer="box"),
        # the same with the closed form of the solve: the interactive case of a single-frequency survey
        _case("reconstruct", 128, 64, 32, 1, "mixed", 8.0, 8.0, "rec128_mixed_rank1", form="rank1", delta=0.01, layer="box"),
        # the same from and to page-locked host memory, as an acquisition loop with several buffers calls it
        _case("host", 128, 64, 32, 1, "mixed", 8.0, 8.0, "host128_mixed_rank1", form="rank1", delta=0.01, layer="box"),
        # a large multi-frequency reconstruction
        _case("reconstruct", 256, 64, 32, 8, "mixed", 2.0, 12.0, "rec256x8_mixed_rank1", form="rank1", delta=0.01, layer="box"),
        # the paper's experiment in FP64: an odd number of planes, three frequencies, a given incident field
        _case("reconstruct", 128, 71, 71, 3, "fp64", 1.0, 3.0, "paper128x71_fp64", form="rank1", delta=1e-5, layer="paper"),
        # many uneven problems in one call (grids 64^2 x 16 .. 256^2 x 64, 1-8 frequencies, 4-32 planes)
        {"name": "batch32_mixed_rank1", "kind": "batch", "count": 32, "draw": 3, "precision": "mixed", "form": "rank1",
         "delta": 0.01, "streams": 16},
        # the sampled-G kernel of Sec. 5 with a plan kept for the geometry, FP64, 3-smooth grid
        _case("sampled", 48, 24, 12, 2, "fp64", 3.0, 7.5, "sampled48_fp64", delta=0.01, layer="box"),
        # single-scattering data of several frequencies on a ragged grid, FP64
        _case("born", 192, 37, 19, 5, "fp64", 2.0, 9.0, "born192x37_fp64", layer="box"),
        # full-scattering data by the fixed point of Algorithm 1, FP64, field on X wanted too
        _case("forward", 128, 64, 32, 1, "fp64", 8.0, 8.0, "forward128_fp64", layer="box"),
        # one gradient step through the reconstruction: forward, loss, gradients of W and log alpha
        _case("diff_step", 128, 64, 32, 4, "mixed", 4.0, 10.0, "diff128x4_mixed", layer="box"),
        # the sensitivity study: 16 perturbations of the data pushed forward from a kept tape
        _case("diff_jvp", 128, 64, 32, 4, "mixed", 4.0, 10.0, "jvp128x4_mixed", dirs=16, layer="box"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["reconstruct", "reconstruct", "reconstruct", "host", "batch", "sampled", "born", "forward",
                       "diff_step", "diff_jvp"])
    precision = rng.choice(["fp64", "mixed"])
    k_lo = round(rng.uniform(2.0, 6.0), 3)
    k_hi = round(rng.uniform(k_lo + 0.5, 12.0), 3)
    if kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 4, 24), "draw": rng.randrange(1 << 20), "precision": "mixed",
                "form": rng.choice(["dense", "rank1"]), "delta": 0.01, "streams": rng.choice([4, 8, 16, 32])}
    if kind == "sampled":
        return _case(kind, rng.choice([16, 24, 32, 48]), rng.randint(8, 24), rng.randint(4, 12), rng.randint(1, 2),
                     precision, k_lo, min(k_hi, 8.0) if k_lo < 7.5 else k_hi, delta=0.01, layer="box")
    if kind == "forward":
        n = rng.choice([16, 24, 32, 48, 64, 96, 128])
        return _case(kind, n, _log_int(rng, 8, 64), _log_int(rng, 4, 32), 1, "fp64", k_lo, min(k_hi, 8.0), layer="box")
    if kind == "born":
        return _case(kind, rng.choice(SIZES[:-1]), _log_int(rng, 4, 37), _log_int(rng, 4, 19), rng.randint(1, 5),
                     precision, k_lo, k_hi, layer="box")
    if kind in ("diff_step", "diff_jvp"):
        n = rng.choice([16, 24, 32, 48, 64, 96])
        c = _case(kind, n, _log_int(rng, 4, 64), _log_int(rng, 4, 32), rng.randint(1, 4), precision, k_lo, k_hi, layer="box")
        if kind == "diff_jvp":
            c["dirs"] = rng.randint(1, 16)
        return c
    form = rng.choice(["dense", "rank1"])
    n = rng.choice(SIZES if precision == "mixed" else SIZES[:-1])
    return _case(kind, n, _log_int(rng, 4, 64 if form == "dense" else 96), _log_int(rng, 4, 32), rng.randint(1, 6),
                 precision, k_lo, k_hi, form=form, delta=rng.choice([0.005, 0.01, 0.05]), layer="box")


# ---- geometry and inputs ---------------------------------------------------------

def _geometry(n, m, m1, layer="box"):
    z1, z2, z3, z4, period = (-0.5, 1.5, 6.01, 6.5, 20.0) if layer == "paper" else (0.2, 1.0, 1.2, 1.6, 2.0)
    zy = tuple(z3 + (z4 - z3) * k / max(m1 - 1, 1) for k in range(m1))
    return Geometry(n=n, m=m, z1=z1, z2=z2, zy=zy, period=period)


def _omegas(case):
    unit = 1.0 if case["layer"] == "paper" else math.pi
    f = case["f"]
    if f == 1:
        return [unit * case["k_lo"]]
    return [unit * (case["k_lo"] + (case["k_hi"] - case["k_lo"]) * j / (f - 1)) for j in range(f)]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _phantom(geom, seed, peak):
    """Three Gaussian inclusions with random centres and widths, peaks +-peak (one sign per inclusion)."""
    r = np.random.default_rng([seed, 17])
    half, hz = 0.5 * geom.period, (geom.z2 - geom.z1) / geom.m
    x = torch.arange(geom.n, device="cuda", dtype=torch.float64) * (geom.period / geom.n) - half
    z = geom.z1 + (torch.arange(geom.m, device="cuda", dtype=torch.float64) + 0.5) * hz
    xi = torch.zeros((geom.m, geom.n, geom.n), device="cuda", dtype=torch.float64)
    for _ in range(3):
        s = r.uniform(0.05, 0.2) * half
        cx, cy, cz = r.uniform(-half + s, half - s), r.uniform(-half + s, half - s), r.uniform(geom.z1, geom.z2)
        p = peak * r.choice([-1.0, 1.0])
        gx, gy = torch.exp(-(x - cx) ** 2 / (2 * s * s)), torch.exp(-(x - cy) ** 2 / (2 * s * s))
        gz = torch.exp(-(z - cz) ** 2 / (2 * s * s))
        xi += p * gz[:, None, None] * gy[None, :, None] * gx[None, None, :]
    return xi


class _Modes:
    """E_k, P_l, q and gamma of the Weyl kernel for every mode of one frequency (FP64)."""

    def __init__(self, geom, om, c0=1.0):
        n, hz = geom.n, (geom.z2 - geom.z1) / geom.m
        mi = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64).mul(n).round()
        msq = mi[:, None] ** 2 + mi[None, :] ** 2
        s2 = (om / c0 * geom.period / (2 * math.pi)) ** 2
        self.graz = (msq - s2).abs() <= 1e-9 * s2
        q = torch.where(self.graz, torch.ones_like(msq), (om / c0) ** 2 - (2 * math.pi / geom.period) ** 2 * msq)
        zero = torch.zeros_like(q)
        root = q.abs().sqrt()
        self.kz = torch.complex(torch.where(q > 0, root, zero), torch.where(q > 0, zero, root))
        self.gamma = torch.where(self.graz, 0.0, om ** 2 * hz * (-0.5j) / self.kz)
        self.ztop = geom.z1 + (geom.m - 0.5) * hz
        zx = geom.z1 + (torch.arange(geom.m, device="cuda", dtype=torch.float64) + 0.5) * hz
        zy = torch.tensor(geom.zy, device="cuda", dtype=torch.float64)
        self.E = self.gamma * torch.exp(1j * self.kz * (zy - self.ztop)[:, None, None])
        self.P = torch.exp(1j * self.kz * (self.ztop - zx)[:, None, None])
        self.q = torch.exp(1j * self.kz * hz)
        self.tr = (self.E.abs() ** 2).sum(0) * (self.P.abs() ** 2).sum(0)

    def interior(self, v):
        """omega^2 T_nu v: gamma (F + B) by the two recurrences of eq. (9)."""
        m = v.shape[0]
        f, out = torch.zeros_like(v[0]), []
        for l in range(m):
            f = self.q * f + v[l]
            out.append(f)
        b = torch.zeros_like(v[0])
        for l in range(m - 1, -1, -1):
            out[l] = self.gamma * (out[l] + b)
            b = self.q * (b + v[l])
        return torch.stack(out)


def _plane_wave(geom, om, c0=1.0):
    hz = (geom.z2 - geom.z1) / geom.m
    z = geom.z1 + (torch.arange(geom.m, device="cuda", dtype=torch.float64) + 0.5) * hz
    return torch.exp(-1j * (om / c0) * z)[:, None, None].expand(geom.m, geom.n, geom.n)


def _point_sources(geom, om, c0=1.0):
    """The field of eleven unit sources (0, y, 6), y = -5..5, on the X planes, periodised."""
    n, hz = geom.n, (geom.z2 - geom.z1) / geom.m
    K = _Modes(geom, om, c0)
    mi = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64).mul(n).round() * (2 * math.pi / geom.period)
    z = geom.z1 + (torch.arange(geom.m, device="cuda", dtype=torch.float64) + 0.5) * hz
    x0 = -0.5 * geom.period
    ph = sum(torch.exp(-1j * (mi[None, :] * (0.0 - x0) + mi[:, None] * (y - x0))) for y in range(-5, 6))
    g = torch.where(K.graz, 0.0, -0.5j / K.kz)
    ut = (n * n / geom.period ** 2) * (g * ph) * torch.exp(1j * K.kz * (6.0 - z)[:, None, None])
    return torch.fft.ifft2(ut)


def _data(geom, omegas, seed, delta, u0=None):
    """Single-scattering data of a phantom plus noise of norm 0.8 delta ||W|| per frequency."""
    xi = _phantom(geom, seed, 0.1)
    gen = _generator(seed)
    W = torch.empty((len(omegas), geom.m1, geom.n, geom.n), device="cuda", dtype=torch.complex128)
    for j, om in enumerate(omegas):
        K = _Modes(geom, om)
        V = torch.fft.fft2(xi * (_plane_wave(geom, om) if u0 is None else u0[j]))
        W[j] = torch.fft.ifft2(K.E * (K.P * V).sum(0))
        e = torch.view_as_complex(torch.randn((geom.m1, geom.n, geom.n, 2), device="cuda", dtype=torch.float64, generator=gen))
        W[j] += (0.8 * delta * torch.linalg.vector_norm(W[j]) / torch.linalg.vector_norm(e)) * e
    return W


def _batch(case):
    """Sizes of the batch's problems (part of the case, not of the data)."""
    r = np.random.default_rng([case["draw"], 4])
    out = []
    for _ in range(case["count"]):
        n, m = BATCH_GRIDS[r.integers(0, 4)]
        om = sorted(float(x) for x in r.uniform(2 * math.pi, 12 * math.pi, int(r.integers(1, 9))))
        out.append((_geometry(n, m, int(r.integers(4, 33))), om))
    return out


def _cdt(case):
    return torch.complex128 if case["precision"] == "fp64" else torch.complex64


def _rdt(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _sampled_tables(geom, om, c0=1.0):
    """A_nu [N, N, M1, M] and the Toeplitz row of T_nu [N, N, M] of the sampled-G kernel."""
    n, m, hz, h = geom.n, geom.m, (geom.z2 - geom.z1) / geom.m, geom.period / geom.n
    k0 = om / c0
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    x = torch.where(i < n // 2, i, i - n) * h
    r2 = x[:, None] ** 2 + x[None, :] ** 2
    zx = geom.z1 + (torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) * hz
    zy = torch.tensor(geom.zy, device="cuda", dtype=torch.float64)
    dz = torch.cat([(zy[:, None] - zx[None, :]).reshape(-1), torch.arange(m, device="cuda", dtype=torch.float64) * hz])
    rho = torch.sqrt(r2 + dz[:, None, None] ** 2)
    own = rho == 0
    g = -h * h * torch.exp(1j * k0 * rho) / (4 * math.pi * torch.where(own, 1.0, rho))
    # the cell at rho = 0: the integral of G over the ball of equal volume, over h_z (series in x = k0 a)
    a = (3 * h * h * hz / (4 * math.pi)) ** (1.0 / 3.0)
    xa = k0 * a
    if xa > 1:
        ball = (1 - (1 - 1j * xa) * complex(math.cos(xa), math.sin(xa))) / k0 ** 2
    else:
        ball = a * a * sum((k - 1) * (1j ** k) * xa ** (k - 2) / math.factorial(k) for k in range(2, 40))
    g = torch.where(own, ball / hz, g)
    t = (om ** 2 * hz * torch.fft.fft2(g)).movedim(0, -1)
    return t[..., :geom.m1 * m].reshape(n, n, geom.m1, m).contiguous(), t[..., geom.m1 * m:].contiguous()


def _sampled_data(geom, omegas, seed, delta):
    xi = _phantom(geom, seed, 0.1)
    gen = _generator(seed)
    W = torch.empty((len(omegas), geom.m1, geom.n, geom.n), device="cuda", dtype=torch.complex128)
    for j, om in enumerate(omegas):
        A, _ = _sampled_tables(geom, om)
        V = torch.fft.fft2(xi * _plane_wave(geom, om)).movedim(0, -1)
        W[j] = torch.fft.ifft2((A @ V[..., None])[..., 0].movedim(-1, 0))
        e = torch.view_as_complex(torch.randn((geom.m1, geom.n, geom.n, 2), device="cuda", dtype=torch.float64, generator=gen))
        W[j] += (0.8 * delta * torch.linalg.vector_norm(W[j]) / torch.linalg.vector_norm(e)) * e
    return W


def _diff_inputs(case, seed):
    geom, om = _geometry(case["n"], case["m"], case["m1"]), _omegas(case)
    W = _data(geom, om, seed, 0.01)
    gen = _generator(seed + 1)
    la = math.log(0.1) + 0.3 * torch.randn(len(om), device="cuda", dtype=torch.float64, generator=gen)
    want = _phantom(geom, seed + 1, 0.1)
    target = (0.02 * torch.linalg.vector_norm(W.reshape(len(om), -1), dim=1)) ** 2 * geom.n ** 2
    return geom, om, W, la, want, target


def _directions(case, W, seed):
    """Perturbations of 1% of ||W|| per frequency, and of log alpha."""
    gen = _generator(seed + 2)
    d = torch.view_as_complex(torch.randn((case["dirs"],) + tuple(W.shape) + (2,), device="cuda", dtype=torch.float32,
                                          generator=gen))
    size = 0.01 * torch.linalg.vector_norm(W.reshape(W.shape[0], -1), dim=1) / math.sqrt(2 * W[0].numel())
    d = d * size.to(torch.float32)[None, :, None, None, None]
    dla = 0.1 * torch.randn((case["dirs"], W.shape[0]), device="cuda", dtype=torch.float64, generator=gen)
    return d, dla


_RC = {}


def _rc():
    """One reconstructor for the program, as a program keeps it."""
    if "rc" not in _RC:
        _RC["rc"] = Reconstructor(0)
    return _RC["rc"]


def _incident(case, geom, omegas):
    if case["layer"] != "paper":
        return None
    return torch.stack([_point_sources(geom, om) for om in omegas])


def prepare(case, seed):
    rc, kind = _rc(), case["kind"]
    if kind == "batch":
        items = [(_data(g, om, seed * 64 + j, case["delta"]).to(torch.complex64), om, g, case["delta"])
                 for j, (g, om) in enumerate(_batch(case))]
        return {"case": case, "rc": rc, "items": items}
    geom, om = _geometry(case["n"], case["m"], case["m1"], case["layer"]), _omegas(case)
    s = {"case": case, "rc": rc, "geom": geom, "om": om}
    if kind in ("reconstruct", "host"):
        u0 = _incident(case, geom, om)
        W = _data(geom, om, seed, case["delta"], u0).to(_cdt(case))
        s["opts"] = {"solve_form": 1} if case["form"] == "rank1" else {}
        if u0 is not None:
            s["opts"].update(incident=u0.to(_cdt(case)), delta_floor=1e-10)
        if kind == "reconstruct":
            s["W"] = W
        else:
            s["W"] = W.cpu().pin_memory()
            s["xi"] = torch.empty((geom.m, geom.n, geom.n), dtype=_rdt(case)).pin_memory()
            s["g"], s["o"] = geom.c_struct(), make_options(**s["opts"])
    elif kind == "sampled":
        s["W"] = _sampled_data(geom, om, seed, case["delta"]).to(_cdt(case))
        s["plan"] = KernelPlan(rc, geom, om, case["precision"])
    elif kind in ("born", "forward"):
        s["xi"] = _phantom(geom, seed, 0.05).to(_rdt(case))
    else:
        _, _, W, la, want, target = _diff_inputs(case, seed)
        s["plan"] = DiffPlan(rc, geom, om, case["precision"])
        s["W"], s["la"] = W.to(_cdt(case)), la
        if kind == "diff_step":
            s["W"].requires_grad_(True)
            s["la"] = la.requires_grad_(True)
            s["want"], s["target"] = want.to(_rdt(case)), target
        else:
            _, _, _, s["tape"] = s["plan"].forward(s["W"], la)
            d, s["dla"] = _directions(case, W, seed)
            s["dW"] = d.to(_cdt(case))
    return s


def _loss(xi, phi, want, target):
    return ((xi - want) ** 2).sum() + ((phi / target - 1.0) ** 2).sum()


def run(s):
    case, rc = s["case"], s["rc"]
    kind = case["kind"]
    if kind == "reconstruct":
        xi, c, _ = rc.reconstruct(s["W"], s["om"], s["geom"], case["delta"], precision=case["precision"], **s["opts"])
        return {"xi": xi, "c": c}
    if kind == "host":
        fs_reconstruct_host(rc.ctx, s["g"], FS_FP64 if case["precision"] == "fp64" else FS_MIXED, s["W"].data_ptr(),
                            s["om"], case["delta"], 1.0, s["o"], s["xi"].data_ptr(), None)
        return {"xi": s["xi"]}
    if kind == "batch":
        opts = {"solve_form": 1} if case["form"] == "rank1" else {}
        res = rc.reconstruct_batch(s["items"], precision=case["precision"], n_streams=case["streams"], **opts)
        return {"xi": [r[0] for r in res], "c": [r[1] for r in res]}
    if kind == "sampled":
        xi, c, _ = rc.reconstruct(s["W"], s["om"], s["geom"], case["delta"], precision=case["precision"],
                                  kernel_plan=s["plan"])
        return {"xi": xi, "c": c}
    if kind == "born":
        return {"W": rc.forward_born(s["xi"], s["om"], s["geom"], precision=case["precision"])}
    if kind == "forward":
        W, u, _ = rc.forward(s["xi"], s["om"], s["geom"], precision=case["precision"], want_u=True)
        return {"W": W, "u": u}
    if kind == "diff_step":
        xi, phi = reconstruct_diff(s["W"], s["la"], s["plan"])
        gW, gla = torch.autograd.grad(_loss(xi, phi, s["want"], s["target"]), (s["W"], s["la"]))
        return {"xi": xi, "phi": phi, "gW": gW, "gla": gla}
    dxi, dphi = s["plan"].jvp(s["tape"], s["dW"], s["dla"])
    return {"dxi": dxi, "dphi": dphi}


# ---- work ------------------------------------------------------------------------

def _fft_flops(n, planes):
    return 5.0 * planes * n * n * 2 * math.log2(n)


def work(case):
    kind = case["kind"]
    s = 16 if case["precision"] == "fp64" else 8
    if kind == "batch":
        b = f = 0.0
        for g, om in _batch(case):
            w = work({**case, "kind": "reconstruct", "n": g.n, "m": g.m, "m1": g.m1, "f": len(om), "layer": "box"})
            b, f = b + w["bytes"], f + w["flops"]
        return {"bytes": b, "flops": f}
    n, m, m1, fr = case["n"], case["m"], case["m1"], case["f"]
    N2, data, vox = n * n, case["f"] * case["m1"] * n * n, case["m"] * n * n
    if kind in ("reconstruct", "host", "sampled"):
        # W in, xi and c out; the forward transforms, and the inverse ones of V and u along x
        inc = fr * vox * s if case["layer"] == "paper" else 0
        return {"bytes": s * data + s * vox + inc, "flops": _fft_flops(n, fr * m1) + _fft_flops(n, 2 * fr * m) / 2 + 8.0 * fr * vox}
    if kind in ("born", "forward"):
        # one application at least: two transforms of the M planes, one of the data planes
        reps = 1 if kind == "born" else 2
        out = s * data + (s * fr * vox if kind == "forward" else 0)
        return {"bytes": s / 2 * vox + out, "flops": reps * _fft_flops(n, fr * m) + _fft_flops(n, fr * m1) + 16.0 * fr * N2 * (m + m1)}
    per_mode = 16.0 * fr * N2 * (m + m1)
    if kind == "diff_step":
        # W in, xi out, gradient of W out; transforms of W, V, u and of their cotangents
        return {"bytes": 2 * s * data + s / 2 * vox, "flops": 2 * (_fft_flops(n, fr * m1) + _fft_flops(n, 2 * fr * m) + 2 * per_mode)}
    d = case["dirs"]
    return {"bytes": d * (s * data + s / 2 * vox), "flops": d * (_fft_flops(n, fr * m1) + _fft_flops(n, 2 * fr * m) + 2 * per_mode)}


# ---- the same outputs in plain FP64 ------------------------------------------------

def _combine(num, den, f, c0=1.0):
    guard = den < EPS_U ** 2 * f
    xi = torch.where(guard, 0.0, num / torch.where(guard, 1.0, den))
    ok = xi < c0 ** -2
    c = torch.where(ok, torch.rsqrt(torch.where(ok, c0 ** -2 - xi, 1.0)), math.nan)
    return xi, c


def _exact_reconstruct(geom, omegas, W, delta, u0=None, floor=DELTA_FLOOR):
    num = torch.zeros((geom.m, geom.n, geom.n), device="cuda", dtype=torch.float64)
    den = torch.zeros_like(num)
    for j, om in enumerate(omegas):
        K = _Modes(geom, om)
        b = torch.fft.fft2(W[j])
        dnu = TAU * max(delta, floor) * torch.linalg.vector_norm(W[j])
        bb = (b.abs() ** 2).sum(0)
        act = (bb > dnu ** 2) & ~K.graz & (K.tr > 0)
        sE = torch.where(act, (K.E.abs() ** 2).sum(0), 1.0)
        beta = (K.E.conj() * b).sum(0)
        c = beta.abs() ** 2 / sE
        p = ((b - K.E * (beta / sE)).abs() ** 2).sum(0)
        lo = ALPHA_REL * K.tr
        at_floor = (ALPHA_REL / (1 + ALPHA_REL)) ** 2 * c + p >= dnu ** 2
        t = torch.sqrt(torch.where(act & ~at_floor, (dnu ** 2 - p) / c, 0.25))
        alpha = torch.where(at_floor, lo, torch.maximum(K.tr * t / (1 - t), lo))
        V = K.P.conj() * torch.where(act, beta / torch.where(act, K.tr + alpha, 1.0), 0.0)
        u = torch.fft.ifft2(K.interior(V)) + (_plane_wave(geom, om) if u0 is None else u0[j])
        V = torch.fft.ifft2(V)
        num += (u.conj() * V).real
        den += u.abs() ** 2
    xi, c = _combine(num, den, len(omegas))
    return {"xi": xi, "c": c}


def _exact_sampled(geom, omegas, W, delta):
    m = geom.m
    num = torch.zeros((m, geom.n, geom.n), device="cuda", dtype=torch.float64)
    den = torch.zeros_like(num)
    lag = torch.tensor([[abs(i - j) for j in range(m)] for i in range(m)], device="cuda")
    for j, om in enumerate(omegas):
        A, row = _sampled_tables(geom, om)
        b = torch.fft.fft2(W[j]).movedim(0, -1)
        dnu = float(TAU * max(delta, DELTA_FLOOR) * torch.linalg.vector_norm(W[j]))
        act = (b.abs() ** 2).sum(-1) > dnu ** 2
        Aa, ba = A[act].cpu().numpy(), b[act].cpu().numpy()
        U, s, Vh = np.linalg.svd(Aa, full_matrices=False)
        beta = np.einsum("akj,ak->aj", U.conj(), ba)
        perp = np.sum(np.abs(ba - np.einsum("akj,aj->ak", U, beta)) ** 2, axis=-1)
        tr = np.sum(s * s, axis=-1)
        phi = lambda a: np.sum((a[:, None] / (s * s + a[:, None])) ** 2 * np.abs(beta) ** 2, axis=-1) + perp
        lo = ALPHA_REL * tr
        at_floor = phi(lo) >= dnu ** 2
        bn = np.linalg.norm(ba, axis=-1)
        l0, l1 = np.log(lo), np.log(np.maximum(tr * dnu / (bn - dnu), lo))
        for _ in range(120):
            mid = 0.5 * (l0 + l1)
            above = phi(np.exp(mid)) >= dnu ** 2
            l0, l1 = np.where(above, l0, mid), np.where(above, mid, l1)
        alpha = np.where(at_floor, lo, np.exp(0.5 * (l0 + l1)))
        v = np.einsum("ajl,aj->al", Vh.conj(), s / (s * s + alpha[:, None]) * beta)
        V = torch.zeros((geom.n, geom.n, m), device="cuda", dtype=torch.complex128)
        V[act] = torch.from_numpy(v).cuda()
        u = torch.fft.ifft2((row[..., lag] @ V[..., None])[..., 0].movedim(-1, 0)) + _plane_wave(geom, om)
        V = torch.fft.ifft2(V.movedim(-1, 0))
        num += (u.conj() * V).real
        den += u.abs() ** 2
    xi, c = _combine(num, den, len(omegas))
    return {"xi": xi, "c": c}


def _exact_diff(geom, omegas, W, la):
    """(xi, Phi, per frequency (modes, V~, U~, V, u)) at fixed alpha, differentiable."""
    num = den = 0.0
    phi, kept = [], []
    for j, om in enumerate(omegas):
        K = _Modes(geom, om)
        b = torch.fft.fft2(W[j])
        a = torch.exp(la[j])
        V = K.P.conj() * ((K.E.conj() * b).sum(0) / (K.tr + a))
        r = b - K.E * (K.P * V).sum(0)
        phi.append((r.real ** 2 + r.imag ** 2).sum())
        u = torch.fft.ifft2(K.interior(V)) + _plane_wave(geom, om)
        v = torch.fft.ifft2(V)
        num = num + u.real * v.real + u.imag * v.imag
        den = den + u.real ** 2 + u.imag ** 2
        kept.append((K, b, V, v, u, r))
    xi = torch.where(den < EPS_U ** 2 * len(omegas), 0.0, num / den)
    return xi, torch.stack(phi), kept


def _exact_jvp(geom, omegas, W, la, dW, dla):
    xi, _, kept = _exact_diff(geom, omegas, W, la)
    den = sum(u.abs() ** 2 for _, _, _, _, u, _ in kept)
    dxi = torch.empty((dW.shape[0],) + tuple(xi.shape), device="cuda", dtype=torch.float64)
    dphi = torch.empty((dW.shape[0], len(omegas)), device="cuda", dtype=torch.float64)
    for d in range(dW.shape[0]):
        top = torch.zeros_like(xi)
        for j, (K, b, V, v, u, r) in enumerate(kept):
            a = torch.exp(la[j])
            db = torch.fft.fft2(dW[d, j])
            dV = K.P.conj() * ((K.E.conj() * db).sum(0) / (K.tr + a)) - dla[d, j] * (a / (K.tr + a)) * V
            dr = db - K.E * (K.P * dV).sum(0)
            dphi[d, j] = 2 * (r.conj() * dr).real.sum()
            du, dv = torch.fft.ifft2(K.interior(dV)), torch.fft.ifft2(dV)
            top += (du.conj() * v + u.conj() * dv).real - 2 * xi * (u.conj() * du).real
        dxi[d] = torch.where(den < EPS_U ** 2 * len(omegas), 0.0, top / den)
    return {"dxi": dxi, "dphi": dphi}


def _exact_field(geom, om, xi):
    """The total field on X: the fixed point of Algorithm 1, iterated to rounding."""
    K, u0 = _Modes(geom, om), _plane_wave(geom, om)
    size = torch.linalg.vector_norm(u0)
    u, last = u0, math.inf
    for _ in range(400):
        new = u0 + torch.fft.ifft2(K.interior(torch.fft.fft2(xi * u)))
        step = float(torch.linalg.vector_norm(new - u) / size)
        u = new
        if step < 1e-15 or (step < 1e-13 and step >= last):
            break
        last = step
    return K, u


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        got = [_exact_reconstruct(g, om, _data(g, om, seed * 64 + j, case["delta"]).to(torch.complex64).to(torch.complex128),
                                  case["delta"]) for j, (g, om) in enumerate(_batch(case))]
        return {"xi": [r["xi"] for r in got], "c": [r["c"] for r in got]}
    geom, om = _geometry(case["n"], case["m"], case["m1"], case["layer"]), _omegas(case)
    if kind in ("reconstruct", "host"):
        u0 = _incident(case, geom, om)
        W = _data(geom, om, seed, case["delta"], u0).to(_cdt(case)).to(torch.complex128)
        if u0 is not None:
            u0 = u0.to(_cdt(case)).to(torch.complex128)
        r = _exact_reconstruct(geom, om, W, case["delta"], u0, DELTA_FLOOR if u0 is None else 1e-10)
        return {"xi": r["xi"].cpu()} if kind == "host" else r
    if kind == "sampled":
        return _exact_sampled(geom, om, _sampled_data(geom, om, seed, case["delta"]).to(_cdt(case)).to(torch.complex128),
                              case["delta"])
    if kind in ("born", "forward"):
        xi = _phantom(geom, seed, 0.05).to(_rdt(case)).double()
        W, us = [], []
        for o in om:
            K, u = (_Modes(geom, o), _plane_wave(geom, o)) if kind == "born" else _exact_field(geom, o, xi)
            W.append(torch.fft.ifft2(K.E * (K.P * torch.fft.fft2(xi * u)).sum(0)))
            us.append(u)
        return {"W": torch.stack(W)} if kind == "born" else {"W": torch.stack(W), "u": torch.stack(us)}
    _, _, W, la, want, target = _diff_inputs(case, seed)
    Wq = W.to(_cdt(case)).to(torch.complex128)
    if kind == "diff_step":
        Wq.requires_grad_(True)
        la.requires_grad_(True)
        xi, phi, _ = _exact_diff(geom, om, Wq, la)
        gW, gla = torch.autograd.grad(_loss(xi, phi, want.to(_rdt(case)).double(), target), (Wq, la))
        return {"xi": xi.detach(), "phi": phi.detach(), "gW": gW, "gla": gla}
    d, dla = _directions(case, W, seed)
    return _exact_jvp(geom, om, Wq, la, d.to(_cdt(case)).to(torch.complex128), dla)
