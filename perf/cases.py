"""Workloads of the fill-in library for timing and for comparing two builds of it.

Every case is one call (or one optimisation step) of a user's program through
the Python binding.  ``listed()`` gives the fixed cases, ``draw(rng)`` more of
the same ranges, ``prepare`` what the program has in hand before the call
(maps on the GPU and the plan it keeps), ``run`` the call itself, ``work`` the
bytes and operations the call cannot do without, ``exact`` the same outputs
from plain torch in FP64, without the library.

The grids, masks, spectra and tolerances are those of the named workloads
(64^2 plain, 1024^2 patch, the mixed-size batch, 32 band powers, 4096^2 wide
cut, the 7000 x 600 flat-sky maps) and of the GPU tests.
"""
import math

import numpy as np
import torch

import paper_1109_0286_gb300 as cg
from paper_1109_0286_gb300 import laplace

TWO_PI = 2.0 * math.pi
DTYPE = {"fp32": torch.float32, "fp64": torch.float64, "mixed": torch.float64}


# --------------------------------------------------------------------- cases

def case(kind, ny, nx, mode, **kw):
    """A case with its defaults: ``band`` (masked full-width rows, share of
    ny), ``discs`` (number of masked discs) with radii in [rmin, rmax]."""
    c = dict(kind=kind, ny=ny, nx=nx, mode=mode, batch=1, precond=True, tol=0.0, band=0.10,
             discs=max(1, round(200 * ny * nx / 2 ** 20)), rmin=2.0, rmax=12.0)
    c.update(kw)
    return c


def listed():
    return [
        # Smallest call: one application of A = P_x C^-1 P_x to a small map, as in
        # an outer iteration (a sampler, a Lanczos run) written by the user.
        case("apply", 64, 64, "fp32", name="apply_64_fp32", band=0.125, discs=5, rmin=3.0, rmax=3.0),
        # The plain method in FP64 on a small torus, converged tightly: reference runs.
        case("realize", 64, 64, "fp64", name="plain_64_fp64", tol=1e-12, band=0.125, discs=5,
             rmin=3.0, rmax=3.0, lorentz=True),
        # A 1024^2 patch with a band and point-source holes, FP32: the ordinary call.
        case("realize", 1024, 1024, "fp32", name="patch_1024_fp32", tol=1e-6),
        # The maximum-likelihood (Wiener) fill of one map in FP64, 512^2.
        case("ml", 512, 512, "fp64", name="ml_512_fp64", tol=1e-12),
        # Many small maps with masks of their own in one call: 16 x 256^2, 12 x 512^2, 4 x 1024^2.
        case("batch", 1024, 1024, "fp32", name="batch_sizes_fp32", tol=1e-6, n256=16, n512=12,
             n1024=4, batch=32),
        # One step of a band-power optimisation: new spectrum, realization, adjoint gradients
        # (refined: the gradients of an FP32 solve are good to four digits only).
        case("grad", 1024, 1024, "mixed", name="grad_1024_mixed", tol=1e-10, nbands=32),
        # Unconstrained simulations in double-float: Monte Carlo input maps.
        case("draw", 2048, 2048, "mixed", name="draw_2048x4_mixed", batch=4),
        # Ragged mixed-radix grid (ny = 375 odd, nx = 1050), FP32, three realizations.
        case("realize", 375, 1050, "fp32", name="odd_375x1050_fp32", tol=1e-6, batch=3, band=0.05),
        # The four 7000 x 600 flat-sky season maps, point sources only: plain CG to 1e-10.
        case("realize", 600, 7000, "mixed", name="flatsky_600x7000_mixed", tol=1e-10, batch=4,
             precond=False, band=0.0, discs=400, rmin=6.7, rmax=6.7),
        # Starting map of a wide cut by the multi-kernel Laplace solver: 50 sweeps, 9 annuli.
        case("laplace", 1024, 1024, "fp32", name="laplace_1024_fp32", sweeps=50, nk=9, band=0.2,
             discs=0),
        # Kernel relaxation of one map in double-float: 20 sweeps.
        case("relax", 1024, 1024, "mixed", name="relax_1024_mixed", sweeps=20),
        # The largest: eight 4096^2 realizations of a wide cut, refined to 1e-10.
        case("realize", 4096, 4096, "mixed", name="wide_4096x8_mixed", tol=1e-10, batch=8,
             band=0.20, discs=2000, rmin=2.0, rmax=20.0),
    ]


def smooth(rng, lo, hi):
    """A product of 2, 3, 5 and 7 in [lo, hi], log-uniform."""
    best, t = None, math.exp(rng.uniform(math.log(lo), math.log(hi)))
    for a in range(13):
        for b in range(8):
            for c in range(6):
                for d in range(5):
                    v = 2 ** a * 3 ** b * 5 ** c * 7 ** d
                    if lo <= v <= hi and (best is None or abs(math.log(v / t)) < abs(math.log(best / t))):
                        best = v
    return best


def grid(rng, lo, hi, odd):
    """Powers of two, or (odd) a mixed-radix grid, each side in [lo, hi]."""
    if odd:
        return smooth(rng, lo, hi), 2 * smooth(rng, lo // 2, hi // 2)
    a, b = round(math.log2(lo)), round(math.log2(hi))
    ny = rng.randint(a, b)
    return 2 ** ny, 2 ** min(b, max(a, ny + rng.choice((-1, 0, 0, 1))))


def draw(rng):
    kind = rng.choice(("realize", "realize", "realize", "ml", "batch", "grad", "draw", "apply",
                       "laplace", "relax"))
    mode = rng.choice(("fp32", "fp32", "mixed", "fp64"))
    tol = {"fp32": 1e-6, "mixed": 1e-10, "fp64": 1e-12}[mode]
    odd = rng.random() < 0.4
    hi = {"fp32": 2048, "mixed": 2048, "fp64": 512}[mode]
    ny, nx = grid(rng, 48 if odd else 64, hi, odd)
    mask = dict(band=round(rng.uniform(0.05, 0.2), 3), rmin=2.0,
                rmax=round(rng.uniform(3.0, 12.0), 2),
                discs=max(1, int(rng.uniform(50, 400) * ny * nx / 2 ** 20)))
    if kind == "batch":
        return case("batch", 1024, 1024, "fp32", tol=1e-6, n256=rng.randint(2, 24),
                    n512=rng.randint(1, 12), n1024=rng.randint(0, 4),
                    batch=0) | {"rmax": mask["rmax"]}
    if kind == "grad":
        ny = nx = min(1024, max(128, nx))
        if odd:
            ny = nx = 2 * smooth(rng, 64, 500)
        return case("grad", ny, nx, "mixed", tol=1e-10, nbands=rng.choice((8, 16, 32)), **mask)
    if kind == "draw":
        return case("draw", ny, nx, mode, batch=rng.choice((1, 2, 4)), **mask)
    if kind == "apply":
        return case("apply", ny, nx, mode, **mask)
    if kind == "laplace":
        ny, nx = max(ny, 256), max(nx, 256)
        nk = 6 if min(ny, nx) < 512 else 8
        return case("laplace", ny, nx, mode, sweeps=rng.randint(10, 50), nk=nk, **(mask | {"discs": 0}))
    if kind == "relax":
        return case("relax", ny, nx, mode, sweeps=rng.randint(5, 40), **mask)
    if kind == "ml":
        return case("ml", ny, nx, mode, tol=tol, **mask)
    point = rng.random() < 0.3   # point sources only: plain CG
    if point:
        mask["band"] = 0.0
    return case("realize", ny, nx, mode, tol=tol, batch=rng.choice((1, 1, 2, 4)),
                precond=not point, **mask)


# -------------------------------------------------------------------- inputs

def kgrid(ny, nx, dev):
    ky = TWO_PI * torch.fft.fftfreq(ny, dtype=torch.float64, device=dev)
    kx = TWO_PI * torch.arange(nx // 2 + 1, dtype=torch.float64, device=dev) / nx
    return torch.sqrt(ky[:, None] ** 2 + kx[None, :] ** 2)


def cmb_signal(k, k_lo, sb=2.0):
    """Red below 2 pi / 200, flat above, damped at 2 pi / 24, beam sb."""
    k_peak, k_d = TWO_PI / 200.0, TWO_PI / 24.0
    kk = torch.clamp(k, min=k_lo)
    red = torch.where(kk < k_peak, (k_peak / kk) ** 2, torch.ones_like(kk))
    return red * torch.exp(-(k / k_d) ** 2) * torch.exp(-(k * sb) ** 2)


def cmb_noise(sb=2.0):
    k_d = TWO_PI / 24.0
    return 1e-3 * math.exp(-1.0) * math.exp(-(k_d * sb) ** 2)


def k_low(c, ny, nx):
    return TWO_PI / min(4096, max(ny, nx))


def spectrum(c, ny, nx, dev):
    """P(k) on the half plane (FP64, GPU)."""
    k = kgrid(ny, nx, dev)
    if c.get("lorentz"):
        k0, sb = TWO_PI / 32.0, 1.5
        return torch.exp(-(k * sb) ** 2) / (k * k + k0 * k0) + \
            1e-4 * math.exp(-(k0 * sb) ** 2) / (2.0 * k0 * k0)
    return cmb_signal(k, k_low(c, ny, nx)) + cmb_noise()


def observed_map(ny, nx, band_rows, discs, rmin, rmax, g, dev):
    """uint8 map (1 = observed): a band of rows plus discs at random centres."""
    masked = torch.zeros((ny, nx), dtype=torch.bool, device=dev)
    if band_rows > 0:
        r0 = ny // 2 - band_rows // 2
        masked[r0:r0 + band_rows] = True
    if discs > 0:
        u = torch.rand((discs, 3), generator=g, dtype=torch.float64).to(dev)
        cy, cx, r = u[:, 0] * ny, u[:, 1] * nx, rmin + (rmax - rmin) * u[:, 2]
        R = int(math.ceil(rmax)) + 1
        o = torch.arange(-R, R + 1, device=dev)
        iy = torch.floor(cy).long()[:, None, None] + o[None, :, None]
        ix = torch.floor(cx).long()[:, None, None] + o[None, None, :]
        inside = (iy - cy[:, None, None]) ** 2 + (ix - cx[:, None, None]) ** 2 <= r[:, None, None] ** 2
        iy, ix = torch.broadcast_tensors(iy % ny, ix % nx)
        masked[iy[inside], ix[inside]] = True
    if band_rows == 0 and discs == 0:
        masked[ny // 2, nx // 2] = True
    return (~masked).to(torch.uint8)


def field(P, ny, nx, g, dev):
    """A Gaussian map with spectrum P (the sky the user observed)."""
    xi = torch.randn((ny, nx), generator=g, dtype=torch.float64, device=dev)
    return torch.fft.irfft2(torch.fft.rfft2(xi) * torch.sqrt(P), s=(ny, nx))


def band_index(ny, nx, k_lo, nbands, dev):
    edges = torch.from_numpy(np.geomspace(k_lo, math.pi * math.sqrt(2.0), nbands + 1)).to(dev)
    b = torch.searchsorted(edges, kgrid(ny, nx, dev).reshape(-1), right=True) - 1
    return b.clamp(0, nbands - 1).to(torch.int32).reshape(ny, nx // 2 + 1)


def seeds_of(seed, n):
    return [(seed * 1000003 + 17 * i + 1) % (1 << 62) for i in range(n)]


def parts(c, seed):
    """(spectrum, observed map, data map) of each plan of the case, on the GPU."""
    dev = torch.device("cuda")
    gh = torch.Generator().manual_seed(seed)
    gd = torch.Generator(device=dev).manual_seed(seed + 1)
    if c["kind"] != "batch":
        ny, nx = c["ny"], c["nx"]
        P = spectrum(c, ny, nx, dev)
        obs = observed_map(ny, nx, round(c["band"] * ny), c["discs"], c["rmin"], c["rmax"], gh, dev)
        d = field(P, ny, nx, gd, dev).to(DTYPE[c["mode"]])
        return [(P, obs, d)]
    out = []
    for n, count in ((256, c["n256"]), (512, c["n512"]), (1024, c["n1024"])):
        P = spectrum(c, n, n, dev)
        for _ in range(count):
            a = 0.05 + 0.20 * torch.rand((), generator=gh, dtype=torch.float64).item()
            r2 = (c["rmin"] ** 2 + c["rmin"] * c["rmax"] + c["rmax"] ** 2) / 3.0
            discs = max(1, round(0.3 * a * n * n / (math.pi * r2)))
            obs = observed_map(n, n, round(0.7 * a * n), discs, c["rmin"], c["rmax"], gh, dev)
            out.append((P, obs, field(P, n, n, gd, dev).to(DTYPE[c["mode"]])))
    return out


def prepare(c, seed):
    ps = parts(c, seed)
    dev = ps[0][0].device
    kind, st = c["kind"], {"case": c}
    host = {}
    for P, _, _ in ps:
        if id(P) not in host:
            host[id(P)] = P.cpu().numpy()
    if kind == "batch":
        st["plans"] = [cg.Plan(host[id(P)], o.cpu().numpy(), mode=c["mode"]) for P, o, _ in ps]
        st["ds"] = [d for _, _, d in ps]
        st["seeds"] = seeds_of(seed, len(ps))
        return st
    P, obs, d = ps[0]
    Ph, oh = host[id(P)], obs.cpu().numpy()
    plan = cg.Plan(Ph, oh, mode=c["mode"], precond=c["precond"], batch=c["batch"],
                   backward=kind == "grad")
    st.update(plan=plan, d=d, seeds=seeds_of(seed, c["batch"]))
    if kind == "grad":
        ny, nx = c["ny"], c["nx"]
        k_lo = k_low(c, ny, nx)
        plan.set_bands(band_index(ny, nx, k_lo, c["nbands"], dev).cpu().numpy(),
                       cmb_signal(kgrid(ny, nx, dev), k_lo).cpu().numpy())
        st.update(P=Ph, masked=(obs == 0).to(d.dtype))
    if kind == "laplace":
        radii = laplace.ms_radii(c["nk"])
        plan.set_annuli([r[0] for r in radii], [r[1] for r in radii])
        st["cls"] = laplace.ms_classes(obs, radii)
    return st


def run(st):
    c = st["case"]
    kind, tol = c["kind"], c["tol"]
    if kind == "batch":
        return cg.realize_batch(st["plans"], st["ds"], st["seeds"], tol)[0]
    plan, d = st["plan"], st["d"]
    if kind == "realize":
        return plan.realize(d, st["seeds"], tol)[0]
    if kind == "ml":
        return plan.ml(d, tol)[0]
    if kind == "draw":
        return plan.draw(st["seeds"])
    if kind == "apply":
        return plan.apply(2, d)
    if kind == "laplace":
        return plan.laplace_ms(d, c["sweeps"], st["cls"])[0]
    if kind == "relax":
        return plan.relax(d, c["sweeps"])[0]
    # loss = sum of the squared filled pixels; the step ends with dL/dd and dL/da_b
    plan.set_spectrum(st["P"])
    x, _ = plan.realize(d, st["seeds"], tol)
    gd, gb, _ = plan.backward(d, 2.0 * x * st["masked"], tol)
    return x, gd, torch.from_numpy(gb).to(d.dtype)


def work(c):
    """One pass: per operator application two real 2D transforms (2.5 n log2 n
    operations each), one read and one write of the map and one read of the
    table; the solves take their usual number of CG iterations (three
    applications with the preconditioner, else one, and five vectors on the
    masked pixels)."""
    size = 4 if c["mode"] == "fp32" else 8

    def one(n, apps, maps, its=0, masked=0.0, elem=4):
        flops = apps * 5.0 * n * math.log2(n)
        nbytes = apps * n * 2.5 * elem + maps * n * size + its * 5 * masked * n * elem
        return nbytes, flops

    def solve(n, batch=1):
        its = {1e-6: 90, 1e-10: 170, 1e-12: 150}.get(c["tol"], 100)
        its = its * (2.5 if n > 2 ** 23 and c["precond"] else 1.0) * (0.6 if not c["precond"] else 1.0)
        m = c["band"] + c["discs"] * math.pi * (c["rmin"] ** 2 + c["rmax"] ** 2) / 2 / (c["ny"] * c["nx"])
        b, f = one(n, its * (3 if c["precond"] else 1), 2, its, min(0.3, m), 8 if c["mode"] == "fp64" else 4)
        return b * batch, f * batch

    n, kind = c["ny"] * c["nx"], c["kind"]
    if kind == "batch":
        w = [solve(s * s, k) for s, k in ((256, c["n256"]), (512, c["n512"]), (1024, c["n1024"])) if k]
        b, f = sum(x[0] for x in w), sum(x[1] for x in w)
    elif kind in ("realize", "ml"):
        b, f = solve(n, c["batch"])
    elif kind == "grad":
        b, f = solve(n)
        b, f = 2 * b + 6 * n * size, 2 * f + 10.0 * n * math.log2(n)
    elif kind == "draw":
        b, f = one(n, 1, 0)
        b, f = c["batch"] * n * (size + 4), c["batch"] * f
    elif kind == "apply":
        b, f = one(n, 1, 0, elem=size)
    elif kind == "relax":
        b, f = one(n, c["sweeps"], 2, elem=size)
    else:
        b, f = one(n, c["sweeps"] * (1 + c["nk"]) / 2.0, 2, elem=size)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------- FP64 reference values

def philox(ctr, seed):
    """Philox4x32-10 words of the counters (j, 0, 0, 0) under the 64-bit key."""
    m = np.uint64(0xFFFFFFFF)
    c = [ctr.astype(np.uint64), *(np.zeros(ctr.shape, np.uint64) for _ in range(3))]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m]
    return c


def noise(ny, nx, seed, dev):
    """Unit white noise of the seed: Box-Muller on 52-bit uniforms."""
    w = philox(np.arange(ny * nx // 2, dtype=np.uint64), seed)
    six, s26 = np.uint64(6), 67108864.0
    u1 = ((w[0] >> six).astype(np.float64) * s26 + (w[1] >> six).astype(np.float64) + 0.5) * 2.0 ** -52
    u2 = ((w[2] >> six).astype(np.float64) * s26 + (w[3] >> six).astype(np.float64) + 0.5) * 2.0 ** -52
    rad = np.sqrt(-2.0 * np.log(u1))
    xi = np.stack((rad * np.cos(TWO_PI * u2), rad * np.sin(TWO_PI * u2)), axis=1)
    return torch.from_numpy(xi.reshape(ny, nx)).to(dev)


def mul(v, table, ny, nx):
    return torch.fft.irfft2(torch.fft.rfft2(v) * table, s=(ny, nx))


def pcg(A, B, b, tol):
    """A u = b; a second, short solve takes out what the recurrence lost."""
    u = torch.zeros_like(b)
    bb = torch.sum(b * b).item()
    for stop in (tol, 1e-15):
        r = b - A(u)
        if torch.sum(r * r).item() <= stop * stop * bb:
            break
        p, rho = torch.zeros_like(b), None
        for it in range(3000 if stop == tol else 60):
            z = B(r) if B else r
            new = torch.sum(r * z).item()
            if new <= 0.0:
                break
            p = z + (new / rho if rho else 0.0) * p
            rho = new
            q = A(p)
            a = rho / torch.sum(p * q).item()
            u = u + a * p
            r = r - a * q
            if torch.sum(r * r).item() <= stop * stop * bb:
                break
    return u


def solve_exact(c, P, obs, d, seed):
    """(x, y, u, A, B) of one realization (seed None: the ML fill)."""
    ny, nx = obs.shape
    M = (obs == 0).to(torch.float64)
    d = d.to(torch.float64)
    sq, inv = torch.sqrt(P), 1.0 / P
    A = lambda v: M * mul(M * v, inv, ny, nx)                          # noqa: E731
    S = lambda v: M * mul(M * v, sq, ny, nx)                           # noqa: E731
    B = (lambda v: S(S(v))) if c["precond"] else None                  # noqa: E731
    y = torch.zeros_like(d) if seed is None else mul(noise(ny, nx, seed, d.device), sq, ny, nx)
    b = -M * mul((1.0 - M) * (d - y), inv, ny, nx)
    u = pcg(A, B, b, 1e-14)
    return torch.where(obs == 0, y + u, d), y, u, A, B


def exact(c, seed):
    kind, ny, nx = c["kind"], c["ny"], c["nx"]
    if kind in ("realize", "ml") and c["batch"] * ny * nx > 3 * 2 ** 23:
        return None   # the FP64 solves take minutes
    ps = parts(c, seed)
    if kind == "batch":
        return [solve_exact(c, P, o, d, s)[0][None] for (P, o, d), s in zip(ps, seeds_of(seed, len(ps)))]
    P, obs, d = ps[0]
    dev, seeds = d.device, seeds_of(seed, c["batch"])
    n = ny * nx
    d64 = d.to(torch.float64)
    obs_b = obs != 0
    if kind == "realize":
        return torch.stack([solve_exact(c, P, obs, d, s)[0] for s in seeds])
    if kind == "ml":
        return solve_exact(c, P, obs, d, None)[0][None]
    if kind == "draw":
        return torch.stack([mul(noise(ny, nx, s, dev), torch.sqrt(P), ny, nx) for s in seeds])
    if kind == "apply":
        M = (~obs_b).to(torch.float64)
        return M * mul(M * d64, 1.0 / P, ny, nx)
    if kind == "relax":
        a = torch.max(1.0 / P)
        x = torch.where(obs_b, d64, torch.zeros_like(d64))
        for _ in range(c["sweeps"]):
            x = torch.where(obs_b, x, x - mul(x, 1.0 / P, ny, nx) / a)
        return x[None]
    if kind == "laplace":
        dy = torch.fft.fftfreq(ny, 1.0 / ny, dtype=torch.float64, device=dev)
        dx = torch.fft.fftfreq(nx, 1.0 / nx, dtype=torch.float64, device=dev)
        r2 = dy[:, None] ** 2 + dx[None, :] ** 2
        gap = torch.fft.rfft2(obs_b.to(torch.float64))
        cls = torch.zeros((ny, nx), dtype=torch.long, device=dev)
        kernels = []
        for j in range(c["nk"]):
            rho, q = 1.5 * 1.55 ** j, math.sqrt(1.55)
            lo, hi = (0.0 if j == 0 else rho / q), rho * q
            ring = ((r2 > lo * lo) & (r2 <= hi * hi) & (r2 > 0)).to(torch.float64)
            kernels.append(torch.fft.rfft2(ring / ring.sum()))
            disc = torch.fft.rfft2((r2 <= hi * hi).to(torch.float64))
            cls[torch.fft.irfft2(gap * disc, s=(ny, nx)) < 0.5] = j
        x = torch.where(obs_b, d64, torch.zeros_like(d64))
        for _ in range(c["sweeps"]):
            X, new = torch.fft.rfft2(x), x.clone()
            for j, K in enumerate(kernels):
                sel = ~obs_b & (cls == j)
                new[sel] = torch.fft.irfft2(X * K, s=(ny, nx))[sel]
            x = new
        return x[None]
    # grad: adjoint gradients of sum(x_M^2) by one more solve with A
    x, y, u, A, B = solve_exact(c, P, obs, d, seeds[0])
    g = 2.0 * torch.where(obs_b, torch.zeros_like(x), x)
    lam = pcg(A, B, g, 1e-14)
    Ql = mul(lam, 1.0 / P, ny, nx)
    gd = torch.where(obs_b, -Ql, torch.zeros_like(Ql))
    h = torch.where(obs_b, Ql, g)
    w = torch.where(obs_b, d64 - y, u)
    F = torch.fft.rfft2
    dot = lambda a, b: (F(a).conj() * F(b)).real                        # noqa: E731
    dP = dot(h, noise(ny, nx, seeds[0], dev)) / (2.0 * n * torch.sqrt(P)) + dot(lam, w) / (n * P ** 2)
    wt = torch.full((nx // 2 + 1,), 2.0, dtype=torch.float64, device=dev)
    wt[0] = wt[-1] = 1.0
    k_lo = k_low(c, ny, nx)
    S = cmb_signal(kgrid(ny, nx, dev), k_lo)
    bands = band_index(ny, nx, k_lo, c["nbands"], dev).long().reshape(-1)
    gb = torch.zeros(c["nbands"], dtype=torch.float64, device=dev)
    gb.index_add_(0, bands, (wt[None, :] * S * dP).reshape(-1))
    return x[None], gd[None], gb[None]
