"""Measured cases: the calls that a program built on this framework makes.

Kinds of case ("kind"):
  mvm      y = x - G(chi x) on the full grid (Grid.matvec): every outer iteration makes two of them, in
           complex64 (mixed mode) or complex128 (plain mode, FP64 residuals).
  precond  y = K2^{-1} b (Grid.precond): the block-diagonal preconditioner, 96 % of a metasurface solve.
  request  one wavelength of a sweep over a served structure: Green spectrum, incident wave, mixed solve,
           bistatic RCS, spectrum released (the whole call chain of a solve request).
  batch    many small scatterers of one grid shape solved together (Batch.solve).

Block solves and system solves are run to tolerances at which the vector returned is fixed by the inputs
(an iterate stopped at 1e-2 is not: two summation orders give vectors that differ by 1e-2). The work of an
iteration is the same at every tolerance; the inner solves inside "request" keep the usual 1e-2.
"""
import math

import numpy as np
import torch

from paper_2501_13512_gb300 import inputs, vie

C64, C128 = "c64", "c128"
_DT = {C64: torch.complex64, C128: torch.complex128}
_VP = {C64: vie.C64, C128: vie.C128}


def listed():
    return [
        # the validation sphere's grid: the smallest product, launches and latency
        {"name": "mvm_c64_16x16x16", "kind": "mvm", "nx": 16, "ny": 16, "nz": 16, "prec": C64},
        # the metasurface grid of the benchmark, the product of its mixed outer iterations
        {"name": "mvm_c64_256x256x16", "kind": "mvm", "nx": 256, "ny": 256, "nz": 16, "prec": C64},
        # the largest served box (a tile in a cubic computational box)
        {"name": "mvm_c64_128x128x128", "kind": "mvm", "nx": 128, "ny": 128, "nz": 128, "prec": C64},
        # odd extents, as a scatterer's own bounding box gives them: no axis near its padded length
        {"name": "mvm_c64_100x37x60", "kind": "mvm", "nx": 100, "ny": 37, "nz": 60, "prec": C64},
        # FP64 residual of the metasurface, and the product of its plain complex128 solve
        {"name": "mvm_c128_256x256x16", "kind": "mvm", "nx": 256, "ny": 256, "nz": 16, "prec": C128},
        # FP64 residual of a medium cubic box
        {"name": "mvm_c128_64x64x64", "kind": "mvm", "nx": 64, "ny": 64, "nz": 64, "prec": C128},
        # the benchmark's preconditioner: 256 uneven pillar blocks
        {"name": "precond_c64_256_pillars", "kind": "precond", "cells": 16, "nz": 16, "block_cells": 0, "vpw": 20,
         "tol": 1e-6, "prec": C64},
        # a 64-voxel tile's preconditioner: 16 pillar blocks, too few to fill the GPU with one block per cluster
        {"name": "precond_c64_16_pillars", "kind": "precond", "cells": 4, "nz": 16, "block_cells": 0, "vpw": 20,
         "tol": 1e-6, "prec": C64},
        # coarser block division (2 x 2 unit cells with their air per block): larger boxes, more iterations
        {"name": "precond_c64_16_coarse", "kind": "precond", "cells": 8, "nz": 16, "block_cells": 2, "vpw": 40,
         "tol": 1e-6, "prec": C64},
        # the preconditioner of a plain complex128 solve
        {"name": "precond_c128_64_pillars", "kind": "precond", "cells": 8, "nz": 16, "block_cells": 0, "vpw": 20,
         "tol": 1e-11, "prec": C128},
        # one wavelength of a served 64-voxel metasurface tile (h = 10 nm)
        {"name": "request_64", "kind": "request", "n": 64, "lam": 600, "deg": 15.0, "ndir": 61, "tol": 1e-12},
        # dielectric particles solved together
        {"name": "batch_8x24", "kind": "batch", "n": 24, "count": 8, "tol": 1e-12},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("mvm", "mvm", "mvm", "precond", "precond", "request", "batch"))
    if kind == "mvm":
        prec = rng.choice((C64, C64, C128))
        most = 1 << 21 if prec == C64 else 1 << 20
        while True:
            nx, ny, nz = (_logint(rng, 4, 256) for _ in range(3))
            if nx * ny * nz <= most:
                return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "prec": prec}
    if kind == "precond":
        prec = rng.choice((C64, C64, C64, C128))
        block_cells = rng.choice((0, 0, 0, 2)) if prec == C64 else 0
        cells = _logint(rng, 2, 16 if prec == C64 and not block_cells else 8)
        return {"kind": kind, "cells": cells, "nz": rng.randint(6, 16), "block_cells": block_cells,
                "vpw": 40 if block_cells else rng.randint(20, 40), "tol": 1e-6 if prec == C64 else 1e-11, "prec": prec}
    if kind == "request":
        return {"kind": kind, "n": 16 * rng.randint(2, 6), "lam": 10 * rng.randint(40, 80), "deg": round(rng.uniform(0, 30), 2),
                "ndir": rng.randint(19, 181), "tol": 1e-12}
    n = _logint(rng, 8, 24)
    return {"kind": kind, "n": n, "count": rng.randint(2, 8 if n > 16 else 24), "tol": 1e-12}


# ---------------------------------------------------------------- inputs
def _randn(shape, seed, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _medium(case, seed):
    """A lossy dielectric of smooth random permittivity 1 .. 4 with 20 % air, and a field of unit size."""
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    u = torch.rand((2, nz, ny, nx), generator=g, device="cuda", dtype=torch.float64)
    air = torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64) < 0.2
    eps = torch.complex(1 + 3 * u[0], -0.3 * u[1])
    eps[air] = 1.0
    return eps.cpu().numpy(), _randn((3, nz, ny, nx), seed + 1, _DT[case["prec"]])


def _pillars(case, seed):
    w = inputs.metasurface(cells=case["cells"], period=16, nz=case["nz"], seed=int(seed), voxels_per_wl=case["vpw"],
                           block_cells=case["block_cells"])
    return w, _randn((3,) + w.eps_r.shape, seed + 1, _DT[case["prec"]])


def _tile(case, seed):
    w = inputs.serving_geometry("metasurface", case["n"], int(seed))
    th = math.radians(case["deg"])
    d = np.linspace(0.0, math.pi, case["ndir"])
    return {"w": w, "h": 10.0, "k0": 2 * math.pi / case["lam"], "khat": np.array([math.sin(th), 0.0, math.cos(th)]),
            "pol": np.array([math.cos(th), 0.0, -math.sin(th)], complex),
            "dirs": np.stack([np.sin(d), 0 * d, np.cos(d)], 1)}


def _particles(case, seed):
    """Level-set particles of permittivity 1.5 .. 4.5, each with its own incident plane wave, h = lambda / 20."""
    ws = [inputs.blob(case["n"], seed=int(seed) * 1000 + i) for i in range(case["count"])]
    eps = [1.0 + 0.5 * (w.eps_r - 1.0) for w in ws]
    r = np.stack(inputs.voxel_centres(ws[0].n, ws[0].h))
    einc = torch.stack([torch.from_numpy(w.pol[:, None, None, None] * np.exp(-1j * w.k0 * np.tensordot(w.khat, r, 1)))
                        for w in ws])
    return eps, ws[0].h, [w.k0 for w in ws], einc.cuda()


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "mvm":
        eps, s["x"] = _medium(case, seed)
        s["grid"] = vie.Grid(eps, 0.05)
        s["spec"] = s["grid"].spectrum(2 * math.pi, precision=_VP[case["prec"]])
        s["y"] = torch.empty_like(s["x"])
    elif case["kind"] == "precond":
        w, s["b"] = _pillars(case, seed)
        s["grid"] = vie.Grid.from_workload(w)
        s["spec"] = s["grid"].spectrum(w.k0)
        s["y"] = torch.empty_like(s["b"])
    elif case["kind"] == "request":
        t = _tile(case, seed)
        s.update(t)
        s["grid"] = vie.Grid(t["w"].eps_r, t["h"], t["w"].block_id)
    else:
        eps, h, s["k0s"], s["einc"] = _particles(case, seed)
        s["batch"] = vie.Batch(eps, h)
        s["e"] = s["batch"].empty()
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "mvm":
        return s["grid"].matvec(s["spec"], s["x"], s["y"])
    if case["kind"] == "precond":
        return s["grid"].precond(s["spec"], s["b"], s["y"], inner_tol=case["tol"], inner_maxit=1000)[0]
    if case["kind"] == "request":
        g, k0 = s["grid"], s["k0"]
        spec = g.spectrum(k0)
        einc = g.plane_wave(k0, s["khat"], s["pol"])
        e, st = g.solve(spec, einc, outer_tol=case["tol"], inner_tol=1e-2, mode=vie.MODE_MIXED)
        rcs = g.far_field_rcs(k0, e, s["dirs"])
        spec.release()
        return {"e": e, "rcs": rcs}
    return s["batch"].solve(s["k0s"], s["einc"], s["e"], outer_tol=case["tol"], outer_maxit=4000)[0]


# ---------------------------------------------------------------- necessary work
def _mvm_work(nx, ny, nz, size):
    """Bytes and operations of one product: x, chi and one octant of the kernel in, y out; pruned transforms
    of the doubled axes (5 L log2 L each) forward and back, and the symmetric 3 x 3 multiply per frequency."""
    n = nx * ny * nz
    fft = lambda m: 5.0 * m * math.log2(m) if m > 1 else 0.0  # noqa: E731
    one = 3 * (ny * nz * fft(2 * nx) + 2 * nx * nz * fft(2 * ny) + 4 * nx * ny * fft(2 * nz))
    return (3 + 1 + 6 + 3) * n * size, 2 * one + 66.0 * 8 * n


def work(case):
    size = 16 if case.get("prec") == C128 else 8
    if case["kind"] == "mvm":
        b, f = _mvm_work(case["nx"], case["ny"], case["nz"], size)
        return {"bytes": b, "flops": f}
    if case["kind"] == "precond":
        # mean inner iterations measured per decade of tolerance: about 19 (pillars), 9 (2 x 2 cells at the finer mesh), 14 in
        # complex128; an average pillar's box is 9 x 9 voxels wide
        side = 16 * case["block_cells"] if case["block_cells"] else 9
        nb = math.ceil(case["cells"] / max(1, case["block_cells"])) ** 2
        its = -math.log10(case["tol"]) * (9 if case["block_cells"] else 19 if case["prec"] == C64 else 14)
        _, f = _mvm_work(side, side, case["nz"], size)
        n = (16 * case["cells"]) ** 2 * case["nz"]
        return {"bytes": 2 * 3 * n * size + nb * side * side * case["nz"] * size, "flops": nb * its * 2 * f}
    if case["kind"] == "request":
        n = case["n"]
        b, f = _mvm_work(n, n, n, 8)
        _, fb = _mvm_work(9, 9, 16, 8)
        outer = 12.0        # mixed outer iterations to the tolerance
        return {"bytes": 2 * outer * b + 2 * 48 * n**3, "flops": 2 * outer * (f + (n // 16) ** 2 * 8 * 2 * fb)}
    b, f = _mvm_work(case["n"], case["n"], case["n"], 8)
    return {"bytes": 2 * 48 * case["count"] * case["n"] ** 3, "flops": case["count"] * 60.0 * 2 * f}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch
def _kernel(nx, ny, nz, h, k0):
    """FFT over the doubled axes of k0^2 G(D h) h^3 with the equivalent-sphere self term, [6][2nz][2ny][2nx]."""
    ax = []
    for n in (nx, ny, nz):
        i = torch.arange(2 * n, device="cuda", dtype=torch.float64)
        ax.append(torch.where(i < n, i, i - 2 * n) * h)
    z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    r2 = x * x + y * y + z * z
    r2[0, 0, 0] = 1.0
    r = torch.sqrt(r2)
    g = torch.polar(0.25 / math.pi / r * h**3, -k0 * r)
    a = g * torch.complex(k0 * k0 - 1 / r2, -k0 / r)
    b = g * torch.complex(3 / r2 - k0 * k0, 3 * k0 / r) / r2
    ka = k0 * h * (3 / (4 * math.pi)) ** (1 / 3)
    self_term = 2 / 3 * ((1 + 1j * ka) * complex(math.cos(ka), -math.sin(ka)) - 1) - 1 / 3
    out = torch.empty((6,) + tuple(r.shape), dtype=torch.complex128, device="cuda")
    for c, (p, q, diag) in enumerate(((x, x, 1), (x, y, 0), (x, z, 0), (y, y, 1), (y, z, 0), (z, z, 1))):
        k = b * (p * q) + (a if diag else 0)
        k[0, 0, 0] = self_term if diag else 0.0
        # offset -n is in no product of two voxels of the box
        k[nz], k[:, ny], k[:, :, nx] = 0, 0, 0
        out[c] = torch.fft.fftn(k)
    return out


def _apply(kf, chi, x):
    """x - G(chi x) for x [..., 3, nz, ny, nx]."""
    nz, ny, nx = x.shape[-3:]
    f = torch.fft.fftn(chi.unsqueeze(-4) * x, s=tuple(kf.shape[-3:]), dim=(-3, -2, -1))
    fx, fy, fz = f.unbind(-4)
    u = torch.stack((kf[0] * fx + kf[1] * fy + kf[2] * fz, kf[1] * fx + kf[3] * fy + kf[4] * fz,
                     kf[2] * fx + kf[4] * fy + kf[5] * fz), -4)
    return x - torch.fft.ifftn(u, dim=(-3, -2, -1))[..., :nz, :ny, :nx]


def _bicgstab(op, b, tol, maxit):
    """Independent systems along the first axis, each to ||r|| <= tol ||b||."""
    dot = lambda u, v: (u.conj() * v).flatten(1).sum(1)  # noqa: E731
    ex = lambda s: s.view((-1,) + (1,) * (b.dim() - 1))  # noqa: E731
    x, r = torch.zeros_like(b), b.clone()
    rh, p, v = r.clone(), torch.zeros_like(b), torch.zeros_like(b)
    one = torch.ones(b.shape[0], dtype=b.dtype, device=b.device)
    rho, alpha, omega = one, one, one
    bn = dot(b, b).real
    live = bn > 0
    for it in range(maxit):
        new = dot(rh, r)
        beta = torch.where(live, new / rho * (alpha / omega), 0)
        p = torch.where(ex(live), r + ex(beta) * (p - ex(omega) * v), p)
        v = torch.where(ex(live), op(p), v)
        alpha = torch.where(live, new / dot(rh, v), alpha)
        s = r - ex(alpha) * v
        t = op(s)
        tt = dot(t, t)
        omega = torch.where(live & (tt.real > 0), dot(t, s) / tt, omega)
        x = torch.where(ex(live), x + ex(alpha) * p + ex(omega) * s, x)
        r = torch.where(ex(live), s - ex(omega) * t, r)
        rho = new
        live = live & (dot(r, r).real > tol * tol * bn)
        if it % 10 == 9 and not bool(live.any()):
            break
    return x


def exact(case, seed):
    if case["kind"] == "mvm":
        eps, x = _medium(case, seed)
        kf = _kernel(case["nx"], case["ny"], case["nz"], 0.05, 2 * math.pi)
        return _apply(kf, torch.from_numpy(eps).cuda() - 1.0, x.to(torch.complex128))
    if case["kind"] == "request":
        t = _tile(case, seed)
        w, n = t["w"], case["n"]
        chi = torch.from_numpy(w.eps_r).cuda() - 1.0
        r = torch.from_numpy(np.stack(inputs.voxel_centres((n, n, n), t["h"]))).cuda()
        einc = torch.from_numpy(t["pol"]).cuda().view(3, 1, 1, 1) * torch.exp(
            -1j * t["k0"] * torch.tensordot(torch.from_numpy(t["khat"]).cuda(), r, 1))
        kf = _kernel(n, n, n, t["h"], t["k0"])
        e = _bicgstab(lambda v: _apply(kf, chi, v), einc.unsqueeze(0), 1e-13, 400)[0]
        u = torch.from_numpy(t["dirs"]).cuda()
        j = (chi * e).reshape(3, -1)
        p = torch.stack([j @ torch.exp(1j * t["k0"] * (d @ r.reshape(3, -1))) for d in u]) * t["h"] ** 3
        p = p - u * (u * p).sum(1, keepdim=True)
        return {"e": e, "rcs": (t["k0"] ** 4 / (4 * math.pi) * p.abs().square().sum(1)).cpu().numpy()}
    if case["kind"] == "batch":
        eps, h, k0s, einc = _particles(case, seed)
        n = case["n"]
        chi = torch.from_numpy(np.stack(eps)).cuda() - 1.0
        kf = _kernel(n, n, n, h, k0s[0])
        return _bicgstab(lambda v: _apply(kf, chi, v), einc, 1e-13, 1500)
    # a block solve in complex64 stops at an iterate within its tolerance: no value of its own in 64 bits
    if case["prec"] == C64:
        return None
    w, b = _pillars(case, seed)
    nb, nz = case["cells"], case["nz"]
    bid = torch.from_numpy(w.block_id).cuda()
    # every pillar in its 16 x 16 unit cell: the operator of the cell, restricted to the pillar's voxels
    cut = lambda v: v.unflatten(-1, (nb, 16)).unflatten(-3, (nb, 16)).movedim((-4, -2), (0, 1)).flatten(0, 1)  # noqa: E731
    chi = cut(torch.from_numpy(w.eps_r).cuda() - 1.0)
    m = (cut(bid) >= 0).unsqueeze(1)
    kf = _kernel(16, 16, nz, w.h, w.k0)
    y = _bicgstab(lambda v: _apply(kf, chi, v) * m, cut(b) * m, 1e-13, 1000)
    y = y.unflatten(0, (nb, nb)).movedim((0, 1), (-4, -2)).reshape(b.shape)
    return torch.where((bid >= 0).unsqueeze(0), y, b)
