"""Workloads of this library, from the smallest system to the paper-scale one, for timing and for
comparing results: the stochastic action of W on pair densities, the exciton matrix and its lowest
eigenvalues, the Chebyshev absorption spectra, and inference and gradients of the learned
surrogate.

A case is a dict of plain values. `prepare` makes what a program holds before the call (context with
grid and orbitals, the pinned result buffer, for the spectra also A or W), `run` makes one pass
through the public entry points, `work` gives the bytes and operations the path cannot do without,
and `exact` evaluates the same quantities in 64 bits with plain torch. Results of the mixed mode,
which are FP32 sums carried in FP64 arrays, are returned as FP32 (as surrogate.training_pairs does
with W); results of the FP64 mode are returned as they are.
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_2205_06690_gb300 import binding as B

DT, GAMMA, ALPHA, SCISSOR = 0.05, 0.1, 1e-4, 0.5
GRIDS = [16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 90, 96]


def _w(name, n, box, wells, n_occ, n_o, pairs, n_s, steps, precision):
    return {"name": name, "kind": "w", "n": n, "box": box, "wells": wells, "n_occ": n_occ, "n_o": n_o, "pairs": pairs,
            "n_s": n_s, "steps": steps, "precision": precision}


def listed():
    return [
        # the 16^3 parity system, whole run in FP64: a small molecule, where launches count
        _w("w16_fp64", 16, 8.0, 4, 4, 2, 3, 10, 200, "fp64"),
        # the smallest system of the 64-system batch (500 steps there)
        _w("w32_mixed", 32, 8.0, 11, 16, 4, 10, 10, 200, "mixed"),
        # a run of a box-size sweep at fixed spacing: an odd grid edge, an odd number of pairs and orbitals
        _w("w45_mixed", 45, 15.0, 20, 30, 5, 15, 7, 60, "mixed"),
        # a 40^3 batch system as an FP64 reference run
        _w("w40_fp64", 40, 10.0, 13, 20, 4, 10, 10, 30, "fp64"),
        # the 48^3, 120-electron system, all 36 pairs
        _w("w48_mixed", 48, 16.0, 40, 60, 8, 36, 10, 100, "mixed"),
        # the paper-scale 96^3, 520-electron system: one block of 68 of its 136 pairs
        _w("w96_mixed", 96, 24.0, 170, 260, 16, 68, 10, 30, "mixed"),
        # A and the lowest ten excitons of the 48^3 system (8 x 16 window)
        {"name": "excitons48_mixed", "kind": "excitons", "n": 48, "box": 16.0, "wells": 40, "n_occ": 60, "n_o": 8,
         "n_c": 16, "k": 10, "precision": "mixed"},
        # the same of the 96^3 system (16 x 32 window; only the states of the window enter)
        {"name": "excitons96_mixed", "kind": "excitons", "n": 96, "box": 24.0, "wells": 40, "n_occ": 20, "n_o": 16,
         "n_c": 32, "k": 10, "precision": "mixed"},
        # absorption spectrum of a 512 x 512 A, 4096 Chebyshev terms
        {"name": "absorption512", "kind": "absorption", "n": 48, "box": 16.0, "wells": 40, "n_occ": 60, "n_o": 16,
         "n_c": 32, "terms": 4096, "broadening": 0.02, "omegas": 400, "axis": 0},
        # absorption spectrum in the mixed hole-grid representation (the whole virtual space)
        {"name": "holegrid32", "kind": "holegrid", "n": 32, "box": 8.0, "wells": 11, "n_occ": 16, "n_o": 4, "n_c": 8,
         "terms": 200, "broadening": 2.0, "omegas": 200, "axis": 2},
        # inference of the configured 64^3 surrogate, one full batch
        {"name": "fno64_forward", "kind": "fno", "n": 64, "width": 32, "modes": 12, "layers": 4, "batch": 4, "train": False},
        # its gradients, one training batch
        {"name": "fno64_gradients", "kind": "fno", "n": 64, "width": 32, "modes": 12, "layers": 4, "batch": 4, "train": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["w", "w", "w", "w64", "excitons", "absorption", "holegrid", "fno", "fno"])
    if kind in ("w", "w64"):
        fp64 = kind == "w64"
        n = rng.choice([g for g in GRIDS if g <= (48 if fp64 else 96)])
        n_occ = _log_int(rng, 4, 30 if fp64 else 120)
        n_o = rng.randint(1, min(6 if fp64 else 9, n_occ))
        pairs = rng.randint(1, n_o * (n_o + 1) // 2)
        n_s = rng.randint(4, 12)
        budget = (5e8 if fp64 else 4e9) / (pairs * n_s * n ** 3)
        return {"kind": "w", "n": n, "box": round(n * rng.uniform(0.25, 0.45), 2), "wells": max(2, 2 * n_occ // 3),
                "n_occ": n_occ, "n_o": n_o, "pairs": pairs, "n_s": n_s,
                "steps": max(3, min(_log_int(rng, 20, 200), int(budget))), "precision": "fp64" if fp64 else "mixed"}
    n = rng.choice([g for g in GRIDS if g <= (64 if kind == "excitons" else 40)])
    case = {"kind": kind, "n": n, "box": round(n * rng.uniform(0.25, 0.45), 2), "wells": rng.randint(4, 40)}
    if kind == "excitons":
        n_o, n_c = rng.randint(1, 12), rng.randint(1, 24)
        case.update({"n_occ": n_o + rng.randint(0, 20), "n_o": n_o, "n_c": n_c, "k": rng.randint(1, min(10, n_o * n_c)),
                     "precision": "fp64" if n <= 36 and rng.random() < 0.3 else "mixed"})
    elif kind == "absorption":
        n_o = rng.randint(2, 12)
        case.update({"n_occ": n_o + rng.randint(0, 20), "n_o": n_o, "n_c": rng.randint(2, 24), "terms": _log_int(rng, 128, 4096),
                     "broadening": 0.05, "omegas": rng.randint(50, 1000), "axis": rng.randint(0, 2)})
    elif kind == "holegrid":
        n_o = rng.randint(1, 5)
        case.update({"n_occ": n_o + rng.randint(0, 12), "n_o": n_o, "n_c": rng.randint(1, 8), "terms": rng.randint(20, 150),
                     "broadening": 2.0, "omegas": rng.randint(50, 400), "axis": rng.randint(0, 2)})
    else:
        n = rng.choice([16, 20, 24, 27, 32, 40, 48, 64])
        case = {"kind": "fno", "n": n, "width": 2 * rng.randint(2, 16), "modes": rng.randint(2, min(12, n // 2)),
                "layers": rng.randint(1, 4), "batch": rng.randint(1, 4), "train": rng.random() < 0.5}
    return case


# ---- inputs ------------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _k2(n, box):
    k = 2.0 * math.pi / box * torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64)
    return k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2


def _wells(n, box, count, seed):
    """Gaussian wells of depth 2..4 Ha and width 0.8..1.2 bohr in the inner half of the box."""
    u = torch.rand((count, 5), generator=_gen(seed), device="cuda", dtype=torch.float64)
    x = torch.arange(n, device="cuda", dtype=torch.float64) * (box / n)
    d = x[None, None, :] - (box / 4 + box / 2 * u[:, 2:5])[:, :, None]
    d = d - box * torch.round(d / box)
    g = torch.exp(-d * d / (2.0 * (0.8 + 0.4 * u[:, 1])[:, None, None] ** 2))
    return -torch.einsum("w,wz,wy,wx->zyx", 2.0 + 2.0 * u[:, 0], g[:, 2], g[:, 1], g[:, 0])


def _inner(x, y, n):
    """x y^T over n^3 grid points, summed plane by plane (one long product of few rows runs on one SM)."""
    return torch.bmm(x.reshape(-1, n, n * n).transpose(0, 1), y.reshape(-1, n, n * n).permute(1, 2, 0)).sum(0)


def _orthonormal(x, n, dv):
    for _ in range(2):
        low = torch.linalg.cholesky(_inner(x, x, n) * dv)
        x = torch.linalg.inv(low) @ x
    return x


def _system(case, seed, n_c):
    """V_loc and approximate eigenstates of H0: random fields through imaginary-time filters of decreasing
    step, each followed by orthonormalisation and the rotation to the Ritz vectors of H0. Returns v (n^3),
    phi (states x n^3), eps (FP64, device)."""
    n, box, m = case["n"], case["box"], case["n_occ"] + n_c
    dv, k2 = (box / n) ** 3, _k2(n, box)
    v = _wells(n, box, case["wells"], seed)
    x = torch.randn((m, n ** 3), generator=_gen(seed + 1), device="cuda", dtype=torch.float64)
    rows = max(1, int(6e7) // n ** 3)
    for tau, sweeps in ((0.1, 8), (0.1, 20), (0.05, 20), (0.02, 20)):
        pv, pk = torch.exp(-0.5 * tau * v).float(), torch.exp(-0.5 * tau * k2[..., :n // 2 + 1]).float()
        for r in range(0, m, rows):
            y = x[r:r + rows].float().reshape(-1, n, n, n)
            for _ in range(sweeps):
                y = pv * torch.fft.irfftn(pk * torch.fft.rfftn(pv * y, dim=(1, 2, 3)), s=(n, n, n), dim=(1, 2, 3))
            x[r:r + rows] = y.reshape(y.shape[0], -1)
        x = _orthonormal(x, n, dv)
        hx = torch.empty_like(x)
        for r in range(0, m, rows):
            y = x[r:r + rows].reshape(-1, n, n, n)
            hx[r:r + rows] = (torch.fft.irfftn(0.5 * k2[..., :n // 2 + 1] * torch.fft.rfftn(y, dim=(1, 2, 3)), s=(n, n, n),
                                               dim=(1, 2, 3)) + v * y).reshape(y.shape[0], -1)
        h = _inner(x, hx, n) * dv
        eps, u = torch.linalg.eigh(0.5 * (h + h.T))
        x = u.T @ x
    return v, x.contiguous(), eps


def _pinned(t):
    out = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    out.copy_(t)
    return out


def _context(case, seed, n_c, precision):
    v, phi, eps = _system(case, seed, n_c)
    ctx = B.Context(0, B.SBSE_FP64 if precision == "fp64" else B.SBSE_MIXED)
    ctx.set_grid(case["n"], case["box"], v.cpu().numpy())
    ctx.set_orbitals(case["n_occ"], case["n_o"], n_c, _pinned(phi).numpy(), eps.cpu().numpy(), SCISSOR)
    return ctx


def _all_pairs(n_o):
    return [(i, j) for i in range(n_o) for j in range(i, n_o)]


def _coeff(case, seed):
    return np.random.default_rng(seed + 2).standard_normal((case["n_s"], case["n_occ"]))


def _fno_shapes(case):
    w, m = case["width"], case["modes"]
    shapes = [("lift_w", (w, 2)), ("lift_b", (w,))]
    for i in range(case["layers"]):
        shapes += [("spec%d" % i, (2 * m, 2 * m, m, w, w, 2)), ("w%d" % i, (w, w)), ("b%d" % i, (w,))]
    return shapes + [("proj_w", (w,)), ("proj_b", (1,))]


def _split(case, flat):
    out, o = {}, 0
    for name, shape in _fno_shapes(case):
        size = math.prod(shape)
        out[name] = flat[o:o + size].reshape(shape)
        o += size
    return out


def _fno_inputs(case, seed):
    """Parameters (initialised as for training, biases at work), inputs and dL/dy: FP32, device."""
    g, n, w, b = _gen(seed), case["n"], case["width"], case["batch"]
    parts = []
    for name, shape in _fno_shapes(case):
        if name.startswith("spec"):
            p = torch.rand(shape, generator=g, device="cuda") / (w * w)
        else:
            p = torch.randn(shape, generator=g, device="cuda")
            p = p * (0.1 if name.startswith("b") or name.endswith("_b") else 0.7 if name == "lift_w" else w ** -0.5)
        parts.append(p.reshape(-1))
    soft = torch.exp(-_k2(n, 8.0) / 8.0).float()
    f = torch.randn((b, 2, n, n, n), generator=g, device="cuda")
    f = torch.fft.ifftn(soft * torch.fft.fftn(f, dim=(2, 3, 4)), dim=(2, 3, 4)).real
    rho = f[:, 0] * f[:, 1]
    x = torch.empty((b, 2, n, n, n), device="cuda")
    x[:, 0] = rho / rho.std()
    v = _wells(n, 16.0, 40, seed + 1).float()
    x[:, 1] = v / v.std()
    dy = torch.randn((b, n, n, n), generator=g, device="cuda") / (b * n ** 3)
    return torch.cat(parts), x, dy


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fno":
        par, x, dy = _fno_inputs(case, seed)
        net = B.FNO(case["n"], width=case["width"], modes=case["modes"], layers=case["layers"], max_batch=case["batch"])
        net.set_params(_pinned(par).numpy())
        state = {"kind": kind, "case": case, "net": net, "x": x}
        if case["train"]:
            state.update({"dy": dy, "grad": torch.empty(net.n_params, dtype=torch.float32, pin_memory=True)})
        else:
            state["y"] = torch.empty((case["batch"],) + (case["n"],) * 3, device="cuda")
        return state
    if kind == "w":
        ctx = _context(case, seed, 1, case["precision"])
        pairs = _all_pairs(case["n_o"])[:case["pairs"]]
        p = B.TDHParams(n_s=case["n_s"], n_steps=case["steps"], clean_every=10, dt=DT, gamma=GAMMA, alpha=ALPHA)
        return {"kind": kind, "ctx": ctx, "params": p.to_c(), "mixed": case["precision"] == "mixed",
                "pi": np.array([a for a, _ in pairs], dtype=np.int32), "pj": np.array([b for _, b in pairs], dtype=np.int32),
                "coeff": _coeff(case, seed), "w": torch.empty((len(pairs), ctx.n_g), dtype=torch.float64, pin_memory=True)}
    ctx = _context(case, seed, case["n_c"], case.get("precision", "fp64"))
    B.sbse_bare_W(ctx.h, _all_pairs(case["n_o"]))  # W of every pair; its values do not change the work
    state = {"kind": kind, "ctx": ctx, "case": case}
    if kind == "absorption":
        ctx.build_A(copy_out=False)
    if kind in ("absorption", "holegrid"):
        state["omega"] = _omegas(case)
    return state


def _omegas(case):
    return np.linspace(0.1, 10.0, case["omegas"])


def _interval(case):
    """Encloses the spectrum of the hole-grid operator: the largest kinetic energy of the grid and a margin."""
    return -8.0, 1.5 * (math.pi * case["n"] / case["box"]) ** 2 + 24.0


def run(state):
    kind = state["kind"]
    if kind == "w":
        # the C entry point with a pinned result buffer that the program keeps
        ctx, ip, dp = state["ctx"], C.POINTER(C.c_int), C.POINTER(C.c_double)
        rc = B.load().sbse_apply_W(ctx.h, C.byref(state["params"]), len(state["pi"]), state["pi"].ctypes.data_as(ip),
                                   state["pj"].ctypes.data_as(ip), state["coeff"].ctypes.data_as(dp),
                                   C.cast(state["w"].data_ptr(), dp))
        if rc != B.SBSE_OK:
            raise B.SbseError(rc, B.sbse_last_error(ctx.h))
        return state["w"].cuda(non_blocking=True).float() if state["mixed"] else state["w"]
    if kind == "excitons":
        a, e = state["ctx"].build_A(), state["ctx"].spectrum(state["case"]["k"])
        if state["case"]["precision"] == "mixed":
            a, e = a.astype(np.float32), e.astype(np.float32)
        return {"A": a, "excitons": e}
    if kind == "absorption":
        c = state["case"]
        sigma, residues = state["ctx"].absorption(c["axis"], c["terms"], c["broadening"], state["omega"])
        return {"sigma": sigma, "residues": residues}
    if kind == "holegrid":
        c = state["case"]
        sigma, residues = B.sbse_absorption_mixed(state["ctx"].h, B.SBSE_Q_OCCUPIED, c["axis"], c["terms"], *_interval(c),
                                                  c["broadening"], state["omega"])
        return {"sigma": sigma, "residues": residues}
    net, c = state["net"], state["case"]
    if not c["train"]:
        net.forward(c["batch"], state["x"].data_ptr(), state["y"].data_ptr())
        return state["y"]
    net.gradients(c["batch"], state["x"].data_ptr(), state["dy"].data_ptr())
    rc = B.load().sbse_fno_get_params(net.h, None, C.cast(state["grad"].data_ptr(), C.POINTER(C.c_float)))
    if rc != B.SBSE_OK:
        raise B.SbseError(rc, "sbse_fno_get_params")
    return _split(c, state["grad"])


def work(case):
    kind, n = case["kind"], case["n"]
    g = n ** 3
    fft = 5.0 * g * math.log2(g)
    if kind == "w":
        # each step reads and writes every propagated orbital once (they exceed the caches on the grids
        # that matter); two transforms and the phases per orbital, two Poisson transforms per two pairs,
        # overlaps and projection at each cleaning
        c = 8 if case["precision"] == "mixed" else 16
        p, s = case["pairs"], case["n_s"]
        orbitals, cleanings = (p + 1) * s, -(-case["steps"] // 10)
        flops = case["steps"] * (orbitals * (2 * fft + 36 * g) + p * fft) + cleanings * p * s * case["n_occ"] * g * 8.0
        return {"bytes": case["steps"] * orbitals * g * 2 * c + (case["n_occ"] + p) * g * 8, "flops": flops}
    t = 4 if case.get("precision") == "mixed" else 8
    if kind == "excitons":
        m, p = case["n_o"] * case["n_c"], case["n_o"] * (case["n_o"] + 1) // 2
        return {"bytes": (case["n_o"] + case["n_c"]) * g * t + p * g * 8 + 8 * m * m,
                "flops": m * fft + 2.0 * g * m * m + 2.0 * g * case["n_c"] ** 2 * p + 4.0 / 3.0 * m ** 3}
    if kind == "absorption":
        m = case["n_o"] * case["n_c"]
        return {"bytes": (case["n_o"] + case["n_c"]) * g * 8 + m * m * 8,
                "flops": 2.0 * m * g + 2.0 * m * m * case["terms"] + 4.0 * case["terms"] ** 2 + 10.0 * case["terms"] * case["omegas"]}
    if kind == "holegrid":
        n_o, p = case["n_o"], case["n_o"] * (case["n_o"] + 1) // 2
        return {"bytes": (case["n_occ"] + p + 1) * g * 8,
                "flops": case["terms"] * ((n_o + 1) * fft + 2.0 * g * n_o * (n_o + 2 * case["n_occ"] + 6))}
    b, w, m, layers = case["batch"], case["width"], case["modes"], case["layers"]
    modes = 4 * m ** 3
    one = b * w * (2 * fft / 2) + 8.0 * b * modes * w * w + 2.0 * b * g * w * w
    weights = layers * modes * w * w * 2
    if case["train"]:
        return {"bytes": 2 * weights + 4 * weights + (layers + 1) * b * w * g * 4 * 2 + 3 * b * g * 4, "flops": 3 * layers * one}
    return {"bytes": 2 * weights + 3 * b * g * 4, "flops": layers * one}


# ---- the same quantities in 64 bits -------------------------------------------------------------------

def _fft(x):
    return torch.fft.fftn(x, dim=(-3, -2, -1))


def _ifft(x):
    return torch.fft.ifftn(x, dim=(-3, -2, -1))


def _coulomb(rho, k2):
    kernel = torch.where(k2 > 0, 4.0 * math.pi / torch.where(k2 > 0, k2, torch.ones_like(k2)), torch.zeros_like(k2))
    return _ifft(kernel * _fft(rho)).real


def _exact_w(case, seed):
    """Stochastic TDH in the difference form d = eta^alpha - eta^0, groups of pairs in step."""
    n, n_s, n_occ, steps = case["n"], case["n_s"], case["n_occ"], case["steps"]
    k2, dv = _k2(n, case["box"]), (case["box"] / n) ** 3
    v, phi, _ = _system(case, seed, 1)
    occ = phi[:n_occ]
    window = occ[n_occ - case["n_o"]:].reshape(-1, n, n, n)
    a0 = (torch.from_numpy(_coeff(case, seed)).cuda() @ occ).reshape(n_s, n, n, n) / math.sqrt(n_s)
    norm0 = (a0 ** 2).sum((1, 2, 3)) * dv
    pv, kin = torch.exp(-0.5j * DT * v), torch.exp(-0.5j * DT * k2)
    t = torch.arange(steps + 1, dtype=torch.float64) * DT
    wt = torch.exp(-0.5 * GAMMA ** 2 * t * t) * DT / ALPHA
    wt[0], wt[-1] = 0.5 * wt[0], 0.5 * wt[-1]

    def weight(a, d):  # |a + d|^2 - |a|^2
        return 2.0 * (a.real * d.real + a.imag * d.imag) + d.real ** 2 + d.imag ** 2

    def half(a, d, u):
        ph = 0.25 * DT * u
        em1 = (-2j * torch.sin(ph) * torch.exp(-1j * ph))[:, None]
        return pv * (em1 * a + (1.0 + em1) * d)

    out, pairs = [], _all_pairs(case["n_o"])[:case["pairs"]]
    group = max(1, int(7e7) // (n_s * n ** 3))
    for g in range(0, len(pairs), group):
        q = _coulomb(torch.stack([window[i] * window[j] for i, j in pairs[g:g + group]]), k2)
        a = a0 + 0j
        d = (-2j * torch.sin(0.5 * ALPHA * q) * torch.exp(-0.5j * ALPHA * q))[:, None] * a
        u, w = torch.zeros_like(q), q.clone()
        for step in range(steps):
            if step % 10 == 0:
                f = torch.view_as_real(d.reshape(-1, n ** 3)).movedim(2, 0).reshape(-1, n ** 3)
                f = f - (_inner(f, occ, n) * dv) @ occ
                d = torch.complex(*f.reshape(2, -1)).reshape(d.shape)
                x = weight(a, d).sum((2, 3, 4)) * dv / norm0
                sq = torch.sqrt(1.0 + x)
                cm1 = (-x / (sq * (1.0 + sq)))[:, :, None, None, None]
                d = (1.0 + cm1) * d + cm1 * a
                u = _coulomb(2.0 * weight(a, d).sum(1), k2)
            w += wt[step].item() * u
            d = _ifft(kin * _fft(half(a, d, u)))
            a = _ifft(kin * _fft(pv * a))
            u = _coulomb(2.0 * weight(a, d).sum(1), k2)
            d, a = half(a, d, u), pv * a
        out.append((w + wt[steps].item() * u).reshape(-1, n ** 3))
    return torch.cat(out)


def _exact_A(case, seed):
    n, n_o, n_c = case["n"], case["n_o"], case["n_c"]
    g, dv, k2 = n ** 3, (case["box"] / case["n"]) ** 3, _k2(case["n"], case["box"])
    _, phi, eps = _system(case, seed, n_c)
    po, pc = phi[case["n_occ"] - n_o:case["n_occ"]], phi[case["n_occ"]:]
    m = n_o * n_c
    pot = torch.empty((m, g), dtype=torch.float64, device="cuda")
    for i in range(n_o):
        pot[i * n_c:(i + 1) * n_c] = _coulomb((po[i] * pc).reshape(n_c, n, n, n), k2).reshape(n_c, g)
    k = torch.empty((m, m), dtype=torch.float64, device="cuda")
    d = torch.empty((n_o, n_c, n_o, n_c), dtype=torch.float64, device="cuda")
    for i in range(n_o):
        k[i * n_c:(i + 1) * n_c] = _inner(po[i] * pc, pot, n) * dv
        for j in range(i, n_o):
            w = _coulomb((po[i] * po[j]).reshape(n, n, n), k2).reshape(g)
            blk = _inner(pc * w, pc, n) * dv
            d[i, :, j], d[j, :, i] = blk, blk.T
    diag = (eps[case["n_occ"]:][None, :] - eps[case["n_occ"] - n_o:case["n_occ"]][:, None] + SCISSOR).reshape(-1)
    return torch.diag(diag) + 2.0 * k - d.reshape(m, m), po, pc


def _coordinate(case):
    n, box = case["n"], case["box"]
    shape = [1, 1, 1]
    shape[2 - case["axis"]] = n
    x = torch.arange(n, device="cuda", dtype=torch.float64) * (box / n) - 0.5 * box
    return x.reshape(shape).expand(n, n, n).reshape(-1)


def _exact_spectrum(case, f0, dot, apply, c, w):
    """Residues of the Chebyshev recursion and the Gaussian-smoothed spectrum on Chebyshev-Gauss nodes."""
    k, s = case["terms"], case["broadening"]
    prev, cur = f0, (apply(f0) - c * f0) / w
    residues = [dot(f0, f0), dot(f0, cur)]
    for _ in range(2, k):
        prev, cur = cur, 2.0 * (apply(cur) - c * cur) / w - prev
        residues.append(dot(f0, cur))
    r = torch.stack(residues)[:k]
    node = (torch.arange(k, dtype=torch.float64, device="cuda") + 0.5) / k
    order = torch.arange(k, dtype=torch.float64, device="cuda")
    weight = torch.where(order == 0, 1.0, 2.0) * r
    dens = torch.cat([torch.cos(math.pi * torch.remainder(b[:, None] * order[None, :], 2.0)) @ weight for b in node.split(512)])
    om = torch.from_numpy(_omegas(case)).cuda()
    e = (c + w * torch.cos(math.pi * node)[None, :] - om[:, None]) / s
    sigma = om / k / (s * math.sqrt(2.0 * math.pi)) * (torch.exp(-0.5 * e * e) @ dens)
    return {"sigma": sigma, "residues": r}


def _exact_absorption(case, seed):
    a, po, pc = _exact_A(case, seed)
    f0 = (_inner(po * _coordinate(case), pc, case["n"]) * (case["box"] / case["n"]) ** 3).reshape(-1)
    dia = torch.diagonal(a)
    rad = a.abs().sum(1) - dia.abs()
    lo, hi = (dia - rad).min(), (dia + rad).max()
    return _exact_spectrum(case, f0, torch.dot, lambda x: a @ x, 0.5 * (lo + hi), 1.01 * 0.5 * (hi - lo))


def _exact_holegrid(case, seed):
    n, n_o, n_occ = case["n"], case["n_o"], case["n_occ"]
    dv, k2 = (case["box"] / n) ** 3, _k2(n, case["box"])
    v, phi, eps = _system(case, seed, case["n_c"])
    occ = phi[:n_occ]
    po, eo = occ[n_occ - n_o:], eps[n_occ - n_o:n_occ]
    w = torch.stack([_coulomb((po[i] * po).reshape(n_o, n, n, n), k2).reshape(n_o, -1) for i in range(n_o)])

    def outside(f):
        return f - (_inner(f, occ, n) * dv) @ occ

    def apply(f):
        kinetic = _ifft(0.5 * k2 * _fft(f.reshape(n_o, n, n, n))).real.reshape(n_o, -1)
        pot = _coulomb((2.0 * (po * f).sum(0)).reshape(n, n, n), k2).reshape(-1)
        return outside(kinetic + (v.reshape(-1) + SCISSOR - eo[:, None]) * f + pot * po - torch.einsum("ir,ijr->jr", f, w))

    f0 = outside(_coordinate(case) * po)
    dot = lambda x, y: (x * y).sum() * dv  # noqa: E731
    lo, hi = _interval(case)
    return _exact_spectrum(case, f0, dot, apply, 0.5 * (lo + hi), 0.5 * (hi - lo))


def _exact_fno(case, seed):
    par, x, dy = _fno_inputs(case, seed)
    n, m = case["n"], case["modes"]
    p = {}
    for name, t in _split(case, par).items():
        # spectral and pointwise weights act as BF16 values
        t = t.bfloat16().double() if name.startswith(("spec", "w")) else t.double()
        p[name] = t.clone().requires_grad_(case["train"])
    kept = torch.cat([torch.arange(m), torch.arange(n - m, n)]).cuda()
    v = torch.einsum("ci,bizyx->bczyx", p["lift_w"], x.double()) + p["lift_b"][:, None, None, None]
    for i in range(case["layers"]):
        f = torch.fft.rfftn(v, dim=(2, 3, 4))[:, :, kept][:, :, :, kept][..., :m]
        g = torch.einsum("bizyx,zyxio->bozyx", f, torch.view_as_complex(p["spec%d" % i]))
        full = torch.zeros(g.shape[:2] + (n, n, n // 2 + 1), dtype=g.dtype, device="cuda")
        zz, yy = torch.meshgrid(kept, kept, indexing="ij")
        full[:, :, zz, yy, :m] = g
        u = torch.fft.irfftn(full, s=(n, n, n), dim=(2, 3, 4)) + torch.einsum("oi,bizyx->bozyx", p["w%d" % i], v)
        u = u + p["b%d" % i][:, None, None, None]
        v = torch.nn.functional.gelu(u) if i + 1 < case["layers"] else u
    y = torch.einsum("c,bczyx->bzyx", p["proj_w"], v) + p["proj_b"]
    if not case["train"]:
        return y
    y.backward(dy.double())
    return {name: t.grad for name, t in p.items()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "w":
        return _exact_w(case, seed)
    if kind == "excitons":
        a, _, _ = _exact_A(case, seed)
        return {"A": a, "excitons": torch.linalg.eigvalsh(0.5 * (a + a.T))[:case["k"]]}
    if kind == "absorption":
        return _exact_absorption(case, seed)
    if kind == "holegrid":
        return _exact_holegrid(case, seed)
    return _exact_fno(case, seed)
