"""What a user of the exact-exchange operator has it do: the measured cases.

Each case goes through the public entry points (``exx.ExxPlan``,
``exx.ExxBatch``, ``autograd.exx_energy``) on seeded orbitals of the kind the
benchmark and the tests use: sums of s/p Gaussians on a cubic mesh, Lowdin
orthonormalised.  Sizes come from the repository's own workloads (32^3 with 4
orbitals in FP64, 96^3 with 64, 128^3, 160^3, uneven batches on 32^3..128^3) and
from the grids its tests run.  ``exact`` is the same operator in 64 bits by
plain padded torch FFTs.
"""

import math

import numpy as np
import torch

from paper_1712_07973_gb300 import autograd, exx

ALPHA = 0.25
# grids drawn from, per boundary condition (compiled sizes of the library)
FREE = (8, 9, 10, 12, 14, 16, 18, 20, 24, 28, 32, 36, 40, 48, 56, 64, 72, 80, 96, 112, 128, 160)
PERIODIC = (16, 24, 32, 48, 64, 96, 128, 192)
SLAB = (16, 32, 48, 64, 96)
WIRE = (16, 32, 48, 64, 96)
BATCH = (32, 40, 48, 64, 80, 96, 112, 128)
# most pair solves times grid points of one pass: 528 pairs on 160^3
MOST = 528 * 160 ** 3


def listed():
    return [
        # the smallest FP64 workload: 4 orbitals on 32^3, one SCF step's E_x and action
        {"name": "apply_fp64_n32_N4", "call": "apply", "bc": "sinc", "prec": "fp64", "n": 32, "N": 4},
        # a small molecule on a small mesh, as in a geometry scan: launches and latency count
        {"name": "apply_fp32_n24_N5", "call": "apply", "bc": "sinc", "prec": "fp32", "n": 24, "N": 5},
        # energies alone along a line search, ragged orbital blocks (20 = 8 + 8 + 4)
        {"name": "energy_fp32_n80_N20", "call": "energy", "bc": "sinc", "prec": "fp32", "n": 80, "N": 20},
        # the 64-orbital workload: E_x and gradient of a medium molecule
        {"name": "gradient_fp32_n96_N64", "call": "gradient", "bc": "sinc", "prec": "fp32", "n": 96, "N": 64},
        # the training path: autograd forward and backward on 128^3, a ragged last block
        {"name": "autograd_fp32_n128_N30", "call": "autograd", "bc": "sinc", "prec": "fp32", "n": 128, "N": 30},
        # the largest mesh (the large-cluster workload's grid)
        {"name": "gradient_fp32_n160_N32", "call": "gradient", "bc": "sinc", "prec": "fp32", "n": 160, "N": 32},
        # the plain FP64 path on a medium mesh
        {"name": "gradient_fp64_n64_N12", "call": "gradient", "bc": "sinc", "prec": "fp64", "n": 64, "N": 12},
        # screened hybrids (short-range kernel), an odd number of orbitals
        {"name": "apply_erfc_fp32_n56_N19", "call": "apply", "bc": "erfc", "prec": "fp32", "n": 56, "N": 19},
        # a periodic cell
        {"name": "apply_periodic_fp32_n96_N32", "call": "apply", "bc": "periodic", "prec": "fp32", "n": 96, "N": 32},
        # a surface: periodic in x and y, free in z
        {"name": "gradient_slab_fp32_n64_N16", "call": "gradient", "bc": "slab", "prec": "fp32", "n": 64, "N": 16},
        # many small molecules of uneven size in one call (CUDA graph)
        {"name": "batch_fp32_24_small", "call": "batch", "bc": "sinc", "prec": "fp32", "mols": 24,
         "n_lo": 32, "n_hi": 48, "N_lo": 8, "N_hi": 24},
        # several uneven molecules of small to large size in one call
        {"name": "batch_fp32_6_mixed", "call": "batch", "bc": "sinc", "prec": "fp32", "mols": 6,
         "n_lo": 48, "n_hi": 128, "N_lo": 8, "N_hi": 32},
    ]


def draw(rng):
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    if rng.random() < 0.2:
        hi = rng.choice((48, 80, 128))
        lo = rng.choice([g for g in BATCH if g <= hi])
        most = 24 if hi > 80 else 32
        N_lo = rng.randint(4, 12)
        return {"call": "batch", "bc": "sinc", "prec": "fp32", "mols": rng.randint(4, 8 if hi > 48 else 28),
                "n_lo": lo, "n_hi": hi, "N_lo": N_lo, "N_hi": rng.randint(N_lo + 1, most)}
    bc = rng.choice(("sinc",) * 7 + ("hockney", "erfc", "periodic", "slab", "wire"))
    prec = "fp64" if rng.random() < 0.2 else "fp32"
    grids = {"periodic": PERIODIC, "slab": SLAB, "wire": WIRE}.get(bc, FREE)
    if prec == "fp64":  # ~25 times FP32's cost per pair
        grids = [g for g in grids if g <= 96]
    want = math.exp(rng.uniform(math.log(grids[0]), math.log(grids[-1])))
    n = min(grids, key=lambda g: abs(math.log(g / want)))
    most_pairs = MOST // n ** 3 // (40 if prec == "fp64" else 1)
    if bc == "periodic" and n == 192:
        most_pairs //= 2
    N_hi = max(2, min(64, int(math.sqrt(2 * most_pairs)) - 1))
    call = rng.choice(("apply", "gradient", "gradient", "energy", "autograd"))
    return {"call": call, "bc": bc, "prec": prec, "n": n, "N": log_int(2, N_hi)}


def _molecules(case):
    """(n, N) of each molecule, the same for every seed of a case."""
    if case["call"] != "batch":
        return [(case["n"], case["N"])]
    grids = [g for g in BATCH if case["n_lo"] <= g <= case["n_hi"]]
    rng = np.random.default_rng([case["mols"], case["n_lo"], case["n_hi"], case["N_lo"], case["N_hi"]])
    return [(int(grids[int(rng.integers(len(grids)))]), int(rng.integers(case["N_lo"], case["N_hi"] + 1)))
            for _ in range(case["mols"])]


def _spacing(n):
    return {128: 0.37, 160: 0.42}.get(n, 0.4 if n >= 24 else 0.45)


def _orbitals(n, N, rng, dtype):
    """N Lowdin-orthonormal sums of s/p Gaussians on n^3, on the GPU."""
    h = _spacing(n)
    x = np.arange(n) * h
    box = (n - 1) * h
    terms = 16 if n >= 32 else 8
    sites = rng.uniform(0.2 * box, 0.8 * box, size=(max(2, N // 2), 3))
    # widths that the mesh resolves and the box holds
    s_lo, s_hi = (0.7, 1.8) if n >= 32 else (0.12 * n * h, 0.2 * n * h)
    cut = [[], [], []]
    for _ in range(N):
        R = sites[rng.integers(0, len(sites), size=terms)]
        s2 = 2.0 * rng.uniform(s_lo, s_hi, size=terms) ** 2
        kind = rng.integers(0, 4, size=terms)
        coef = rng.standard_normal(terms)
        for a in range(3):
            d = x[None, :] - R[:, a, None]
            g = np.exp(-d * d / s2[:, None]) * np.where(kind[:, None] == a + 1, d, 1.0)
            cut[a].append(g * (coef[:, None] if a == 2 else 1.0))
    X, Y, Z = (torch.from_numpy(np.stack(c)).cuda() for c in cut)  # (N, terms, n)
    phi = torch.empty((N, n ** 3), dtype=torch.float64, device="cuda")
    for o in range(N):
        yx = (Y[o][:, :, None] * X[o][:, None, :]).reshape(terms, n * n)
        phi[o] = (Z[o].T @ yx).reshape(-1)
    S = (phi @ phi.T).cpu().numpy() * h ** 3
    w, U = np.linalg.eigh(S + 1e-10 * np.trace(S) / N * np.eye(N))
    psi = torch.from_numpy((U / np.sqrt(w)) @ U.T).cuda() @ phi
    return psi.reshape(N, n, n, n).to(dtype).contiguous()


def _inputs(case, seed):
    dtype = torch.float64 if case["prec"] == "fp64" else torch.float32
    rng = np.random.default_rng([seed, 17])
    out = []
    for n, N in _molecules(case):
        psi = _orbitals(n, N, rng, dtype)
        # mostly doubly occupied, a few fractional levels
        occ = np.where(np.arange(N) < N - N // 4, 2.0, rng.uniform(0.2, 2.0, size=N))
        out.append((psi, occ))
    return out


def _omega(case):
    return 0.11 if case["bc"] == "erfc" else 0.0


def prepare(case, seed):
    """The orbitals, and the plan (or batch) and output buffers that a program keeps from step to step."""
    ins = _inputs(case, seed)
    if case["call"] == "batch":
        mols = [{"n": p.shape[-1], "h": _spacing(p.shape[-1]), "alpha": ALPHA, "occupations": occ} for p, occ in ins]
        batch = exx.ExxBatch(mols, kernel=case["bc"])
        psis = [p for p, _ in ins]
        outs = [torch.empty_like(p) for p in psis]
        batch.set_buffers(psis, outs)
        batch.graph(True)
        return {"call": "batch", "batch": batch, "psis": psis, "outs": outs, "stream": torch.cuda.Stream(),
                "E": torch.zeros(len(mols), dtype=torch.float64, device="cuda")}
    psi, occ = ins[0]
    n = case["n"]
    plan = exx.ExxPlan(n, _spacing(n), ALPHA, occ, precision=case["prec"], kernel=case["bc"], omega=_omega(case))
    state = {"call": case["call"], "plan": plan, "psi": psi}
    if case["call"] in ("apply", "gradient"):
        state["out"] = torch.empty_like(psi)
    elif case["call"] == "autograd":
        state["psi"] = psi.requires_grad_(True)
    return state


def run(state):
    call = state["call"]
    if call == "batch":
        s = state["stream"]
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            state["batch"].gradient(state["E"], stream=s)
            E = state["E"].float()  # the energies, in the precision this path computes in
        torch.cuda.current_stream().wait_stream(s)
        return {"E": E, "grad": state["outs"]}
    plan, psi = state["plan"], state["psi"]
    if call == "energy":
        return {"E": plan.energy(psi)}
    if call == "apply":
        E, vx = plan.apply(psi, state["out"])
        return {"E": E, "vx": vx}
    if call == "gradient":
        E, g = plan.gradient(psi, state["out"])
        return {"E": E, "grad": g}
    E = autograd.exx_energy(psi, plan)
    (g,) = torch.autograd.grad(E, psi)
    return {"E": E.item(), "grad": g}


def work(case):
    """Orbitals read once, the action or gradient written once (the energy alone: nothing more), and the
    real-to-complex transforms of the pair densities, there and back (there alone for the energy)."""
    size = 8 if case["prec"] == "fp64" else 4
    total_bytes, flops = 0, 0.0
    for n, N in _molecules(case):
        total_bytes += N * n ** 3 * size * (1 if case["call"] == "energy" else 2) + 8
        px, py, pz = (2 if a in _free_axes(case) else 1 for a in "xyz")
        # lines x 2.5 L log2 L (real, x) or 5 L log2 L (complex) of each axis, empty lines left out
        one = n * n * 2.5 * px * n * math.log2(px * n)
        one += (px * n / 2) * n * 5.0 * py * n * math.log2(py * n)
        one += (px * n / 2) * py * n * 5.0 * pz * n * math.log2(pz * n)
        flops += N * (N + 1) / 2 * one * (1 if case["call"] == "energy" else 2)
    return {"bytes": total_bytes, "flops": flops}


# ------------------------------------------------------------- 64-bit values
def _free_axes(case):
    return {"periodic": "", "slab": "z", "wire": "xy"}.get(case["bc"], "xyz")


def _kernel_hat(n, h, case):
    """Kernel spectrum on the padded mesh, axes z, y, x (x halved), in 64 bits.

    4 pi / k^2 = int_0^inf (2 pi / t^3) e^(-k^2 / 4 t^2) dt: a periodic axis
    contributes e^(-k_d^2 / 4 t^2), a free one the Gaussian's band-limited
    transform f(t, m).  The divergent entry of each mixed cell is regularised
    as the library documents it.
    """
    dev, dt = "cuda", torch.float64
    free = _free_axes(case)
    ax = {a: (a in free) for a in "zyx"}
    if case["bc"] == "hockney":
        d = torch.arange(n + 1, dtype=dt, device=dev)
        r = torch.sqrt(d[:, None, None] ** 2 + d[None, :, None] ** 2 + d[None, None, :] ** 2)
        W = h ** 3 / (h * r)
        W[0, 0, 0] = h ** 2 * (3.0 * math.log(2.0 + math.sqrt(3.0)) - math.pi / 2.0)
    else:
        # tau = t h on a trapezoid in log tau
        u = torch.arange(-42.0, 19.0, 0.11, dtype=dt, device=dev)
        w_u = 0.11
        if case["bc"] == "erfc":  # erfc(w r)/r: t from w up
            gx, gw = np.polynomial.legendre.leggauss(600)
            lo, hi = math.log(_omega(case) * h), 19.0
            u = torch.from_numpy(0.5 * (hi - lo) * gx + 0.5 * (hi + lo)).to(dev)
            w_u = torch.from_numpy(0.5 * (hi - lo) * gw).to(dev)
        tau = torch.exp(u)
        m = torch.arange(n + 1, dtype=dt, device=dev)
        gq, gw = np.polynomial.legendre.leggauss(480)
        q = torch.from_numpy(0.5 * math.pi * (gq + 1.0)).to(dev)
        wq = torch.from_numpy(0.5 * math.pi * gw).to(dev)
        wide = tau >= 0.2
        tw = torch.where(wide, tau, torch.ones_like(tau))
        f_q = (torch.exp(-(q[None, :] / (2 * tw[:, None])) ** 2) * wq) @ torch.cos(q[:, None] * m[None, :]) / math.pi
        f_g = tau[:, None] / math.sqrt(math.pi) * torch.exp(-(tau[:, None] * m[None, :]) ** 2)
        f = torch.where(wide[:, None], f_q, f_g)
        k = 2.0 * math.pi / n * torch.arange(n // 2 + 1, dtype=dt, device=dev)
        e = torch.exp(-(k[None, :] / (2 * tau[:, None])) ** 2)
        # integrand in log tau, in units of h: (2 pi / tau^2) prod, times h^2
        c = h ** 2 * w_u * 2.0 * math.pi / tau ** 2
        fz, fy, fx = (f if ax[a] else e for a in "zyx")
        sizes = [t.shape[1] for t in (fz, fy, fx)]
        W = torch.empty(sizes, dtype=dt, device=dev)
        cx = (c[:, None] * fx)
        for z in range(sizes[0]):
            W[z] = (fz[:, z, None] * fy).T @ cx
        if free == "":
            W = torch.zeros(sizes, dtype=dt, device=dev)
            k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2
            W = torch.where(k2 > 0, 4.0 * math.pi * h ** 2 / torch.where(k2 > 0, k2, torch.ones_like(k2)), W)
        elif free == "z":
            W[:, 0, 0] = (c[:, None] * (f - f[:, :1])).sum(0) - h ** 2 * 4.0 / math.pi
        elif free == "xy":
            p = (c[:, None, None] * (f[:, :, None] * f[:, None, :] - f[:, :1, None] * f[:, None, :1])).sum(0)
            catalan = 0.915965594177219015054603514932
            shift = -2.0 * math.log(math.pi / h) - 2.0 * 0.577215664901532860606512 + 4.0 * catalan / math.pi
            W[0, :, :] = p - h ** 2 * shift
    for i, a in enumerate("zyx"):
        half = n if ax[a] else n // 2
        L = 2 * n if ax[a] else n
        idx = torch.tensor([min(j, L - j) for j in range(L)], device=dev)
        assert W.shape[i] == half + 1
        W = W.index_select(i, idx)
    dims = [i for i, a in enumerate("zyx") if ax[a]]
    if dims:
        W = torch.fft.fftn(W, dim=dims).real
    return W[..., : W.shape[-1] // 2 + 1].contiguous()


def exact(case, seed):
    out_E, out_v = [], []
    for psi, occ in _inputs(case, seed):
        psi = psi.double()
        N, n = psi.shape[0], psi.shape[-1]
        h = _spacing(n)
        K = _kernel_hat(n, h, case)
        s = [2 * n if a in _free_axes(case) else n for a in "zyx"]
        chunk = max(1, int(1.5e8 // (s[0] * s[1] * s[2])))
        f = torch.from_numpy(occ).cuda()
        E, vx = 0.0, torch.zeros_like(psi)
        for i in range(N):
            for j0 in range(i, N, chunk):
                j1 = min(N, j0 + chunk)
                rho = psi[i] * psi[j0:j1]
                V = torch.fft.irfftn(torch.fft.rfftn(rho, s=s, dim=(1, 2, 3)) * K, s=s, dim=(1, 2, 3))
                V = V[:, :n, :n, :n]
                mult = torch.full((j1 - j0,), 2.0, dtype=torch.float64, device="cuda")
                if j0 == i:
                    mult[0] = 1.0
                E = E + f[i] * torch.sum(mult * f[j0:j1] * h ** 3 * (rho * V).sum((1, 2, 3)))
                vx[i] += torch.einsum("j,jzyx,jzyx->zyx", f[j0:j1], V, psi[j0:j1])
                lo = 1 if j0 == i else 0
                vx[j0 + lo:j1] += f[i] * V[lo:] * psi[i]
        vx *= -ALPHA
        if case["call"] != "apply":
            vx *= 2.0 * h ** 3 * f[:, None, None, None]
        out_E.append(-0.5 * ALPHA * E)
        out_v.append(vx)
    if case["call"] == "batch":
        return {"E": torch.stack(out_E), "grad": out_v}
    if case["call"] == "energy":
        return {"E": float(out_E[0])}
    return {"E": float(out_E[0]), ("vx" if case["call"] == "apply" else "grad"): out_v[0]}
