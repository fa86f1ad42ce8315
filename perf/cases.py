"""Performance cases of the inverse-homogenization library, through its public Python entry
points (paper_2301_08911_gb300.binding, the ctypes names of include/homo.h).

A case is one call, or one short sequence of calls, that a program of this library makes in
its optimisation loop or in the setup of its warm-start network, at a grid size n the
library accepts (n = m 2^k, coarsest level at most 8 cells per axis, so the ragged sizes
are 3, 5 and 7 times a power of two). listed() names the measured ones and says what each
stands for, draw() gives others of the same ranges, prepare() makes a program's state from
a seed, run() is one pass, work() its unavoidable bytes and flops, exact() the same outputs
in 64 bits from plain torch.

Densities are blurred-noise inclusions (a fraction vf of solid voxels, the rest 1e-3), as
the benchmark and the parity tests use, passed through the radius-2 filter where the call
takes a filtered density.
"""
import math

import numpy as np
import torch

from paper_2301_08911_gb300 import binding

E0, NU, P, EMIN, RADIUS, RHO_MIN, MOVE = 1.0, 0.3, 3.0, 1e-9, 2.0, 1e-3, 0.05
TAPS = [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
BLOCKS = 5                                   # residual blocks of the warm-start network


def listed():
    return [
        # The smallest whole call: the first iteration (cold start, 1e-6) of a 16^3 cell, a
        # few hundred short kernels in series with a host decision per CG iteration.
        {"name": "iteration_16", "kind": "iteration", "n": 16, "vf": 0.3, "tol": 1e-6, "warm": False,
         "objective": "bulk"},
        # The benchmark's second size: one later iteration of a 256^3 run, every solve started
        # from the previous iterate.
        {"name": "iteration_256", "kind": "iteration", "n": 256, "vf": 0.3, "tol": 1e-5, "warm": True,
         "objective": "bulk"},
        # Cells of uneven size solved as one lockstep batch, a stream per cell, CG iterations as
        # CUDA graphs (the batched workload's sizes).
        {"name": "batch_uneven", "kind": "batch", "sizes": "32,48,64,96", "vf": 0.3, "tol": 1e-5},
        # The setup a changed density costs every iteration: moduli, loads, Galerkin levels and
        # the coarsest factorisation; 96 halves to a 6^3 coarsest level.
        {"name": "hierarchy_96", "kind": "hierarchy", "n": 96, "vf": 0.35},
        # One preconditioner application on a small ragged cell (24, 12, 6): launches count.
        {"name": "vcycle_24", "kind": "vcycle", "n": 24, "vf": 0.4, "precision": "fp32"},
        # The same at an ordinary size, where the small levels' many sweeps take most of it.
        {"name": "vcycle_64", "kind": "vcycle", "n": 64, "vf": 0.3, "precision": "fp32"},
        # The mixed-precision workload's preconditioner (BF16 coarse stencils), 256^3, vf 0.2.
        {"name": "vcycle_256_mixed", "kind": "vcycle", "n": 256, "vf": 0.2, "precision": "mixed"},
        # The largest single operator: K u for the 6 load cases on a 320^3 cell.
        {"name": "product_320", "kind": "product", "n": 320, "vf": 0.3},
        # The accurate true residual that certifies every solve, on a double-float field.
        {"name": "residual_160", "kind": "residual", "n": 160, "vf": 0.3},
        # What follows every solve: C^H, objective, sensitivities, filter, OC update.
        {"name": "design_192", "kind": "design", "n": 192, "vf": 0.3, "objective": "bulk"},
        # The warm-start network's forward at the size the benchmark evaluates it at.
        {"name": "predict_64", "kind": "predict", "n": 64, "vf": 0.3},
        # One step of its training at the benchmark's training size: forward, loss, backward, Adam.
        {"name": "train_64", "kind": "train", "n": 64, "vf": 0.3},
    ]


def _size(rng, lo, hi):
    """A grid size m 2^k (m = 1, 3, 5, 7) in [lo, hi], its logarithm spread over the range."""
    sizes = sorted(m << k for m in (1, 3, 5, 7) for k in range(2, 10) if lo <= (m << k) <= hi)
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(sizes, key=lambda s: abs(math.log(s / x)))


def draw(rng):
    kind = rng.choice(["iteration", "iteration", "batch", "hierarchy", "vcycle", "vcycle", "product", "residual",
                       "design", "predict", "train"])
    c = {"kind": kind, "vf": round(rng.uniform(0.1, 0.5), 4)}
    if kind == "batch":
        c["sizes"] = ",".join(str(_size(rng, 16, 96)) for _ in range(rng.randint(2, 5)))
        c["tol"] = rng.choice([1e-4, 1e-5])
        return c
    lo, hi = {"iteration": (16, 224), "hierarchy": (16, 256), "vcycle": (16, 256), "product": (16, 320),
              "residual": (16, 192), "design": (16, 256), "predict": (16, 96), "train": (16, 64)}[kind]
    c["n"] = _size(rng, lo, hi)
    if kind == "iteration":
        c["tol"] = rng.choice([1e-4, 1e-5])
        c["warm"] = rng.random() < 0.7
    if kind in ("iteration", "design"):
        c["objective"] = rng.choice(["bulk", "shear"])
    if kind == "vcycle":
        c["precision"] = rng.choice(["fp32", "fp32", "mixed"])
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed, stream=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + stream)


def _blur(x, n, sigma):
    """Periodic Gaussian blur of (..., n, n, n)."""
    f = torch.fft.fftfreq(n, device=x.device, dtype=x.dtype) ** 2
    h = torch.fft.rfftfreq(n, device=x.device, dtype=x.dtype) ** 2
    w = torch.exp(-2 * math.pi ** 2 * sigma ** 2 * (f[:, None, None] + f[None, :, None] + h[None, None, :]))
    return torch.fft.irfftn(torch.fft.rfftn(x, dim=(-3, -2, -1)) * w, s=(n, n, n), dim=(-3, -2, -1))


def _inclusions(n, vf, seed):
    """Blurred-noise inclusions: about vf of the n^3 voxels 1, the rest RHO_MIN (flat, x fastest)."""
    s = _blur(torch.rand((n, n, n), generator=_gen(seed), device="cuda"), n, 1.5 * n / 16).reshape(-1)
    cut = torch.sort(s).values[int(round((1 - vf) * n ** 3))]
    return torch.where(s >= cut, 1.0, RHO_MIN).to(torch.float32)


def _shift(a, dx, dy, dz):
    """s(v) = a(v + d) on the last three axes (z, y, x)."""
    return torch.roll(a, (-dz, -dy, -dx), (-3, -2, -1))


def _filter(a, n):
    """Periodic linear-cone filter of radius 2, in the type of a."""
    g, s, w = a.reshape(n, n, n), 0, 0.0
    for dx, dy, dz in TAPS:
        k = RADIUS - math.sqrt(dx * dx + dy * dy + dz * dz)
        if k > 0:
            s, w = s + k * _shift(g, dx, dy, dz), w + k
    return (s / w).reshape(-1)


def _filtered(case, seed):
    return _filter(_inclusions(case["n"], case["vf"], seed).double(), case["n"]).float()


def _smooth_field(n, seed, amplitude):
    """18 smooth mean-free planes, the size of a cell's displacement in voxel units."""
    out = torch.empty((18, n ** 3), device="cuda")
    for p in range(18):
        x = torch.randn((n, n, n), generator=_gen(seed, 1 + p), device="cuda")
        x = _blur(x, n, n / 12).reshape(-1)
        x = x - x.mean()
        out[p] = amplitude * x / x.std()
    return out.reshape(-1)


def _net_params(seed):
    """He-normal weights [(27, 32, c_in), (32,)] per layer, flat, gains 1 / 0.5 / 0.1 as the benchmark draws them."""
    g = torch.Generator().manual_seed(int(seed) + 77)
    gains = [1.0] + [1.0, 0.5] * BLOCKS + [0.1]
    flat = []
    for shape, gain in zip(binding.net_layer_shapes(BLOCKS), gains):
        flat.append((gain * math.sqrt(2 / (27 * shape[2])) * torch.randn(shape, generator=g)).reshape(-1))
        flat.append(0.01 * torch.randn(32, generator=g))
    return torch.cat(flat).numpy()


def _scale(n):
    return [0.11 * n, 0.12 * n, 0.1 * n, 0.03 * n, 0.035 * n, 0.04 * n]


# ------------------------------------------------------------------ one program's state
def _loop_state(case, seed):
    n = case["n"]
    rho = _inclusions(n, case["vf"], seed)
    s = {"hom": binding.Homogenization(n, E0, NU, P, EMIN), "rho": rho}
    s.update({k: torch.empty_like(rho) for k in ("filtered", "sens", "dc", "new")})
    s["u"] = torch.empty(18 * n ** 3, device="cuda")
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        cells = []
        for i, n in enumerate(int(t) for t in case["sizes"].split(",")):
            stream = torch.cuda.Stream()
            hom = binding.Homogenization(n, E0, NU, P, EMIN, stream=stream, graphs=True)
            rho = _filtered({"n": n, "vf": case["vf"]}, 16 * int(seed) + i)
            cells.append({"hom": hom, "stream": stream, "rho": rho, "u": torch.empty(18 * n ** 3, device="cuda")})
        torch.cuda.synchronize()
        return {"case": case, "cells": cells}
    n = case["n"]
    if kind == "iteration":
        s = _loop_state(case, seed)
        if case["warm"]:      # the two iterations before the measured one
            _iterate(s, case, False)
            s["rho"].copy_(s["new"])
            _iterate(s, case, True)
            s["rho"].copy_(s["new"])
        s["hi"], s["lo"] = torch.empty_like(s["u"]), torch.empty_like(s["u"])
        if case["warm"]:
            s["hom"].save_displacement(s["hi"], s["lo"])
        return {"case": case, **s}
    if kind in ("predict", "train"):
        s = {"case": case, "net": binding.WarmStartNet(BLOCKS, _net_params(seed)), "rho": _filtered(case, seed)}
        s["u"] = _smooth_field(n, seed, 0.08 * n) if kind == "train" else torch.empty(18 * n ** 3, device="cuda")
        return s
    s = {"case": case, "rho": _filtered(case, seed),
         "hom": binding.Homogenization(n, E0, NU, P, EMIN, precision=case.get("precision", "fp32"))}
    if kind == "hierarchy":
        s["out"] = [torch.empty(243 * s["hom"].level_size(k) ** 3, device="cuda")
                    for k in range(1, s["hom"].num_levels)]
        return s
    s["hom"].set_density(s["rho"])
    s["out"] = torch.empty(18 * n ** 3, device="cuda") if kind != "design" else None
    if kind == "vcycle":      # the first residual of a cold solve; the hierarchy is built before the loop
        s["in"] = _loads(_moduli(s["rho"].double()), n).float()
        s["hom"].vcycle(s["in"], s["out"])
        return s
    s["in"] = _smooth_field(n, seed, 0.05 * n)
    if kind == "residual":
        g = _gen(seed, 40)
        low = 3e-8 * s["in"] * (2 * torch.rand(s["in"].shape, generator=g, device="cuda") - 1)
        s["hom"].restore_displacement(s["in"], low)
        s["low"] = low
        s["hom"].residual("fp32")         # forms the loads, as the solve before it has
    if kind == "design":      # a solved state at the given displacement (any residual meets this tolerance)
        s["hom"].set_displacement(s["in"])
        s["hom"].solve_cases(1e30, 1, warm_start=True)
        s["design"] = _inclusions(n, case["vf"], seed)
        s.update({k: torch.empty_like(s["rho"]) for k in ("sens", "dc", "new")})
    return s


# ------------------------------------------------------------------ one pass
def _after_solve(s, case, rho):
    """C^H, objective, sensitivities, filter adjoint and OC update of a solved cell."""
    hom = s["hom"]
    C = hom.CH()
    f, g = binding.objective(case["objective"], C)
    hom.sensitivity(g, s["sens"])
    hom.filter(RADIUS, s["sens"], s["dc"])
    s["new"].copy_(rho)
    hom.update(s["dc"], s["new"], case["vf"], MOVE)
    return {"CH": C, "objective": f, "sensitivity": s["sens"], "filtered": s["dc"], "density": s["new"]}


def _iterate(s, case, warm):
    hom = s["hom"]
    hom.filter(RADIUS, s["rho"], s["filtered"])
    hom.set_density(s["filtered"])
    hom.solve_cases(case["tol"], 500, warm_start=warm)
    return _after_solve(s, case, s["rho"])


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "iteration":
        if case["warm"]:
            s["hom"].restore_displacement(s["hi"], s["lo"])
        out = _iterate(s, case, case["warm"])
        s["hom"].get_displacement(s["u"])
        return {**out, "displacement": s["u"]}
    if kind == "batch":
        cells = s["cells"]
        for c in cells:
            c["hom"].set_density(c["rho"])
        binding.solve_batch([c["hom"] for c in cells], case["tol"], 500, warm_start=False)
        CH = [c["hom"].CH() for c in cells]
        for c in cells:
            c["hom"].get_displacement(c["u"])
        return {"CH": CH, "displacement": [c["u"] for c in cells]}
    if kind == "hierarchy":
        s["hom"].set_density(s["rho"])
        for k, out in enumerate(s["out"]):
            s["hom"].get_stencil(k + 1, out)
        return s["out"]
    if kind == "vcycle":
        s["hom"].vcycle(s["in"], s["out"])
        return s["out"]
    if kind == "product":
        s["hom"].apply_K(s["in"], s["out"])
        return s["out"]
    if kind == "residual":
        s["hom"].residual_field("double_float", s["out"])
        return s["out"]
    if kind == "design":
        return _after_solve(s, case, s["design"])
    if kind == "predict":
        s["net"].predict(case["n"], s["rho"], _scale(case["n"]), s["u"])
        return s["u"]
    loss = s["net"].train_step(case["n"], s["rho"], s["u"], _scale(case["n"]), 1e-3)
    return {"loss": loss, "gradients": s["net"].grads()}


# ------------------------------------------------------------------ unavoidable work
# Bytes and flops per fine vertex. An 18-plane field is 72 B, a scalar 4 B; K u is 27 3x3
# blocks on 6 cases (2916 flops). A V-cycle reads the residual and the moduli and writes the
# correction; its flops are two sweeps and a residual per level and sweep count. A CG
# iteration adds the product, p, and r and the correction read and written.
def _vcycle_work(n):
    b, f, m, level, sweeps = (72 * 2 + 4) * n ** 3, 3 * 2916 * n ** 3, n, 0, 1
    while m % 2 == 0 and m // 2 >= 4:
        m //= 2
        level += 1
        sweeps = 1 if level == 1 else min(64, 3 * sweeps)
        b += 972 * m ** 3                                  # the stencil, once
        f += (2 * sweeps + 1) * 2916 * m ** 3
    return b, f


def _solve_work(n, iterations):
    vb, vf = _vcycle_work(n)
    setup = 8 * n ** 3 + 2 * 72 * n ** 3                   # moduli, the double-float start
    return setup + iterations * (vb + (4 + 72 * 7) * n ** 3), iterations * (vf + 3400 * n ** 3)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_solve_work(int(t), 9) for t in case["sizes"].split(",")]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    n = case["n"]
    N = n ** 3
    if kind == "iteration":
        b, f = _solve_work(n, 8 if case["warm"] else 10)
        return {"bytes": b + (72 + 144 + 24) * N, "flops": f + 8000 * N}
    if kind == "hierarchy":
        m, b, f = n, 8 * N, 0
        while m % 2 == 0 and m // 2 >= 4:
            m //= 2
            b += 2 * 972 * m ** 3                          # the stored stencil and its copy out
            f += 2 * 8 * 243 * 4 * m ** 3
        return {"bytes": b, "flops": f + 2 * (3 * m ** 3) ** 3}
    if kind == "vcycle":
        b, f = _vcycle_work(n)
        return {"bytes": b, "flops": f}
    if kind == "product":
        return {"bytes": (4 + 72 + 72) * N, "flops": 2916 * N}
    if kind == "residual":
        return {"bytes": (4 + 5 * 72) * N, "flops": 12 * 1404 * N}
    if kind == "design":
        return {"bytes": (144 + 8 + 7 * 4) * N, "flops": 8000 * N}
    conv = 2 * 27 * 32 * (16 + 32 * (2 * BLOCKS + 1)) * N
    if kind == "predict":
        return {"bytes": (4 + 72) * N, "flops": conv}
    return {"bytes": (4 + 72) * N, "flops": 3 * conv}


# ------------------------------------------------------------------ the same in 64 bits
# Fields here are (6 cases, 3 components, z, y, x); a stencil is [27](3, 3, z, y, x).
def _element():
    """Element stiffness (24 x 24, 2x2x2 Gauss) of the unit voxel and the unit-strain displacements (6, 24)."""
    lam, mu = NU / ((1 + NU) * (1 - 2 * NU)), 1 / (2 * (1 + NU))
    D = np.diag([2 * mu] * 3 + [mu] * 3)
    D[:3, :3] += lam
    K, g = np.zeros((24, 24)), (0.5 - 0.5 / math.sqrt(3), 0.5 + 0.5 / math.sqrt(3))
    for p in [(a, b, c) for a in g for b in g for c in g]:
        B = np.zeros((6, 24))
        for j in range(8):
            bit = [j & 1, j >> 1 & 1, j >> 2]
            N1 = [p[k] if bit[k] else 1 - p[k] for k in range(3)]
            s = [2 * b - 1 for b in bit]
            d = (s[0] * N1[1] * N1[2], N1[0] * s[1] * N1[2], N1[0] * N1[1] * s[2])
            for k in range(3):
                B[k, 3 * j + k] = d[k]
            for row, (a, b) in enumerate([(0, 1), (1, 2), (0, 2)]):
                B[3 + row, 3 * j + a], B[3 + row, 3 * j + b] = d[b], d[a]
        K += B.T @ D @ B / 8
    chi = np.zeros((6, 8, 3))
    for j in range(8):
        x = (j & 1, j >> 1 & 1, j >> 2)
        for k in range(3):
            chi[k, j, k] = x[k]
        for i, (a, b) in enumerate([(0, 1), (1, 2), (0, 2)]):
            chi[3 + i, j, a], chi[3 + i, j, b] = x[b] / 2, x[a] / 2
    return torch.tensor(K, device="cuda"), torch.tensor(chi.reshape(6, 24), device="cuda")


def _bits(j):
    return j & 1, j >> 1 & 1, j >> 2


def _moduli(rho):
    return EMIN + rho ** P * (E0 - EMIN)


def _scatter(fe, n):
    """Element vectors (24, z, y, x) summed at the vertices (3, z, y, x)."""
    return sum(torch.roll(fe[3 * j:3 * j + 3], _bits(j)[::-1], (-3, -2, -1)) for j in range(8))


def _loads(E, n):
    """Loads of the 6 unit strains (flat, 18 planes), in the type of E; zero where E is uniform."""
    K, chi = _element()
    g = E.reshape(1, n, n, n)
    f = torch.stack([_scatter((K @ chi[i])[:, None, None, None] * g, n) for i in range(6)])
    return f.reshape(-1)


def _product(E, u, n):
    """K u of 64-bit u (18 planes)."""
    K, _ = _element()
    out = torch.empty((6, 3, n, n, n), device="cuda", dtype=torch.float64)
    for i, ui in enumerate(u.reshape(6, 3, n, n, n)):
        ue = torch.cat([_shift(ui, *_bits(j)) for j in range(8)])
        out[i] = _scatter((K @ ue.reshape(24, -1)).reshape(24, n, n, n) * E.reshape(1, n, n, n), n)
        del ue
    return out.reshape(-1)


def _fine_stencil(E, n):
    K, _ = _element()
    g = E.reshape(n, n, n)
    st = torch.zeros((27, 3, 3, n, n, n), device="cuda", dtype=torch.float64)
    for i in range(8):
        Ei = torch.roll(g, _bits(i)[::-1], (-3, -2, -1))       # the element whose vertex i is v
        for j in range(8):
            d = [_bits(j)[k] - _bits(i)[k] for k in range(3)]
            t = d[0] + 1 + 3 * (d[1] + 1) + 9 * (d[2] + 1)
            st[t] += K[3 * i:3 * i + 3, 3 * j:3 * j + 3, None, None, None] * Ei
    return st


def _coarsen(st):
    """Galerkin product R st I, one axis at a time (x, y, z are tensor axes 5, 4, 3 of st)."""
    for ax, step in ((5, 1), (4, 3), (3, 9)):
        m = st.shape[ax]
        out = None
        pick = {a: (torch.arange(m // 2, device="cuda") * 2 + a) % m for a in (-1, 0, 1)}
        for t in range(27):
            D = t // step % 3 - 1
            acc = 0
            for a in (-1, 0, 1):
                for e in (-1, 0, 1):
                    b = 2 * D + e - a
                    if -1 <= b <= 1:
                        acc = acc + (0.5 if a else 1.0) * (0.5 if e else 1.0) * st[t + (b - D) * step].index_select(ax - 1, pick[a])
            if out is None:
                out = torch.empty((27,) + acc.shape, device="cuda", dtype=acc.dtype)
            out[t] = acc
        st = out
    return st


def _restrict(u):
    for ax in (-1, -2, -3):
        m = u.shape[ax]
        i = torch.arange(0, m, 2, device="cuda")
        u = u.index_select(ax, i) + 0.5 * (u.index_select(ax, (i + 1) % m) + u.index_select(ax, (i - 1) % m))
    return u


def _prolong(u):
    for ax in (-1, -2, -3):
        v = torch.stack([u, 0.5 * (u + torch.roll(u, -1, ax))], dim=u.dim() + ax + 1)
        u = v.flatten(u.dim() + ax, u.dim() + ax + 1)
    return u


def _apply(st, u, diagonal=True):
    return sum(torch.einsum("rczyx,kczyx->krzyx", st[t], _shift(u, *d)) for t, d in enumerate(TAPS)
               if diagonal or t != 13)


def _sweep(st, f, u, colours):
    n = u.shape[-1]
    i = torch.arange(n, device="cuda") % 2
    colour = i[None, None, :] + 2 * i[None, :, None] + 4 * i[:, None, None]
    inv = torch.linalg.inv(st[13].permute(2, 3, 4, 0, 1)).permute(3, 4, 0, 1, 2)
    for c in colours:
        new = torch.einsum("rczyx,kczyx->krzyx", inv, f - _apply(st, u, False))
        u = torch.where(colour == c, new, u)
    return u


def _cycle(levels, sweeps, f, k=0):
    if k + 1 == len(levels):
        n = f.shape[-1]
        A = _dense(levels[k], n)
        r = f.reshape(6, -1).clone()
        x = torch.zeros_like(r)
        keep = torch.ones(3 * n ** 3, dtype=torch.bool, device="cuda")
        keep[[0, n ** 3, 2 * n ** 3]] = False
        r = (r.reshape(6, 3, -1) - r.reshape(6, 3, -1).mean(-1, keepdim=True)).reshape(6, -1)
        x[:, keep] = torch.linalg.solve(A[keep][:, keep], r[:, keep].T).T
        x = x.reshape(6, 3, -1)
        return (x - x.mean(-1, keepdim=True)).reshape(f.shape)
    u = torch.zeros_like(f)
    for _ in range(sweeps[k]):
        u = _sweep(levels[k], f, u, range(8))
    u = u + _prolong(_cycle(levels, sweeps, _restrict(f - _apply(levels[k], u)), k + 1))
    for _ in range(sweeps[k]):
        u = _sweep(levels[k], f, u, range(7, -1, -1))
    return u


def _dense(st, n):
    """Matrix of a stencil, unknown 3-component planes (component, z, y, x)."""
    N = n ** 3
    v = torch.arange(N, device="cuda").reshape(n, n, n)
    A = torch.zeros((3, N, 3, N), device="cuda", dtype=torch.float64)
    for t, d in enumerate(TAPS):
        w = _shift(v, *d).reshape(-1)
        for r in range(3):
            for c in range(3):
                A[r, v.reshape(-1), c, w] += st[t, r, c].reshape(-1)
    return A.reshape(3 * N, 3 * N)


def _hierarchy(E, n):
    levels = [_coarsen(_fine_stencil(E, n))]
    while levels[-1].shape[-1] % 2 == 0 and levels[-1].shape[-1] // 2 >= 4:
        levels.append(_coarsen(levels[-1]))
    return levels


def _oc(rho, dc, vf):
    base = rho * (-dc).clamp(min=0).sqrt()
    lo, hi = (rho - MOVE).clamp(min=RHO_MIN), (rho + MOVE).clamp(max=1.0)
    a, b = 1e-30, 1e30
    for _ in range(300):
        s = math.sqrt(a * b)
        if torch.minimum(torch.maximum(base * s, lo), hi).mean() <= vf:
            a = s
        else:
            b = s
    return torch.minimum(torch.maximum(base * a, lo), hi)


def _exact_design(rt, u, rho, case, n):
    K, chi = _element()
    C = torch.zeros((6, 6), device="cuda", dtype=torch.float64)
    E, g = _moduli(rt), np.zeros((6, 6))
    if case["objective"] == "bulk":
        g[:3, :3] = -1 / 9
    else:
        g[3, 3] = g[4, 4] = g[5, 5] = -1 / 3
    q = torch.zeros(n ** 3, device="cuda", dtype=torch.float64)
    w = [(chi[i][:, None] - torch.cat([_shift(u.reshape(6, 3, n, n, n)[i], *_bits(j)) for j in range(8)]).reshape(24, -1))
         for i in range(6)]
    for i in range(6):
        y = K @ w[i]
        for j in range(i, 6):
            e = (y * w[j]).sum(0)
            C[i, j] = C[j, i] = (E * e).mean()
            q += (g[i, j] if i == j else 2 * g[i, j]) * e
    del w
    sens = P * rt ** (P - 1) * (E0 - EMIN) * q / n ** 3
    dc = _filter(sens, n)
    C = C.cpu().numpy()
    return {"CH": C, "objective": float((C * g).sum()), "sensitivity": sens, "filtered": dc,
            "density": _oc(rho, dc, case["vf"])}


def _exact_iteration(case, seed):
    n = case["n"]
    rho = _inclusions(n, case["vf"], seed).double()
    rt = _filter(rho, n)
    E = _moduli(rt)
    A, f = _dense(_fine_stencil(E, n), n), _loads(E, n).reshape(6, -1)
    keep = torch.ones(3 * n ** 3, dtype=torch.bool, device="cuda")
    keep[[0, n ** 3, 2 * n ** 3]] = False
    u = torch.zeros_like(f)
    L = torch.linalg.cholesky(A[keep][:, keep])
    u[:, keep] = torch.cholesky_solve(f[:, keep].T, L).T
    u = u.reshape(18, -1)
    u = (u - u.mean(1, keepdim=True)).reshape(-1)
    return {**_exact_design(rt, u, rho, case, n), "displacement": None}   # held to the solve's tolerance, not to 64 bits


def _exact_net(case, seed):
    with torch.set_grad_enabled(case["kind"] == "train"):
        return _exact_net_of(case, seed)


def _exact_net_of(case, seed):
    n = case["n"]
    x = _filtered(case, seed).double()
    flat = torch.tensor(_net_params(seed), device="cuda").double().requires_grad_(True)
    layers = [(flat[a:a + 27 * 32 * c].reshape(27, 32, c), flat[a + 27 * 32 * c:a + 27 * 32 * c + 32])
              for a, c in _offsets()]

    def conv(x, layer):
        W, b = layer
        y = 0
        for t, d in enumerate(TAPS):
            y = y + _shift(x, *d).flatten(1).T @ W[t].T
        return (y + b).T.reshape(32, n, n, n)

    zero = torch.zeros_like(x)
    h = torch.relu(conv(torch.stack([x, x * x, x ** 3] + [zero] * 13).reshape(16, n, n, n), layers[0]))
    for k in range(BLOCKS):
        h = torch.relu(conv(torch.relu(conv(h, layers[1 + 2 * k])), layers[2 + 2 * k]) + h)
    y = conv(h, layers[-1])[:18].reshape(18, -1)
    s = torch.tensor(_scale(n), device="cuda", dtype=torch.float64).repeat_interleave(3)[:, None]
    if case["kind"] == "predict":
        return (s * y).detach().reshape(-1)
    loss = ((y - _smooth_field(n, seed, 0.08 * n).double().reshape(18, -1) / s) ** 2).mean()
    loss.backward()
    return {"loss": loss.item(), "gradients": flat.grad.cpu().numpy()}


def _offsets():
    at = 0
    for shape in binding.net_layer_shapes(BLOCKS):
        yield at, shape[2]
        at += 27 * 32 * shape[2] + 32


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None
    n = case["n"]
    if kind == "iteration":       # dense Cholesky of 3 n^3 unknowns
        return _exact_iteration(case, seed) if n <= 16 and not case["warm"] else None
    if kind in ("predict", "train"):
        return _exact_net(case, seed)
    rt = _filtered(case, seed).double()
    E = _moduli(rt)
    if kind == "hierarchy":
        if n > 192:
            return None
        return [st.permute(3, 4, 5, 0, 1, 2).reshape(-1) for st in _hierarchy(E, n)]
    if kind == "vcycle":
        if n > 64 or case["precision"] != "fp32":
            return None
        levels = [_fine_stencil(E, n)] + _hierarchy(E, n)
        sweeps = [1, 1] + [min(64, 3 ** k) for k in range(1, len(levels))]
        f = _loads(E, n).float().double().reshape(6, 3, n, n, n)
        return _cycle(levels, sweeps, f).reshape(-1)
    u = _smooth_field(n, seed, 0.05 * n)
    if kind == "product":
        return _product(E, u.double(), n)
    if kind == "residual":
        low = 3e-8 * u * (2 * torch.rand(u.shape, generator=_gen(seed, 40), device="cuda") - 1)
        return _loads(E, n) - _product(E, u.double() + low.double(), n)
    return _exact_design(rt, u.double(), _inclusions(n, case["vf"], seed).double(), case, n)
