"""Performance cases: the work a user of this library has it do, through its public entry points.

A solve case is one complete PCG solve (``Solver.solve`` or ``msmg_solve_batched``) on a set-up the user
keeps; a ``step`` case is one pressure step of a time loop, where the permeability is new on every call
(``Solver.refresh`` then ``Solver.solve``); ``transport`` is the rest of that step (face velocities, mass balance
and the saturation sub-steps); ``forward`` and ``gradients`` are the warm-start network's two directions.

Solutions are taken to a relative residual of 1e-10 (the tolerance of this repository's coupled-flow tests) so
that a converged solution is determined to well below the 1e-9 at which two correct solvers are compared.

Fields and right-hand sides are seeded and synthetic, drawn on the GPU: lognormal Gaussian fields with exponential
covariance, high-contrast inclusions (spheres and channels), and layered fields with sinuous channels.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2403_19342_gb300 as msmg

P_BH = 4000.0          # producers' bottom-hole pressure of the two-phase runs
M_SUB, DS_MAX = 50, 1e-3


# ------------------------------------------------------------------ the cases
def _solve(name, grid, field, *, contrast, block, levels, L, mixed, n_rhs=1, ratio=(2, 2, 2), iters=20,
           problems=1, autotune=False, wells=False, kind="solve", rtol=1e-10):
    c = {"kind": kind, "nx": grid[0], "ny": grid[1], "nz": grid[2], "field": field, "contrast": contrast,
         "bx": block[0], "by": block[1], "bz": block[2], "rx": ratio[0], "ry": ratio[1], "rz": ratio[2],
         "levels": levels, "L": L, "mixed": mixed, "n_rhs": n_rhs, "problems": problems, "iters": iters,
         "autotune": autotune, "wells": wells, "rtol": rtol}
    if name:
        c["name"] = name
    return c


def _net(name, kind, batch, n_in, h1, h2, n_vec):
    c = {"kind": kind, "batch": batch, "n_in": n_in, "h1": h1, "h2": h2, "n_vec": n_vec}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest solve: a 32^3 parity-size field, where launches and host work count
        _solve("solve_32_fp64", (32, 32, 32), "lognormal", contrast=1e3, block=(4, 4, 4), levels=3, L=4, mixed=False,
               iters=15),
        # an ordinary solve in full double precision
        _solve("solve_96_fp64", (96, 96, 96), "lognormal", contrast=1e4, block=(8, 8, 8), levels=3, L=6, mixed=False,
               iters=22),
        # the benchmark's grid and hierarchy: 128^3 inclusions, mixed precision, variants timed at set-up
        _solve("solve_128_inclusions", (128, 128, 128), "inclusions", contrast=1e4, block=(8, 8, 8), levels=4, L=6,
               mixed=True, iters=135, autotune=True),
        # the largest single solve
        _solve("solve_256_mixed", (256, 256, 256), "lognormal", contrast=1e6, block=(8, 8, 8), levels=5, L=4,
               mixed=True, iters=43),
        # a reservoir-shaped grid with small non-cubic elements and wells (the run-time geometry)
        _solve("solve_wells_ragged", (60, 220, 85), "layered", contrast=1e6, block=(4, 4, 5), levels=3, L=4, mixed=True,
               ratio=(3, 5, 1), iters=57, wells=True),
        # many right-hand sides of one operator in one call
        _solve("solve_96_rhs16", (96, 96, 96), "lognormal", contrast=1e4, block=(8, 8, 8), levels=3, L=4, mixed=True,
               n_rhs=16, iters=24),
        # several operators at once, several right-hand sides each
        _solve("batched_4x64_rhs4", (64, 64, 64), "lognormal", contrast=1e4, block=(8, 8, 8), levels=3, L=4,
               mixed=True, n_rhs=4, problems=4, iters=26, kind="batched"),
        # a new permeability: set-up in place and one solve, 8^3 elements (iterative local eigensolver)
        _solve("step_128_new_field", (128, 128, 128), "lognormal", contrast=1e4, block=(8, 8, 8), levels=4, L=6,
               mixed=True, iters=24, kind="step"),
        # the pressure step of a two-phase run: new mobility, wells, small elements, a large coarsest level
        _solve("step_wells_ragged", (60, 220, 85), "layered", contrast=1e6, block=(4, 4, 5), levels=3, L=4, mixed=True,
               ratio=(3, 5, 1), iters=57, wells=True, kind="step"),
        # the transport part of that step: velocities, balance, 50 saturation sub-steps
        {"name": "transport_reservoir", "kind": "transport", "nx": 60, "ny": 220, "nz": 85},
        # warm-start network, inference over the elements of a large field
        _net("net_forward_8192", "forward", 8192, 512, 1024, 1024, 5),
        # warm-start network, training: loss and gradients of one batch
        _net("net_gradients_512", "gradients", 512, 512, 1024, 1024, 11),
    ]


def _log_between(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batched", "step", "step", "transport", "forward", "gradients"])
    if kind == "transport":
        side = (3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 20, 24, 25)
        return {"kind": kind, "nx": 4 * rng.choice(side[:9]), "ny": 4 * rng.choice(side), "nz": 5 * rng.choice(side[1:] + (17,))}
    if kind in ("forward", "gradients"):
        top = 8192 if kind == "forward" else 1024
        width = lambda: 64 * rng.randint(4, 16) if rng.random() < 0.75 else rng.randint(200, 1000)
        return _net(None, kind, int(_log_between(rng, 16, top)), rng.choice([512, 512, 216]), width(), width(),
                    rng.randint(3, 11))
    # a hierarchy: elements, then the element grid as top-level grid times the ratio per level
    block = rng.choice([(8, 8, 8), (8, 8, 8), (4, 4, 4), (4, 4, 5), (6, 4, 5)])
    small = block[0] * block[1] * block[2] <= 128
    levels = 3 if small else rng.choice([3, 3, 4])
    most = 2.0e6 if kind != "step" else 1.0e6
    target = _log_between(rng, 2.0e4, most)
    r = 2 ** (levels - 2)
    edge = [r * b for b in block]
    side = target ** (1.0 / 3.0)
    grid = [e * max(1, round(side * _log_between(rng, 0.7, 1.4) / e)) for e in edge]
    if grid[0] * grid[1] * grid[2] <= edge[0] * edge[1] * edge[2]:
        grid[0] = 2 * edge[0]
    # the coarsest level is dense: keep it to a few thousand unknowns
    L = rng.choice([4, 4, 6] if not small else [4])
    while (grid[0] // edge[0]) * (grid[1] // edge[1]) * (grid[2] // edge[2]) * L > 3000:
        k = max(range(3), key=lambda d: grid[d] // edge[d])
        grid[k] = edge[k] * max(1, grid[k] // edge[k] // 2)
    wells = rng.random() < 0.3
    field = rng.choice(["lognormal", "lognormal", "layered"])
    return _solve(None, grid, field, contrast=round(_log_between(rng, 1e2, 1e5)), block=block, levels=levels, L=L,
                  mixed=rng.random() < 0.7, n_rhs=1 if kind == "step" else rng.choice([1, 1, 3, 8]),
                  problems=rng.randint(2, 4) if kind == "batched" else 1, iters=30, wells=wells, kind=kind)


# ------------------------------------------------------------------ inputs
def _gen(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(int(seed) & 0x7FFFFFFF)


def _grf(shape, seed, modes=256, corr=0.1):
    """Unit-variance Gaussian field, exponential covariance, by random Fourier modes (FP32 phases)."""
    rng = np.random.default_rng(seed)
    k = rng.standard_normal((modes, 3)) / np.sqrt(rng.chisquare(1.0, size=(modes, 1))) / corr
    kt = torch.tensor(k, dtype=torch.float32, device="cuda")
    ph = torch.tensor(rng.uniform(0.0, 2.0 * math.pi, size=modes), dtype=torch.float32, device="cuda")
    nz, ny, nx = shape
    ax = [(torch.arange(m, device="cuda", dtype=torch.float32) + 0.5) / m for m in (nx, ny, nz)]
    pxy = ax[0][:, None, None] * kt[:, 0] + ax[1][None, :, None] * kt[:, 1] + ph      # [nx, ny, modes]
    pxy = pxy.transpose(0, 1)                                                             # [ny, nx, modes]
    out = torch.empty(shape, dtype=torch.float64, device="cuda")
    for z in range(nz):
        out[z] = torch.cos(pxy + ax[2][z] * kt[:, 2]).sum(dim=-1).double()
    return out * math.sqrt(2.0 / modes)


def _spread(y, contrast):
    """Log-permeability y, rescaled so that max / min of the permeability is the contrast."""
    lo, hi = y.min(), y.max()
    return torch.exp((y - lo) / (hi - lo) * math.log(contrast))


def _inclusions(shape, seed, k_hi):
    """Background 1; per 128^3 cells 200 spheres of 1.5-6 cells and 20 full-length 2x2 channels at k_hi."""
    rng = np.random.default_rng(seed)
    nz, ny, nx = shape
    n = nx * ny * nz
    k = torch.ones(shape, dtype=torch.float64, device="cuda")
    for _ in range(max(4, round(200 * n / 128 ** 3))):
        c = rng.uniform(0.0, 1.0, size=3) * (nz, ny, nx)
        r = rng.uniform(1.5, 6.0)
        lo = np.maximum((c - r).astype(int) - 1, 0)
        hi = np.minimum((c + r).astype(int) + 2, shape)
        d = [torch.arange(lo[i], hi[i], device="cuda", dtype=torch.float64) + 0.5 - c[i] for i in range(3)]
        inside = d[0][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[2][None, None, :] ** 2 <= r * r
        k[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]][inside] = k_hi
    for _ in range(max(2, round(20 * (n / 128 ** 3) ** (2 / 3)))):
        axis = int(rng.integers(0, 3))
        a, b = (int(v) for v in rng.integers(0, min(shape) - 1, size=2))
        if axis == 0:
            k[a:a + 2, b:b + 2, :] = k_hi
        elif axis == 1:
            k[a:a + 2, :, b:b + 2] = k_hi
        else:
            k[:, a:a + 2, b:b + 2] = k_hi
    return k


def _layered(shape, seed, contrast, lattice=(60, 220)):
    """Layers of laterally correlated lognormal noise; sinuous channels in the lower layers."""
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    z = rng.standard_normal((nz, lattice[1], lattice[0]))
    for _ in range(3):
        z = (np.roll(z, 1, 1) + 2 * z + np.roll(z, -1, 1)) / 4
        z = (np.roll(z, 1, 2) + 2 * z + np.roll(z, -1, 2)) / 4
    z /= z.std(axis=(1, 2), keepdims=True)
    yi = np.minimum(np.arange(ny) * lattice[1] // ny, lattice[1] - 1)
    xi = np.minimum(np.arange(nx) * lattice[0] // nx, lattice[0] - 1)
    k = np.exp(np.clip(z[:, yi][:, :, xi], -3, 3) / 6.0 * 0.5 * math.log(contrast))
    k_ch = math.sqrt(contrast) * k.min()
    xg, yg = (np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny
    for layer in range(nz - nz * 50 // 85, nz):
        for _ in range(int(rng.integers(2, 5))):
            xc = rng.uniform(0, 1) + rng.uniform(0.02, 0.15) * np.sin(2 * math.pi * yg / rng.uniform(0.2, 0.8)
                                                                      + rng.uniform(0, 2 * math.pi))
            k[layer][np.abs(xg[None, :] - xc[:, None]) <= rng.integers(3, 9) / nx / 2] = k_ch * math.sqrt(contrast)
    return torch.tensor(k / k.min(), device="cuda")


def _kappa(case, seed):
    shape = (case["nz"], case["ny"], case["nx"])
    if case["field"] == "inclusions":
        k = _inclusions(shape, seed, case["contrast"])
    elif case["field"] == "layered":
        k = _layered(shape, seed, case["contrast"])
    else:
        k = _spread(_grf(shape, seed), case["contrast"])
    if case["wells"]:                       # vertical permeability a tenth of the lateral one
        k = torch.stack([k, k, 0.1 * k]).contiguous()
    return k


def _spacing(case):
    if case.get("wells") or case["kind"] == "transport":
        return (20.0, 10.0, 2.0)            # feet
    return (1.0 / case["nx"], 1.0 / case["ny"], 1.0 / case["nz"])


def _well_index(h):
    """Well index per unit permeability of a producer's cell (two-point neighbours at three and one cells)."""
    r1 = math.sqrt(9 * h[0] ** 2 + h[1] ** 2) / 2
    r2 = math.sqrt(h[0] ** 2 + 9 * h[1] ** 2) / 2
    return (1 / h[0] ** 2 + 1 / h[1] ** 2) / ((2 / math.pi) * (h[1] / h[0] * math.log(r1) + h[0] / h[1] * math.log(r2)) - 1)


def _producers(ny, nx):
    return ((0, 0), (0, nx - 1), (ny - 1, 0), (ny - 1, nx - 1))


def _well_terms(case, kappa, seed):
    """Cell term W of the producers' columns and the right-hand side with the central injector."""
    shape = (case["nz"], case["ny"], case["nx"])
    w = torch.zeros(shape, dtype=torch.float64, device="cuda")
    wi = _well_index(_spacing(case))
    for j, i in _producers(shape[1], shape[2]):
        w[:, j, i] = wi * kappa[0, :, j, i]
    b = w * P_BH
    b[:, shape[1] // 2, shape[2] // 2] += 1.0e3
    return w, b


def _rhs(case, seed, n_rhs):
    """Corner source and sink; then four line sources and a central line; further ones seeded white noise."""
    shape = (case["nz"], case["ny"], case["nx"])
    f = torch.zeros((n_rhs,) + shape, dtype=torch.float64, device="cuda")
    f[0, 0, 0, 0], f[0, -1, -1, -1] = 1.0, -1.0
    if n_rhs > 1:
        for j, i in _producers(shape[1], shape[2]):
            f[1, :, j, i] = 1.0
        f[1, :, shape[1] // 2, shape[2] // 2] -= 4.0
    if n_rhs > 2:
        f[2:] = torch.randn(f[2:].shape, dtype=torch.float64, device="cuda", generator=_gen(seed))
        f[2:] -= f[2:].mean(dim=(1, 2, 3), keepdim=True)
    return f if n_rhs > 1 else f[0]


def _options(case, w=None):
    return msmg.Options(n_levels=case["levels"], block=(case["bx"], case["by"], case["bz"]),
                        ratio=[(case["rx"], case["ry"], case["rz"])] * (case["levels"] - 2),
                        n_eig=[case["L"]] * (case["levels"] - 1), precision=msmg.MIXED if case["mixed"] else msmg.FP64,
                        eig_tol=1e-8, autotune=case["autotune"], cell_diag=w)


def _problem(case, seed):
    """(kappa, cell term or None, right-hand sides) of one operator."""
    kappa = _kappa(case, seed)
    if case["wells"]:
        w, b = _well_terms(case, kappa, seed)
        if case["n_rhs"] > 1:               # the injection rate varies from one right-hand side to the next
            s = torch.linspace(0.5, 1.5, case["n_rhs"], dtype=torch.float64, device="cuda")[:, None, None, None]
            q = torch.where(w > 0, torch.zeros_like(b), b)
            b = (w * P_BH)[None] + s * q[None]
        return kappa, w, b.contiguous()
    return kappa, None, _rhs(case, seed, case["n_rhs"])


def _transport_inputs(case, seed):
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    shape = (nz, ny, nx)
    h = _spacing(case)
    k = _layered(shape, seed, 1e4)
    kappa = torch.stack([k, k, 0.1 * k]).contiguous()
    g = _gen(seed)
    phi = 0.05 + 0.25 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=g)
    S = 0.2 + 0.5 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=g)
    # pressure: an injector and four producers in line, plus the local variation a heterogeneous field gives it
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5)[None, None, :] * h[0]
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5)[None, :, None] * h[1]
    at = lambda j, i: -torch.log((x - (i + 0.5) * h[0]) ** 2 + (y - (j + 0.5) * h[1]) ** 2 + h[0] ** 2)
    p = 4.0 * at(ny // 2, nx // 2) - sum(at(j, i) for j, i in _producers(ny, nx))
    p = P_BH + 100.0 * (p - p[:, :1, :1]) + 0.1 * torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)
    wi = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for j, i in _producers(ny, nx):
        wi[:, j, i] = _well_index(h)
    q = torch.zeros(shape, dtype=torch.float64, device="cuda")
    q[:, ny // 2, nx // 2] = 20.0
    return kappa, phi, S, p.contiguous(), wi, q


def _net_inputs(case, seed):
    g = _gen(seed)
    x = 0.5 * torch.randn(case["batch"], case["n_in"], device="cuda", generator=g)
    x -= x.mean(dim=1, keepdim=True)                       # log-permeability patches, mean removed
    t = torch.randn(case["batch"], case["n_vec"], case["n_in"], device="cuda", generator=g)
    t = t * torch.exp(4 * (x - x.amax(dim=1, keepdim=True)))[:, None, :]
    t = t / t.norm(dim=2, keepdim=True)                    # unit vectors weighted like sqrt(S)
    return x, t.reshape(case["batch"], -1).contiguous()


def _net_params(case, seed):
    """{name: tensor} of the network: weights as fan-in uniform, the last layer a quarter of that, small biases."""
    g = _gen(seed + 1)
    dims = [case["n_in"], case["h1"], case["h2"], case["n_vec"] * case["n_in"]]
    P = {}
    for l in range(3):
        a = math.sqrt(6.0 / dims[l]) * (0.25 if l == 2 else 1.0)
        P["w%d" % l] = a * (2 * torch.rand(dims[l], dims[l + 1], device="cuda", generator=g) - 1)
        P["b%d" % l] = 0.02 * torch.randn(dims[l + 1], device="cuda", generator=g)
    return P


# ------------------------------------------------------------------ prepare / run
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradients"):
        x, t = _net_inputs(case, seed)
        net = msmg.WarmStartNet(n_in=case["n_in"], hidden=(case["h1"], case["h2"]), n_vec=case["n_vec"],
                                batch_max=case["batch"], seed=seed % 1000)
        flat = net.get_params()
        flat.zero_()
        w_off, b_off = net.offsets()
        for l in range(3):
            P = _net_params(case, seed) if l == 0 else P
            flat[w_off[l]:w_off[l] + P["w%d" % l].numel()] = P["w%d" % l].reshape(-1)
            flat[b_off[l]:b_off[l] + P["b%d" % l].numel()] = P["b%d" % l]
        net.set_params(flat)
        return {"case": case, "net": net, "x": x, "t": t, "w_off": w_off, "b_off": b_off}
    if kind == "transport":
        kappa, phi, S, p, wi, q = _transport_inputs(case, seed)
        fluid = msmg.make_fluid()
        ke, w, b = msmg.msmg_impes_pressure_terms(fluid, S, kappa, wi, q, P_BH)
        # the context of the pressure solve: its grid and face coefficients are what this part uses
        sol = msmg.Solver(ke, msmg.Options(n_levels=3, block=(4, 4, 5), ratio=[_ratio(case)], n_eig=[1, 1],
                                           precision=msmg.MIXED, eig_tol=1e-8, cell_diag=w), h=_spacing(case))
        return {"case": case, "solver": sol, "fluid": fluid, "p": p, "b": b, "w": w, "q": q, "phi": phi, "S": S}
    if kind == "batched":
        sols, rhs = [], []
        for k in range(case["problems"]):
            kappa, w, f = _problem(case, seed + 1000 * k)
            sols.append(msmg.Solver(kappa, _options(case, w), h=_spacing(case), n_rhs=case["n_rhs"]))
            rhs.append(f)
        return {"case": case, "solvers": sols, "rhs": rhs, "x": [torch.zeros_like(f) for f in rhs]}
    if kind == "step":
        k0, w0, _ = _problem(case, seed + 7)
        sol = msmg.Solver(k0, _options(case, w0), h=_spacing(case))
        kappa, w, f = _problem(case, seed)
        return {"case": case, "solver": sol, "kappa": kappa, "w": w, "rhs": f}
    kappa, w, f = _problem(case, seed)
    sol = msmg.Solver(kappa, _options(case, w), h=_spacing(case), n_rhs=case["n_rhs"])
    return {"case": case, "solver": sol, "rhs": f}


def _ratio(case):
    """A ratio per direction that divides the grid of 4 x 4 x 5 elements, at most 5 each and 96 in all."""
    out = [max((r for r in (1, 2, 3, 4, 5) if m % r == 0 and m > r), default=1)
           for m in (case["nx"] // 4, case["ny"] // 4, case["nz"] // 5)]
    while out[0] * out[1] * out[2] > 96:
        out[out.index(max(out))] = 1
    return tuple(out)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "forward":
        return state["net"].forward(state["x"])
    if kind == "gradients":
        loss, g = state["net"].gradients(state["x"], state["t"])
        dims = [case["n_in"], case["h1"], case["h2"], case["n_vec"] * case["n_in"]]
        out = {"loss": loss}
        for l in range(3):
            out["w%d" % l] = g[state["w_off"][l]:state["w_off"][l] + dims[l] * dims[l + 1]].reshape(dims[l], dims[l + 1])
            out["b%d" % l] = g[state["b_off"][l]:state["b_off"][l] + dims[l + 1]]
        return out
    if kind == "transport":
        v, balance = state["solver"].velocity(state["p"], state["b"])
        S = state["S"].clone()
        dt = msmg.msmg_impes_transport(state["solver"].ctx, state["fluid"], v, state["p"], state["w"], P_BH, state["q"],
                                       state["phi"], S, M_SUB, DS_MAX)
        return {"v": v, "S": S, "dt": dt, "balance": balance[0], "source": balance[1]}
    if kind == "batched":
        msmg.msmg_solve_batched([s.ctx for s in state["solvers"]], state["rhs"], state["x"], case["rtol"], 4000)
        return state["x"]
    if kind == "step":
        state["solver"].refresh(state["kappa"], cell_diag=state["w"])
    x, _, _ = state["solver"].solve(state["rhs"], rtol=case["rtol"], max_iter=4000)
    return x


# ------------------------------------------------------------------ work
def work(case):
    kind = case["kind"]
    if kind in ("forward", "gradients"):
        B, no = case["batch"], case["n_vec"] * case["n_in"]
        w = case["n_in"] * case["h1"] + case["h1"] * case["h2"] + case["h2"] * no
        if kind == "forward":
            return {"bytes": 4.0 * B * (case["n_in"] + no) + 2.0 * w, "flops": 2.0 * B * w}
        # forward, weight gradients, and activation gradients of the two upper layers
        return {"bytes": 4.0 * B * (case["n_in"] + no) + 6.0 * w,
                "flops": 4.0 * B * w + 2.0 * B * (w - case["n_in"] * case["h1"])}
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "transport":
        # velocity: p, b, the three face coefficients in, v out; per sub-step: S in and out, v, p, w, q, phi in
        return {"bytes": 64.0 * n + M_SUB * 72.0 * n, "flops": M_SUB * 40.0 * n}
    v = 4 if case["mixed"] else 8
    # per cell and iteration and right-hand side: x, r, p read and written, q written and read, z read and written (FP64)
    # and the V-cycle's two vectors; per operator: four FP64 coefficients, four of the V-cycle's, L basis values
    it = case["iters"] * case["problems"]
    vec = 80 + 4 * v
    coef = 32 + (4 + case["L"]) * v
    one = {"bytes": float(it * n * (vec * case["n_rhs"] + coef)),
           "flops": float(it * n * case["n_rhs"] * (60 + 4 * case["L"]))}
    if kind == "step":
        nb = case["bx"] * case["by"] * case["bz"]
        nc = n // nb * case["L"]
        for _ in range(case["levels"] - 2):
            nc //= case["rx"] * case["ry"] * case["rz"]
        # set-up: the basis written, about 40 products of the element operators, the dense coarsest inverse
        one["bytes"] += float(n * (64 + 8 * case["L"])) + 16.0 * nc * nc
        one["flops"] += float(n * case["L"] * 40 * 13) + 2.0 * nc ** 3
    return one


# ------------------------------------------------------------------ exact values in 64 bits
def _faces(kappa, h):
    """Face coefficients [3] (x, y, z), each over the faces between cells."""
    k = [kappa] * 3 if kappa.dim() == 3 else list(kappa)
    out = []
    for d in range(3):
        a = k[d] / h[d] ** 2
        m = a.shape[2 - d]
        lo, hi = a.narrow(2 - d, 0, m - 1), a.narrow(2 - d, 1, m - 1)
        out.append(2.0 / (1.0 / lo + 1.0 / hi))
    return out


def _apply(T, w, x):
    """A x for a batch x [R, nz, ny, nx]."""
    q = torch.zeros_like(x) if w is None else w * x
    for d in range(3):
        dim = 3 - d
        m = x.shape[dim]
        f = T[d] * (x.narrow(dim, 1, m - 1) - x.narrow(dim, 0, m - 1))
        q.narrow(dim, 0, m - 1).sub_(f)
        q.narrow(dim, 1, m - 1).add_(f)
    return q


def _exact_solve(kappa, w, f, h, most=25000):
    """The solution of A x = f by Jacobi-preconditioned conjugate gradients in 64 bits, refined once."""
    T = _faces(kappa, h)
    f = f if f.dim() == 4 else f[None]
    dims = (1, 2, 3)
    if w is None:
        f = f - f.mean(dim=dims, keepdim=True)
    one = torch.ones((1,) + tuple(f.shape[1:]), dtype=torch.float64, device=f.device)
    diag = torch.zeros_like(one) if w is None else w[None].clone()
    for d in range(3):
        dim, m = 3 - d, one.shape[3 - d]
        diag.narrow(dim, 0, m - 1).add_(T[d])
        diag.narrow(dim, 1, m - 1).add_(T[d])
    inv = 1.0 / diag
    dot = lambda a, b: (a * b).sum(dim=dims, keepdim=True)
    x = torch.zeros_like(f)
    for _ in range(2):
        r = f - _apply(T, w, x)
        if w is None:
            r -= r.mean(dim=dims, keepdim=True)
        e = torch.zeros_like(f)
        z = inv * r
        p = z.clone()
        rz = dot(r, z)
        stop = 1e-25 * rz.clone()
        for it in range(most):
            q = _apply(T, w, p)
            al = rz / dot(p, q)
            al = torch.nan_to_num(al, 0.0, 0.0, 0.0)
            e += al * p
            r -= al * q
            z = inv * r
            new = dot(r, z)
            if it % 50 == 49 and bool((new <= stop).all()):
                break
            p = z + torch.nan_to_num(new / rz, 0.0, 0.0, 0.0) * p
            rz = new
        x = x + e
    if w is None:
        x -= x.mean(dim=dims, keepdim=True)
    return x


def _exact_net(case, seed):
    x, t = _net_inputs(case, seed)
    P = {k: v.double() for k, v in _net_params(case, seed).items()}
    W = [P["w%d" % l].float().bfloat16().double() for l in range(3)]
    bf = lambda a: a.float().bfloat16().double()           # the operands are rounded where the path rounds them
    xd = x.double()
    wgt = torch.softmax(8 * xd, dim=1).sqrt()
    xb = bf(xd)
    h1 = torch.relu(xb @ W[0] + P["b0"])
    h1b = bf(h1)
    h2 = torch.relu(h1b @ W[1] + P["b1"])
    h2b = bf(h2)
    B, nv, ni = case["batch"], case["n_vec"], case["n_in"]
    y = ((h2b @ W[2] + P["b2"]).view(B, nv, ni) * wgt[:, None, :])
    if case["kind"] == "forward":
        return y.reshape(B, nv * ni)
    td = t.double().view(B, nv, ni)
    pt = (y * td).sum(-1)
    loss = ((y * y).sum(-1) + (td * td).sum(-1) - 2 * pt.abs()).mean()
    d = 2.0 / (B * nv) * (y - torch.where(pt >= 0, 1.0, -1.0)[..., None] * td) * wgt[:, None, :]
    d = d.reshape(B, nv * ni)
    d2 = (d @ W[2].T) * (h2 > 0)
    d1 = (d2 @ W[1].T) * (h1 > 0)
    return {"loss": loss, "w0": xb.T @ d1, "b0": d1.sum(0), "w1": h1b.T @ d2, "b1": d2.sum(0), "w2": h2b.T @ d,
            "b2": d.sum(0)}


def _exact_transport(case, seed):
    kappa, phi, S, p, wi, q = _transport_inputs(case, seed)
    h = _spacing(case)

    def mobility(S):
        s = ((S - 0.2) / (1.0 - 0.2 - 0.2)).clamp(0.0, 1.0)
        mw, mo = s * s / 0.3, (1 - s) ** 2 / 3.0
        return mw + mo, mw / (mw + mo)

    lam, _ = mobility(S)
    w = wi * kappa[0] * lam
    b = q + w * P_BH
    T = _faces(kappa * lam, h)
    v = torch.zeros((3,) + tuple(S.shape), dtype=torch.float64, device=S.device)
    for d in range(3):
        dim, m = 2 - d, S.shape[2 - d]
        v[d].narrow(dim, 0, m - 1).copy_(-T[d] * h[d] * (p.narrow(dim, 1, m - 1) - p.narrow(dim, 0, m - 1)))

    def divergence(flux):
        out = torch.zeros_like(S)
        for d in range(3):
            dim, m = 2 - d, S.shape[2 - d]
            f = flux[d].narrow(dim, 0, m - 1) / h[d]
            out.narrow(dim, 0, m - 1).add_(f)
            out.narrow(dim, 1, m - 1).sub_(f)
        return out

    net = b - w * p
    balance, source = (divergence(v) - net).norm(), net.norm()
    S, total = S.clone(), 0.0
    for _ in range(M_SUB):
        _, fw = mobility(S)
        flux = torch.zeros_like(v)
        for d in range(3):
            dim, m = 2 - d, S.shape[2 - d]
            vf = v[d].narrow(dim, 0, m - 1)
            up = torch.where(vf >= 0, fw.narrow(dim, 0, m - 1), fw.narrow(dim, 1, m - 1))
            flux[d].narrow(dim, 0, m - 1).copy_(up * vf)
        rate = (q + fw * w * (P_BH - p) - divergence(flux)) / phi
        dt = DS_MAX / rate.abs().max()
        S = S + dt * rate
        total = total + dt
    return {"v": v, "S": S, "dt": total, "balance": balance, "source": source}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradients"):
        return _exact_net(case, seed)
    if kind == "transport":
        return _exact_transport(case, seed)
    h = _spacing(case)
    if kind == "batched":
        return [_exact_solve(*_problem(case, seed + 1000 * k), h) for k in range(case["problems"])]
    kappa, w, f = _problem(case, seed)
    x = _exact_solve(kappa, w, f, h)
    return x if f.dim() == 4 else x[0]
