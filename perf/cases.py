"""The library's work as its users have it done, for timing and for comparing two builds.

A case is a dict of plain values; `listed` gives the fixed ones, `draw` more of the same
ranges, `prepare` what a program holds before the call, `run` one pass through the public
entry points, `work` what the pass cannot do without, `exact` its result in plain FP64.

Four kinds of pass:

* "apply"      Y[s] = P(z_s) X[s] for a batch of systems: `ApplyPlan` (a program that applies
               the operator many times) or `apply` (a single call with host twists),
* "shifted"    the batched primal and dual shifted solves, `solve_shifted`, plain FP64 BiCG or
               complex64 BiCG with FP64 refinement,
* "solve"      the whole method for a list of energies, `solve`,
* "objective"  the ring objective and its gradient, `objective`.

The unit cells are the repository's synthetic ones: Gaussian wells at seeded centres, four
separable projectors per atom, isotropic spacing.  A program keeps its crystal and changes the
vectors: the cell follows from the case, the vector blocks from the seed.
"""
import functools
import math

import numpy as np
import torch

from paper_1709_09347_gb300 import cbs, synth


# ------------------------------------------------------------------ cases
def listed():
    return [
        # one small cell, one system, called once: launches, allocation and host work
        dict(name="apply_8x8x4_single", kind="apply", nx=8, ny=8, nz=4, h=0.4, fd=4, atoms=0,
             L=16, systems=1, dtype="c128", plan=False),
        # odd sizes, the widest stencil, an odd number of columns
        dict(name="apply_13x10x6_fd12", kind="apply", nx=13, ny=10, nz=6, h=0.4, fd=12, atoms=4,
             L=33, systems=4, dtype="c128", plan=True),
        # the FP64 BiCG iteration of the molecular-crystal cell: 16 points and their duals
        dict(name="apply_32x32x16", kind="apply", nx=32, ny=32, nz=16, h=0.35, fd=8, atoms=40,
             L=32, systems=32, dtype="c128", plan=True),
        # the largest cell of the uneven-cells workload
        dict(name="apply_96x96x20", kind="apply", nx=96, ny=96, nz=20, h=0.35, fd=8, atoms=270,
             L=24, systems=8, dtype="c128", plan=True),
        # the complex64 BiCG phase on the precision workload's cell
        dict(name="apply_64x64x24_c64", kind="apply", nx=64, ny=64, nz=24, h=0.35, fd=8, atoms=120,
             L=32, systems=32, dtype="c64", plan=True),
        # the tiny cell's whole ring at one energy
        dict(name="shifted_8x8x4", kind="shifted", nx=8, ny=8, nz=4, h=0.4, fd=4, atoms=0,
             L=16, points=32, energy=0.3, lambda_min=0.5, precision="fp64", tol=1e-12),
        # a few points of the molecular-crystal cell in plain FP64 and with refinement
        dict(name="shifted_32x32x16", kind="shifted", nx=32, ny=32, nz=16, h=0.35, fd=8, atoms=40,
             L=16, points=4, energy=-0.4, lambda_min=0.5, precision="fp64", tol=1e-12),
        dict(name="shifted_32x32x16_refine", kind="shifted", nx=32, ny=32, nz=16, h=0.35, fd=8,
             atoms=40, L=8, points=2, energy=-0.45, lambda_min=0.5, precision="fp32_refine", tol=1e-12),
        # the whole method on the tiny cell, as in the package's smoke run
        dict(name="solve_8x8x4", kind="solve", nx=8, ny=8, nz=4, h=0.4, fd=4, atoms=0, L=16, M=8,
             n_int=32, e_lo=0.3, e_hi=0.3, energies=1, lambda_min=0.5, multi_shift=0,
             extraction="hankel", tol=1e-14),
        # the whole method with one Krylov sequence for several energies
        dict(name="solve_32x32x16_family", kind="solve", nx=32, ny=32, nz=16, h=0.35, fd=8, atoms=40,
             L=16, M=8, n_int=16, e_lo=-0.1, e_hi=0.1, energies=4, lambda_min=0.5, multi_shift=1,
             extraction="rr", tol=1e-12),
        # value and gradient of the ring objective with respect to the potential
        dict(name="objective_12x10x6", kind="objective", nx=12, ny=10, nz=6, h=0.4, fd=4, atoms=3,
             L=8, M=4, n_int=16, energy=0.2, lambda_min=0.5, tol=1e-12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# grid points x columns x systems of the largest listed apply
_MOST_OUTPUTS = 96 * 96 * 20 * 24 * 8


def draw(rng):
    kind = rng.choice(("apply", "apply", "apply", "apply", "shifted", "shifted", "solve", "objective"))
    if kind == "apply":
        while True:
            fd = rng.choice((2, 4, 6, 8, 8, 8, 10, 12))
            nx, ny = _log(rng, 6, 96), _log(rng, 6, 96)
            nz = _log(rng, max(4, fd // 2), 24)
            L, systems = _log(rng, 1, 64), _log(rng, 1, 64)
            if 1000 <= nx * ny * nz * L * systems <= _MOST_OUTPUTS:
                break
        volume = nx * ny * nz * 0.35 ** 3
        atoms = rng.choice((0, 1, 1, 1)) * max(1, int(volume / 17.5))
        return dict(kind="apply", nx=nx, ny=ny, nz=nz, h=0.35, fd=fd, atoms=atoms, L=L, systems=systems,
                    dtype=rng.choice(("c128", "c64")), plan=rng.random() < 0.75)
    if kind == "solve":
        energies = rng.randint(1, 4)
        lo = round(rng.uniform(-0.1, 0.1 - 0.05 * (energies - 1)), 3)
        return dict(kind="solve", nx=32, ny=32, nz=16, h=0.35, fd=8, atoms=40, L=16, M=8, n_int=rng.choice((16, 18)),
                    e_lo=lo, e_hi=round(lo + 0.05 * (energies - 1), 3), energies=energies, lambda_min=0.5,
                    multi_shift=1 if energies > 1 else rng.randint(0, 1), extraction="rr", tol=1e-12)
    nx, ny, nz = rng.randint(6, 14), rng.randint(6, 14), rng.randint(4, 8)
    fd = rng.choice((4, 6, 8))
    atoms = rng.randint(0, 4)
    if kind == "shifted":
        return dict(kind="shifted", nx=nx, ny=ny, nz=nz, h=0.4, fd=fd, atoms=atoms, L=_log(rng, 2, 32),
                    points=rng.randint(1, 16), energy=round(rng.uniform(-0.4, 0.4), 3), lambda_min=0.5,
                    precision=rng.choice(("fp64", "fp32_refine")), tol=1e-12)
    return dict(kind="objective", nx=nx, ny=ny, nz=nz, h=0.4, fd=fd, atoms=atoms, L=_log(rng, 2, 12), M=rng.randint(2, 6),
                n_int=2 * rng.randint(4, 10), energy=round(rng.uniform(-0.4, 0.4), 3), lambda_min=0.5, tol=1e-12)


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=None)
def _cell(nx, ny, nz, h, fd, atoms):
    """Grid, local potential and projector table of a case's crystal."""
    g = synth.Grid(nx, ny, nz, h, h, h, fd)
    edge = min(g.cell)
    rng = np.random.default_rng([nx, ny, nz, fd, atoms])
    wells = max(atoms, 3)
    centres = rng.uniform(0.0, 1.0, (wells, 3)) * np.array(g.cell)
    depths = rng.uniform(-1.0, 0.0, wells)
    vloc = synth.gaussian_wells(g, centres, depths, 0.8)
    r_c = min(2.0, 0.45 * edge)
    proj = synth.make_projectors(g, centres, r_c=r_c, sigma=r_c / 4) if atoms else None
    return g, vloc, proj


def _case_cell(c):
    return _cell(c["nx"], c["ny"], c["nz"], c["h"], c["fd"], c["atoms"])


def _ring(c, n):
    """The outer circle's points: radius 1 / lambda_min, angles 2 pi (j - 1/2) / n."""
    theta = 2 * np.pi * (np.arange(n) + 0.5) / n
    return np.exp(1j * theta) / c["lambda_min"]


def _systems(c):
    """Twists and energies of an apply batch: ring points, then their duals."""
    n = c["systems"]
    half = (n + 1) // 2
    outer = 2.0 * np.exp(2j * np.pi * (np.arange(half) + 0.5) / half)
    z = np.concatenate([outer, 1.0 / np.conj(outer)])[:n]
    return z, np.linspace(-0.5, 0.5, n)


def _block(c, seed, shape, dtype):
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 7919 * c["nx"])
    return torch.randn(shape, dtype=dtype, device="cuda", generator=gen)


def _rhs(c, seed, complex_rhs):
    n = c["nx"] * c["ny"] * c["nz"]
    make = synth.random_rhs_complex if complex_rhs else synth.random_rhs
    return make(n, c["L"], int(seed))


def prepare(case, seed):
    c = case
    grid, vloc, proj = _case_cell(c)
    H = cbs.Hamiltonian(grid, vloc, proj)
    state = {"case": c, "H": H}
    if c["kind"] == "apply":
        dtype = torch.complex128 if c["dtype"] == "c128" else torch.complex64
        state["z"], state["E"] = _systems(c)
        state["X"] = _block(c, seed, (c["systems"], grid.n, c["L"]), dtype)
        if c["plan"]:
            state["plan"] = cbs.ApplyPlan(H, state["z"], state["E"], c["L"], dtype)
            state["Y"] = torch.empty_like(state["X"])
    elif c["kind"] == "shifted":
        state["z"] = _ring(c, c["points"])
        state["B"] = torch.from_numpy(_rhs(c, seed, True)).cuda()
        state["opts"] = cbs.options(tol=c["tol"], precision=c["precision"])
    elif c["kind"] == "solve":
        state["V"] = _rhs(c, seed, False)
        state["energies"] = np.linspace(c["e_lo"], c["e_hi"], c["energies"])
        state["opts"] = cbs.options(tol=c["tol"], multi_shift=c["multi_shift"], extraction=c["extraction"])
    else:
        state["V"] = _rhs(c, seed, False)
        state["opts"] = cbs.options(tol=c["tol"])
        state["grad"] = torch.empty(grid.n, dtype=torch.float64, device="cuda")
    return state


# ------------------------------------------------------------------ one pass
def _ordered(lam):
    """Order of eigenvalues by |lambda| and angle, where the moduli of a conjugate pair, equal up
    to rounding, count as equal."""
    return np.lexsort((np.angle(lam), np.round(np.abs(lam), 6)))


def _folded(c, k):
    """k of a negative real lambda lies on the zone boundary: taken at +pi / a."""
    a = c["nz"] * c["h"]
    return np.where(k.real * a < -np.pi + 1e-6, k + 2 * np.pi / a, k)


def run(state):
    c, H = state["case"], state["H"]
    if c["kind"] == "apply":
        if c["plan"]:
            return state["plan"](state["X"], state["Y"])
        return cbs.apply(H, state["z"], state["E"], state["X"])
    if c["kind"] == "shifted":
        Y, Yd, _, _ = cbs.solve_shifted(H, state["z"], c["energy"], state["B"], state["opts"])
        return {"Y": Y, "Yd": Yd}
    if c["kind"] == "solve":
        res = cbs.solve(H, state["energies"], c["lambda_min"], c["n_int"], c["L"], c["M"], state["V"],
                        state["opts"])
        out = []
        for e in res.energies:
            o = _ordered(e["lam"])
            out.append({"lam": e["lam"][o], "k": _folded(c, e["k"][o]), "mu": e["mu"]})
        return out
    J, g, gE = cbs.objective(H, c["energy"], c["lambda_min"], c["n_int"], c["L"], c["M"], state["V"],
                             state["opts"], grad=True, grad_out=state["grad"])
    return {"J": float(J), "grad_vloc": g, "grad_E": float(gE)}


# ------------------------------------------------------------------ algorithmic work
def _apply_work(c, outputs, real_bytes):
    """Of one operator apply: the vectors in and out once, the potential and the projector table
    once; per output 2 (diagonal) + 18 per half-width step + the projector terms."""
    n = c["nx"] * c["ny"] * c["nz"]
    _, _, proj = _case_cell(c)
    nnz = proj.nnz if proj is not None else 0
    return (2 * outputs * 2 * real_bytes + n * real_bytes + nnz * (4 * real_bytes + 5),
            outputs * (2 + 9 * c["fd"] + 34.0 * nnz / n))


# BiCG iterations counted for a solve: about what the listed cells take to 1e-12
_ITERS = 100


def work(case):
    c = case
    n = c["nx"] * c["ny"] * c["nz"]
    if c["kind"] == "apply":
        b, f = _apply_work(c, n * c["L"] * c["systems"], 8 if c["dtype"] == "c128" else 4)
        return {"bytes": b, "flops": f}
    if c["kind"] == "shifted":
        points, solutions = c["points"], 2
    elif c["kind"] == "solve":
        points, solutions = c["n_int"] // 2, c["energies"] * 2
    else:
        points, solutions = 2 * c["n_int"], 2
    outputs = 2 * points * n * c["L"]
    _, f = _apply_work(c, outputs, 8)
    return {"bytes": 16 * n * c["L"] * (1 + solutions * points), "flops": _ITERS * (f + 36 * outputs)}


# ------------------------------------------------------------------ results in plain FP64
def _fd_weights(order):
    """Central second-derivative weights c_0 .. c_m of the given order, unit spacing."""
    m = order // 2
    w = [0.0] * (m + 1)
    for k in range(1, m + 1):
        w[k] = 2.0 * (-1) ** (k + 1) * math.factorial(m) ** 2 / (k * k * math.factorial(m - k) * math.factorial(m + k))
    w[0] = -2.0 * sum(w[1:])
    return w


def _plain_apply(c, z, E, X):
    """P(z) X = E X - H(z) X for one block X [N, L], with shifted copies of the grid."""
    grid, vloc, proj = _case_cell(c)
    nx, ny, nz, L = grid.nx, grid.ny, grid.nz, X.shape[1]
    w = _fd_weights(c["fd"])
    x = X.reshape(nz, ny, nx, L)
    v = torch.from_numpy(vloc).to(X.device).reshape(nz, ny, nx, 1)
    y = (E - v) * x + 0.5 * 3 * w[0] / c["h"] ** 2 * x
    for k in range(1, len(w)):
        s = torch.roll(x, k, 2) + torch.roll(x, -k, 2) + torch.roll(x, k, 1) + torch.roll(x, -k, 1)
        up, down = torch.roll(x, -k, 0).clone(), torch.roll(x, k, 0).clone()
        up[nz - k:] *= z                      # neighbours in the next cell
        down[:k] /= z                         # and in the one before
        y = y + 0.5 * w[k] / c["h"] ** 2 * (s + up + down)
    y = y.reshape(-1, L)
    if proj is not None:
        idx = torch.from_numpy(proj.sup_idx.astype(np.int64)).to(X.device)
        wrap = torch.from_numpy(proj.sup_wrap.astype(np.int64)).to(X.device)
        atom = torch.from_numpy(np.repeat(np.arange(proj.n_atoms), np.diff(proj.sup_ptr))).to(X.device)
        p = torch.from_numpy(proj.sup_val).to(X.device)
        h = torch.from_numpy(proj.h).to(X.device).to(X.dtype)
        images = torch.tensor([1.0 / z, 1.0, z], dtype=X.dtype, device=X.device)   # z^m at m = -1, 0, 1
        gathered = X[idx] * images[1 - wrap][:, None]
        coef = torch.zeros((proj.n_atoms, proj.n_proj, L), dtype=X.dtype, device=X.device)
        for mu in range(proj.n_proj):
            part = torch.view_as_real(gathered * p[:, mu:mu + 1]).contiguous()
            acc = torch.zeros((proj.n_atoms, L, 2), dtype=torch.float64, device=X.device)
            coef[:, mu] = torch.view_as_complex(acc.index_add_(0, atom, part))
        D = h @ coef
        back = sum(p[:, mu:mu + 1] * D[atom, mu] for mu in range(proj.n_proj)) * images[1 + wrap][:, None]
        out = torch.view_as_real(y).contiguous()
        out.index_add_(0, idx, -torch.view_as_real(back).contiguous())
        y = torch.view_as_complex(out)
    return y


def _dense(c, z, E):
    n = c["nx"] * c["ny"] * c["nz"]
    return _plain_apply(c, z, E, torch.eye(n, dtype=torch.complex128, device="cuda"))


def _ring_solutions(c, E, z, B):
    """Solutions at the outer-circle points z and their duals, P(z)^dagger = P(1 / conj z)."""
    P = [_dense(c, zz, E) for zz in z]
    return ([torch.linalg.solve(p, B) for p in P], [torch.linalg.solve(p.conj().T, B) for p in P], P)


def _exact_solve(c, E, V):
    n, n_int, M = V.shape[0], c["n_int"], c["M"]
    z1 = _ring(c, n_int)
    Y1, Y2, _ = _ring_solutions(c, E, z1, V)
    z2 = 1.0 / np.conj(z1)
    mu = torch.zeros((2 * M, c["L"], c["L"]), dtype=torch.complex128, device="cuda")
    for j in range(n_int):
        G1, G2 = V.conj().T @ Y1[j], V.conj().T @ Y2[j]
        for k in range(2 * M):
            mu[k] += complex(z1[j] ** (k + 1) / n_int) * G1 - complex(z2[j] ** (k + 1) / n_int) * G2
    # -z P(z) = z^2 H+ + z (H0 - E) + H-: the blocks from three twists, then the eigenvalues
    # through z = s + 1 / mu, which turns them into those of a monic quadratic
    a, b, d = -_dense(c, 1.0, E), -_dense(c, -1.0, E), -_dense(c, 1j, E)
    A1 = (a + b) / 2
    plus, minus = (a - b) / 2, (d - A1) / 1j
    A2, A0 = (plus + minus) / 2, (plus - minus) / 2
    s = 0.7 * np.exp(2.4j)
    inv = torch.linalg.inv(A2 * s * s + A1 * s + A0)
    top = torch.cat([-(inv @ (2 * s * A2 + A1)), -(inv @ A2)], 1)
    eye = torch.eye(n, dtype=torch.complex128, device="cuda")
    comp = torch.cat([top, torch.cat([eye, torch.zeros_like(eye)], 1)], 0)
    m = np.linalg.eigvals(comp.cpu().numpy())
    lam = s + 1.0 / m[np.abs(m) > 1e-8]
    lam = lam[(np.abs(lam) > c["lambda_min"]) & (np.abs(lam) < 1 / c["lambda_min"])]
    lam = lam[_ordered(lam)]
    k = (np.angle(lam) - 1j * np.log(np.abs(lam))) / (c["nz"] * c["h"])
    return {"lam": lam, "k": _folded(c, k), "mu": mu}


def _exact_objective(c, E, V):
    n_int, M = c["n_int"], c["M"]
    z1 = _ring(c, n_int)
    z2 = 1.0 / np.conj(z1)
    Y1, Y2, P = _ring_solutions(c, E, z1, V)
    J, gE = 0.0, 0.0
    gV = torch.zeros(V.shape[0], dtype=torch.float64, device="cuda")
    for j in range(n_int):
        c1 = float(np.sum(z1[j] ** np.arange(1, M + 1)).real) / n_int
        c2 = -float(np.sum(z2[j] ** np.arange(1, M + 1)).real) / n_int
        G1, G2 = torch.linalg.solve(P[j].conj().T, Y1[j]), torch.linalg.solve(P[j], Y2[j])
        J += float(c1 * Y1[j].abs().square().sum() + c2 * Y2[j].abs().square().sum())
        g = 2 * (c1 * (G1.conj() * Y1[j]).real.sum(1) + c2 * (G2.conj() * Y2[j]).real.sum(1))
        gV += g
        gE -= float(g.sum())
    return {"J": J, "grad_vloc": gV, "grad_E": gE}


def exact(case, seed):
    c = case
    n = c["nx"] * c["ny"] * c["nz"]
    if c["kind"] == "apply":
        dtype = torch.complex128 if c["dtype"] == "c128" else torch.complex64
        X = _block(c, seed, (c["systems"], n, c["L"]), dtype)
        z, E = _systems(c)
        return torch.stack([_plain_apply(c, complex(zz), float(e), X[s].to(torch.complex128))
                            for s, (zz, e) in enumerate(zip(z, E))])
    if n > 1600:                       # dense solves of larger cells take too long
        return None
    if c["kind"] == "shifted":
        B = torch.from_numpy(_rhs(c, seed, True)).cuda()
        Y, Yd, _ = _ring_solutions(c, c["energy"], _ring(c, c["points"]), B)
        return {"Y": torch.stack(Y), "Yd": torch.stack(Yd)}
    V = torch.from_numpy(_rhs(c, seed, False)).cuda()
    if c["kind"] == "solve":
        return [_exact_solve(c, float(E), V) for E in np.linspace(c["e_lo"], c["e_hi"], c["energies"])]
    return _exact_objective(c, c["energy"], V)
