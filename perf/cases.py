"""The work that programs using this framework have it do, as cases that can be prepared, run and
checked: H psi, the preconditioner, Gram matrices, Ritz rotations, the subspace solve of Eq. 1,
LOBPCG and the SCF step, in the FP64 form, the mixed form (FP32 data path, split-BF16 tensor-core
products) and the real Gamma-point form.

A case is a dict: "kind" says which call, (nx, ny, nz) the grid, "bands" the orbitals, "reps" the
diamond supercell (8 reps^3 atoms with seeded thermal displacements), h the grid spacing in bohr.
`draw` covers the same kinds over the grids, band counts and subspace sizes of the repository's
workloads: 5-smooth grids of 20 to 96 points per axis, odd and unequal ones among them, 8 to 160
orbitals and subspaces of 24 to 480.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2512_04447_gb300 import rsdft

SMOOTH = (20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 90, 96)
RC, RCUT, Z, SIGMA = 1.0, 3.0, 4.0, 0.6   # pseudo-atoms of the workloads


def _case(kind, grid, **kw):
    nx, ny, nz = grid if isinstance(grid, tuple) else (grid,) * 3
    return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "h": 0.21, **kw}


def listed():
    return [
        # H psi of the 8-atom cell of the fixed-potential runs: the smallest call, launches and latency
        _case("hpsi", 24, h=10.0 / 24, bands=16, reps=1, fp32=False, name="hpsi_24_fp64"),
        # H psi of the 64-atom SCF cell, every orbital at once, in the FP64 form
        _case("hpsi", 64, bands=144, reps=2, fp32=False, name="hpsi_64_fp64"),
        # H psi of the mixed form's FP32 data path on the 216-atom cell, a third of its orbitals
        _case("hpsi", 96, bands=160, reps=3, fp32=True, name="hpsi_96_fp32"),
        # preconditioner of one of the uneven cells of a batch: odd grid, odd number of residuals
        _case("tpa", 45, bands=53, name="tpa_45_fp64"),
        # subspace matrix <Y|HY> of the 64-atom cell, Y = [X W P] of 3 x 144 rows, FP64 form
        _case("gram", 64, rows=432, cols=432, real=False, name="gram_64_fp64"),
        # Ritz rotation of the same block, 432 rows to 144 orbitals, FP64 form
        _case("rotate", 64, rows=432, bands=144, real=False, base=False, name="rotate_64_fp64"),
        # subspace matrix of the real Gamma-point form, odd band count on a 60^3 metal-cell grid
        _case("gram", 60, rows=285, cols=285, real=True, name="gram_60_real"),
        # G_S and G_H of the mixed form, split-BF16 on the tensor cores
        _case("gram_pair_tc", 64, rows=432, name="gram_pair_64_tc"),
        # Ritz rotation of the mixed form on the tensor cores: new X and new P
        _case("rotate_tc", 64, rows=432, bands=144, name="rotate_64_tc"),
        # generalised eigenproblem of Eq. 1 as the mixed form solves it at 3 x 144
        _case("ritz", 20, rows=432, bands=144, double_float=True, name="ritz_432_df"),
        # a whole FP64 solve of a fixed number of iterations from a random start block
        _case("lobpcg", 48, bands=72, reps=1, iterations=3, real=False, name="lobpcg_48_fp64"),
        # one SCF step of the headline cell and form: potential, 3 LOBPCG iterations, density, mixing
        _case("scf", 64, bands=144, reps=2, name="scf_64_mixed"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi, most):
    """A 5-smooth grid of lo..hi points per axis (half of them cubic) and at most `most` points."""
    axis = [v for v in SMOOTH if lo <= v <= hi]
    while True:
        g = (rng.choice(axis),) * 3 if rng.random() < 0.5 else tuple(rng.choice(axis) for _ in range(3))
        if g[0] * g[1] * g[2] <= most:
            return g


def draw(rng):
    kind = rng.choice(["hpsi", "hpsi", "tpa", "gram", "gram", "rotate", "rotate", "gram_pair_tc", "rotate_tc", "ritz",
                       "lobpcg", "scf"])
    if kind == "hpsi":
        g = _grid(rng, 30, 96, 96 ** 3)
        reps = max(1, min(3, round(min(g) * 0.21 / 6.74)))
        most = 160 * 96 ** 3 // (2 * g[0] * g[1] * g[2])
        return _case(kind, g, bands=_log(rng, 8, max(16, min(160, most))), reps=reps, fp32=rng.random() < 0.5)
    if kind == "tpa":
        g = _grid(rng, 20, 80, 64 ** 3)
        return _case(kind, g, bands=_log(rng, 8, 144))
    if kind in ("gram", "rotate"):
        g = _grid(rng, 20, 64, 64 ** 3)
        k = _log(rng, 24, 432)
        real = rng.random() < 0.4
        if kind == "gram":
            cols = k if rng.random() < 0.5 else _log(rng, 24, 432)
            return _case(kind, g, rows=k, cols=cols, real=real)
        return _case(kind, g, rows=k, bands=max(8, k // 3), real=real, base=rng.random() < 0.3)
    if kind == "gram_pair_tc":
        return _case(kind, _grid(rng, 24, 64, 64 ** 3), rows=_log(rng, 48, 480))
    if kind == "rotate_tc":
        k = _log(rng, 48, 480)
        return _case(kind, _grid(rng, 24, 64, 64 ** 3), rows=k, bands=max(16, k // 3))
    if kind == "ritz":
        k = _log(rng, 48, 440)
        return _case(kind, 20, rows=k, bands=max(16, k // 3), double_float=rng.random() < 0.5)
    if kind == "lobpcg":
        return _case(kind, _grid(rng, 32, 48, 48 ** 3), bands=_log(rng, 16, 72), reps=1, iterations=rng.choice([2, 3]),
                     real=rng.random() < 0.5)
    return _case(kind, _grid(rng, 32, 60, 60 ** 3), bands=_log(rng, 24, 72), reps=1)


# ---- what a program has in hand ---------------------------------------------------------------

def _shape(c):
    return c["nz"], c["ny"], c["nx"]


def _edges(c):
    return tuple(c["h"] * c[a] for a in ("nx", "ny", "nz"))


def _n(c):
    return c["nx"] * c["ny"] * c["nz"]


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + stream)
    return g


def _atoms(c, seed):
    """Diamond-cubic sites of reps^3 cells stretched over the box, displaced by about 0.05 bohr as in a
    run at temperature, and the Kleinman-Bylander energies."""
    reps, rng = c["reps"], np.random.default_rng([int(seed), 17])
    fcc = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
    basis = np.concatenate([fcc, fcc + 0.25])
    cells = np.array([[i, j, k] for i in range(reps) for j in range(reps) for k in range(reps)], float)
    pos = (cells[:, None] + basis[None]).reshape(-1, 3) / reps * np.array(_edges(c))
    pos += rng.normal(0.0, 0.05, pos.shape)
    return np.ascontiguousarray(pos), rng.uniform(0.5, 2.0, (len(pos), 4))


def _displacements(c, pos):
    """Minimal-image displacements from each atom along each axis: three tensors [atom][points]."""
    out = []
    for a, key in enumerate(("nx", "ny", "nz")):
        L = _edges(c)[a]
        d = torch.arange(c[key], device="cuda", dtype=torch.float64) * (L / c[key]) - torch.from_numpy(pos[:, a:a + 1]).cuda()
        out.append(d - L * torch.floor(d / L + 0.5))
    return out


def _vloc(c, pos):
    """Local potential [n]: minus Z times a Gaussian about every atom."""
    ex, ey, ez = (torch.exp(-d * d / (2 * SIGMA * SIGMA)) for d in _displacements(c, pos))
    return -Z * torch.einsum("az,ay,ax->zyx", ez, ey, ex).reshape(-1)


def _context(c, seed, atoms):
    if not atoms:
        return rsdft.Context(_edges(c), (c["nx"], c["ny"], c["nz"]), np.zeros(_n(c)))
    pos, e_kb = _atoms(c, seed)
    rcut = min(RCUT, 0.49 * min(_edges(c)))
    return rsdft.Context(_edges(c), (c["nx"], c["ny"], c["nz"]), _vloc(c, pos).cpu().numpy(), pos, RC, rcut, e_kb, 4)


def _bump(c):
    """A smooth positive function of the grid with a maximum at every site of a 2x2x2 lattice."""
    ax = [0.5 + 0.5 * torch.cos(4 * math.pi * torch.arange(c[k], device="cuda", dtype=torch.float64) / c[k])
          for k in ("nx", "ny", "nz")]
    return 0.25 + torch.einsum("z,y,x->zyx", *[a * a for a in reversed(ax)])


def _orbitals(c, rows, seed, stream, real=False, dtype=torch.complex128):
    """Rows like the basis of an iteration: smooth, larger near the atoms, unit norm, the later rows
    (preconditioned residuals, directions) with more of the short wavelengths."""
    g, shape = _gen(seed, stream), _shape(c)
    k2 = sum(k * k for k in torch.meshgrid(*[torch.fft.fftfreq(s, 1.0 / s, device="cuda", dtype=torch.float64)
                                             for s in shape], indexing="ij"))
    bump, dv = _bump(c), float(np.prod(_edges(c))) / _n(c)
    out = torch.empty(rows, _n(c), device="cuda", dtype=torch.float64 if real else dtype)
    step = max(1, (1 << 24) // _n(c))
    for r in range(0, rows, step):
        m = min(step, rows - r)
        cut = 6.0 + 20.0 * (torch.arange(r, r + m, device="cuda", dtype=torch.float64) / rows).view(-1, 1, 1, 1)
        z = torch.randn((m, *shape), device="cuda", dtype=torch.complex128, generator=g) / (1.0 + k2 / (cut * cut)) ** 1.5
        z = torch.fft.ifftn(z, dim=(1, 2, 3)) * bump
        z = (z.real if real else z).reshape(m, -1)
        out[r:r + m] = (z / (torch.linalg.vector_norm(z, dim=1, keepdim=True) * math.sqrt(dv))).to(out.dtype)
    return out


def _coefficients(c, seed, real=False):
    """Ritz coefficients [rows][bands]: the lowest vectors are mostly their own old row."""
    k, m = c["rows"], c["bands"]
    z = torch.randn((k, m), device="cuda", dtype=torch.float64 if real else torch.complex128, generator=_gen(seed, 5))
    z = z * (0.3 / math.sqrt(k))
    z[:m] += torch.eye(m, device="cuda", dtype=z.dtype)
    return z.contiguous()


def _subspace_pair(c, seed):
    """G_S and G_H of a basis [X W P]: X orthonormal, W and P normalised and overlapping."""
    k, m, g = c["rows"], c["bands"], _gen(seed, 6)
    r = torch.randn((k, k), device="cuda", dtype=torch.complex128, generator=g)
    over = 0.25 * (r + r.conj().T) / math.sqrt(4 * k)
    over[:m, :m] = 0
    over.fill_diagonal_(0)
    gs = torch.eye(k, device="cuda", dtype=torch.complex128) + over
    e = torch.sort(torch.rand(k, device="cuda", dtype=torch.float64, generator=g) ** 2 * 40.0 - 1.0).values
    r = torch.randn((k, k), device="cuda", dtype=torch.complex128, generator=g)
    gh = torch.diag(e).to(torch.complex128) + 0.5 * (r + r.conj().T) / math.sqrt(k)
    return gh.contiguous(), gs.contiguous()


def _t(c, seed):
    return 0.5 + 4.0 * torch.rand(c["bands"], device="cuda", dtype=torch.float64, generator=_gen(seed, 7))


def _start_block(c, seed):
    return torch.randn((c["bands"], _n(c)), device="cuda", dtype=torch.float64 if c["real"] else torch.complex128,
                       generator=_gen(seed, 8))


def _scf_options(c):
    # the headline form: FP32 data path, tensor-core Grams and rotations, aufbau over eight ninths of the bands
    return rsdft.Context.scf_opts(n_electrons=2.0 * (c["bands"] * 8 // 9), precision=rsdft.MIXED, tensor_cores=2)


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c, "ctx": _context(c, seed, kind in ("hpsi", "lobpcg", "scf"))}
    if kind == "hpsi":
        s["x"] = _orbitals(c, c["bands"], seed, 1, dtype=torch.complex64 if c["fp32"] else torch.complex128)
        s["out"] = torch.empty_like(s["x"])
    elif kind == "tpa":
        s["x"], s["t"] = _orbitals(c, c["bands"], seed, 1), _t(c, seed)
        s["out"] = torch.empty_like(s["x"])
    elif kind == "gram":
        s["a"], s["b"] = (_orbitals(c, c[k], seed, i, c["real"]) for i, k in ((1, "rows"), (2, "cols")))
        s["out"] = torch.empty(c["rows"], c["cols"], device="cuda", dtype=s["a"].dtype)
    elif kind == "rotate":
        s["y"], s["c"] = _orbitals(c, c["rows"], seed, 1, c["real"]), _coefficients(c, seed, c["real"])
        s["base"] = _orbitals(c, c["bands"], seed, 2, c["real"]) if c["base"] else None
        s["out"] = torch.empty(c["bands"], _n(c), device="cuda", dtype=s["y"].dtype)
    elif kind == "gram_pair_tc":
        s["y"] = _orbitals(c, c["rows"], seed, 1, dtype=torch.complex64)
        s["hy"] = s["y"] * (4.0 * _bump(c).reshape(-1)).to(torch.float32)
        s["gs"], s["gh"] = (torch.empty(c["rows"], c["rows"], device="cuda", dtype=torch.complex128) for _ in range(2))
    elif kind == "rotate_tc":
        s["y"], s["c"] = _orbitals(c, c["rows"], seed, 1, dtype=torch.complex64), _coefficients(c, seed)
        s["x"], s["p"] = (torch.empty(c["bands"], _n(c), device="cuda", dtype=torch.complex64) for _ in range(2))
    elif kind == "ritz":
        s["gh"], s["gs"] = _subspace_pair(c, seed)
        s["z"] = torch.empty(c["rows"], c["bands"], device="cuda", dtype=torch.complex128)
        s["ctx"].set_dense(rsdft.DENSE_DF if c["double_float"] else rsdft.DENSE_FP64)
    elif kind == "lobpcg":
        s["x0"] = _start_block(c, seed)
        s["x"] = torch.empty_like(s["x0"])
        s["opts"] = s["ctx"].lobpcg_opts(maxit=c["iterations"], tol=0.0)
    else:
        # an SCF run past its first, converged step; each pass is the next step of it
        s["x"] = _start_block({**c, "real": False}, seed)
        s["opts"] = _scf_options(c)
        s["ctx"].scf_init(c["bands"], s["opts"])
        s["ctx"].scf_step(s["x"], s["opts"])
    return s


class _Field:
    """A float64 field of the context, for torch."""

    def __init__(self, ptr, n):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<f8", "data": (ptr, False), "version": 2}


def run(state):
    s, c, ctx = state, state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "hpsi":
        ctx.apply_h(s["x"], s["out"], rsdft.MIXED if c["fp32"] else rsdft.FP64)
        return s["out"]
    if kind == "tpa":
        ctx.precondition_tpa(s["x"], s["out"], s["t"])
        return s["out"]
    if kind == "gram":
        (ctx.gram_real if c["real"] else ctx.gram)(s["a"], s["b"], s["out"])
        return s["out"]
    if kind == "rotate":
        (ctx.rotate_real if c["real"] else ctx.rotate)(s["y"], s["c"], s["out"], s["base"], -1 if c["base"] else 1)
        return s["out"]
    if kind == "gram_pair_tc":
        ctx.gram_sh_bf16x3(s["y"], s["hy"], s["gs"], s["gh"])
        # products of split FP32 values: the results carry FP32 accuracy and go by that type
        return {"gs": s["gs"].to(torch.complex64), "gh": s["gh"].to(torch.complex64)}
    if kind == "rotate_tc":
        ctx.rotate_bf16x3(s["y"], s["c"], s["x"], s["p"])
        return {"x": s["x"], "p": s["p"]}
    if kind == "ritz":
        lam, _ = ctx.rayleigh_ritz(s["gh"], s["gs"], c["bands"], s["z"], pivot_tol=1e-3)
        # an eigenvector's phase is free: the weight of each basis row in each vector
        return {"lam": lam, "weight": s["z"].real.square() + s["z"].imag.square()}
    if kind == "lobpcg":
        s["x"].copy_(s["x0"])
        eig, res, _, _ = (ctx.lobpcg_real if c["real"] else ctx.lobpcg)(s["x"], s["opts"])
        x = s["x"]
        # the orbitals without their free phases: the charge of each
        return {"eig": eig, "res": res, "charge": x.square() if c["real"] else x.real.square() + x.imag.square()}
    out, eig, occ = ctx.scf_step(s["x"], s["opts"])
    # FP32 iterations: the results go by that type; the next step's density stands for the orbitals, whose
    # phases and rotations within near-degenerate groups are free
    rho = torch.as_tensor(_Field(ctx.scf_density_ptr(), _n(c)), device="cuda").to(torch.float32)
    return {"eig": eig.astype(np.float32), "occ": occ.astype(np.float32), "e_tot": np.float32(out.e_tot), "rho": rho}


# ---- what a pass cannot do without --------------------------------------------------------------

def _h_flops(c, complex_bands):
    """Two 3D transforms, the potential, and (atoms) four projectors per sphere point, gathered and scattered."""
    n = _n(c)
    inside = 8 * c["reps"] ** 3 * 4.0 / 3.0 * math.pi * (min(RCUT, 0.49 * min(_edges(c))) / c["h"]) ** 3
    return complex_bands * (10.0 * n * math.log2(n) + 10.0 * n + 32.0 * inside)


def work(case):
    c, kind, n = case, case["kind"], _n(case)
    if kind == "hpsi":
        e = 8 if c["fp32"] else 16
        return {"bytes": 2.0 * e * n * c["bands"] + e / 2 * n, "flops": _h_flops(c, c["bands"])}
    if kind == "tpa":
        return {"bytes": 32.0 * n * c["bands"], "flops": c["bands"] * n * (10.0 * math.log2(n) + 20.0)}
    if kind == "gram":
        e, f = (8, 2) if c["real"] else (16, 8)
        return {"bytes": e * (float(n) * (c["rows"] + c["cols"]) + c["rows"] * c["cols"]),
                "flops": f * float(n) * c["rows"] * c["cols"]}
    if kind == "rotate":
        e, f = (8, 2) if c["real"] else (16, 8)
        return {"bytes": e * float(n) * (c["rows"] + c["bands"] * (2 if c["base"] else 1)),
                "flops": f * float(n) * c["rows"] * c["bands"]}
    if kind == "gram_pair_tc":
        k = c["rows"]
        return {"bytes": 16.0 * n * k, "flops": 8.0 * n * k * (k + 1)}   # two Hermitian matrices
    if kind == "rotate_tc":
        return {"bytes": 8.0 * n * (c["rows"] + 2 * c["bands"]), "flops": 8.0 * n * c["rows"] * c["bands"]}
    k, m = c.get("rows", 3 * c["bands"]), c["bands"]
    dense = 4.0 / 3.0 * k ** 3 + 8.0 * k ** 3 + 16.0 / 3.0 * k ** 3 + 12.0 * k * k * m
    if kind == "ritz":
        return {"bytes": 16.0 * (2 * k * k + k * m), "flops": dense}
    # one iteration: H W, the preconditioner, the two Gram matrices, four rotations (X, P, HX, HP) as two
    real = bool(c.get("real"))
    its, f = (c["iterations"], 2 if real else 8) if kind == "lobpcg" else (3, 8)
    e = (8 if real else 16) if kind == "lobpcg" else 8
    step = (_h_flops(c, m / 2 if real else m) + m * n * 10.0 * math.log2(n)
            + f * n * (m * m * 2.0 + k * (k + 1.0) + 2.0 * k * m) + dense)
    return {"bytes": its * e * n * 6.0 * m, "flops": its * step}


# ---- the same in plain 64-bit torch --------------------------------------------------------------

def _hamiltonian(c, seed):
    """x -> H x on rows [m][n], in 64 bits."""
    pos, e_kb = _atoms(c, seed)
    dx, dy, dz = _displacements(c, pos)
    dv = float(np.prod(_edges(c))) / _n(c)
    v, rcut = _vloc(c, pos), min(RCUT, 0.49 * min(_edges(c)))
    beta = []
    for a in range(len(pos)):
        x, y, z = dx[a].view(1, 1, -1), dy[a].view(1, -1, 1), dz[a].view(-1, 1, 1)
        d2 = x * x + y * y + z * z
        g = torch.where(d2 < rcut * rcut, torch.exp(-d2 / (2 * RC * RC)), torch.zeros((), device="cuda", dtype=torch.float64))
        b = torch.stack([t.expand_as(g).reshape(-1) for t in (g, x / RC * g, y / RC * g, z / RC * g)])
        beta.append(b / torch.linalg.vector_norm(b, dim=1, keepdim=True) / math.sqrt(dv))
    beta, e = torch.cat(beta), torch.from_numpy(e_kb).cuda().reshape(-1, 1)
    g2 = _g2(c)

    def apply(x):
        kin = _filter(c, x, 0.5 * g2)
        parts = [x] if not x.is_complex() else [x.real.contiguous(), x.imag.contiguous()]
        nl = [(e * (beta @ p.T * dv)).T @ beta for p in parts]
        return kin + v * x + (nl[0] if not x.is_complex() else torch.complex(nl[0], nl[1]))

    return apply, v, beta, e, dv


def _g2(c):
    ax = [2 * math.pi / L * torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
          for L, n in zip(reversed(_edges(c)), _shape(c))]
    return sum(k * k for k in torch.meshgrid(*ax, indexing="ij"))


def _filter(c, x, f):
    """Rows x with their spectrum times f, a few rows at a time; f: [nz][ny][nx] or one of it per row."""
    out, step = torch.empty_like(x), max(1, (1 << 25) // _n(c))
    for r in range(0, x.shape[0], step):
        y = torch.fft.ifftn(torch.fft.fftn(x[r:r + step].reshape(-1, *_shape(c)), dim=(1, 2, 3))
                            * (f[r:r + step] if f.dim() == 4 else f), dim=(1, 2, 3)).reshape(-1, _n(c))
        out[r:r + step] = y if x.is_complex() else y.real
    return out


def _tpa(c, r, t):
    g2, out = _g2(c), torch.empty_like(r)
    for b in range(r.shape[0]):
        x = 0.5 * g2 / t[b]
        p = 27 + 18 * x + 12 * x ** 2 + 8 * x ** 3
        out[b:b + 1] = _filter(c, r[b:b + 1], p / (p + 16 * x ** 4))
    return out


def _dot(a, b):
    """conj(a) b^T, the long sum in pieces that are added at the end."""
    n, step = a.shape[1], 4096
    parts = [a[:, i:i + step].conj() @ b[:, i:i + step].T for i in range(0, n, step)]
    while len(parts) > 1:
        parts = [sum(parts[i:i + 2]) for i in range(0, len(parts), 2)]
    return parts[0]


def _solve_pencil(gh, gs):
    low = torch.linalg.cholesky(gs)
    k = torch.linalg.solve_triangular(low, gh, upper=False)
    k = torch.linalg.solve_triangular(low, k.mH.contiguous(), upper=False)
    lam, z = torch.linalg.eigh(0.5 * (k + k.mH))
    return lam, torch.linalg.solve_triangular(low.mH, z, upper=True)


def _lobpcg(c, seed):
    """The iteration of the solver: preconditioned residuals off X, Rayleigh-Ritz over [X W P]."""
    h, v, beta, e, dv = _hamiltonian(c, seed)
    x = _start_block(c, seed)
    m = x.shape[0]

    def herm(a, b):
        g = _dot(a, b) * dv
        return 0.5 * (g + g.mH)

    hx = h(x)
    lam, z = _solve_pencil(herm(x, hx), herm(x, x))
    x, hx, p = z.T @ x, z.T @ hx, None
    for _ in range(c["iterations"]):
        proj = _dot(beta.to(x.dtype), x) * dv
        t = lam - dv * (v * x.abs().square()).sum(1) - (e * proj.abs().square()).sum(0)
        w = _tpa(c, hx - lam.view(-1, 1) * x, t)
        w = w - (_dot(x, w) * dv).T @ x
        w = w / (torch.linalg.vector_norm(w, dim=1, keepdim=True) * math.sqrt(dv))
        y, hy = [x, w], [hx, h(w)]
        if p is not None:
            s = torch.linalg.vector_norm(p, dim=1, keepdim=True) * math.sqrt(dv)
            y, hy = y + [p / s], hy + [hp / s]
        y, hy = torch.cat(y), torch.cat(hy)
        lam, z = _solve_pencil(herm(y, hy), herm(y, y))
        lam, z = lam[:m], z[:, :m]
        p, hp = z[m:].T @ y[m:], z[m:].T @ hy[m:]
        x, hx = z[:m].T @ x + p, z[:m].T @ hx + hp
    res = torch.linalg.vector_norm(hx - lam.view(-1, 1) * x, dim=1) * math.sqrt(dv)
    return {"eig": lam, "res": res, "charge": x.abs().square()}


def exact(case, seed):
    c, kind = case, case["kind"]
    dv = float(np.prod(_edges(c))) / _n(c)
    if kind == "hpsi":
        x = _orbitals(c, c["bands"], seed, 1, dtype=torch.complex64 if c["fp32"] else torch.complex128)
        return _hamiltonian(c, seed)[0](x.to(torch.complex128))
    if kind == "tpa":
        return _tpa(c, _orbitals(c, c["bands"], seed, 1), _t(c, seed))
    if kind == "gram":
        a, b = (_orbitals(c, c[k], seed, i, c["real"]) for i, k in ((1, "rows"), (2, "cols")))
        return _dot(a, b) * dv
    if kind == "rotate":
        y, z = _orbitals(c, c["rows"], seed, 1, c["real"]), _coefficients(c, seed, c["real"])
        return _orbitals(c, c["bands"], seed, 2, c["real"]) - z.T @ y if c["base"] else z.T @ y
    if kind == "gram_pair_tc":
        y = _orbitals(c, c["rows"], seed, 1, dtype=torch.complex64)
        hy = y * (4.0 * _bump(c).reshape(-1)).to(torch.float32)
        y, hy = y.to(torch.complex128), hy.to(torch.complex128)
        return {"gs": _dot(y, y) * dv, "gh": _dot(y, hy) * dv}
    if kind == "rotate_tc":
        y, z = _orbitals(c, c["rows"], seed, 1, dtype=torch.complex64).to(torch.complex128), _coefficients(c, seed)
        p = z[c["bands"]:].T @ y[c["bands"]:]
        return {"x": z[:c["bands"]].T @ y[:c["bands"]] + p, "p": p}
    if kind == "ritz":
        lam, z = _solve_pencil(*_subspace_pair(c, seed))
        return {"lam": lam[:c["bands"]], "weight": z[:, :c["bands"]].abs().square()}
    if kind == "lobpcg":
        return _lobpcg(c, seed)
    return None   # a step of a running SCF: its inputs are the run's own, to FP32 accuracy
