"""What the speed of this library is measured on: calls of its public Python
entry points as an ensemble study, a solver of one's own or an adjoint run
issues them, from one 32 x 32 realization to batches of 512 x 512 and two of
2048 x 2048, plus the 3D form.

``listed()`` gives the fixed cases, ``draw(rng)`` further ones of the same
ranges; ``prepare`` makes what a program holds before the call, ``run`` is one
call, ``work`` the bytes and operations the call cannot do without, and
``exact`` the result in 64 bits by plain torch and numpy (its own field
generator, roll-based stencils and FFT-preconditioned CG).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1903_12227_gb300 import rve, rve3, studies, workloads

FP64, MIXED = "fp64", "mixed"


# -------------------------------------------------------------------- cases --
def listed() -> list:
    return [
        # one small realization in double precision: a call dominated by latency
        _ensemble("single_32_fp64", 4, 8, 1, 10.0, FP64, 1e-12),
        # the ensemble throughput workload, 512 x 512, mixed precision, an odd batch
        _ensemble("ensemble_512_mixed", 32, 16, 125, 10.0, MIXED, 1e-10),
        # large cells at high contrast (variance study), few realizations at a time
        _ensemble("large_2048_mixed", 256, 8, 2, 100.0, MIXED, 1e-10),
        # uneven sizes and contrasts in one captured plan
        {"name": "uneven_plan_mixed", "kind": "plan", "batch": 250, "precision": MIXED, "tol": 1e-10},
        # the paper's statistics: many small cells, lumped scheme, low contrast
        {"name": "paper_64_lumped", "kind": "study", "L": 16, "batch": 1500, "precision": MIXED,
         "tol": 1e-8},
        # A_hom and its gradient per cell in double precision (forward and backward)
        {"name": "adjoint_1024_fp64", "kind": "adjoint", "L": 64, "m0": 16, "batch": 1,
         "contrast": 100.0, "tol": 1e-13, "scheme": "consistent"},
        # nodal load through the mass matrix, double-precision solve of a given right-hand side
        {"name": "fem_load_512_fp64", "kind": "fem", "L": 8, "m0": 64, "batch": 3, "contrast": 10.0,
         "tol": 1e-10, "scheme": "consistent"},
        # operator and preconditioner applications, the building blocks of a solver of one's own
        {"name": "stiffness_512_fp32", "kind": "stiffness", "L": 32, "m0": 16, "batch": 96,
         "contrast": 10.0, "precision": MIXED, "scheme": "consistent", "coef": False},
        {"name": "stiffness_1024_fp64_coef", "kind": "stiffness", "L": 64, "m0": 16, "batch": 11,
         "contrast": 100.0, "precision": FP64, "scheme": "consistent", "coef": True},
        {"name": "precond_512_fp64", "kind": "precond", "L": 32, "m0": 16, "batch": 25,
         "contrast": 10.0, "precision": FP64, "delta": 0.0},
        # Chebyshev moments of the density of states (random sign vectors, lumped scheme)
        {"name": "dos_64", "kind": "dos", "L": 8, "m0": 8, "batch": 16, "K": 512,
         "scheme": "lumped"},
        # the 3D form: field, three correctors and A_hom
        {"name": "cubes_64_mixed", "kind": "cubes", "L": 4, "m0": 16, "batch": 15,
         "contrast": 10.0, "precision": MIXED, "tol": 1e-10, "scheme": "consistent"},
    ]


def _ensemble(name, L, m0, batch, contrast, precision, tol, scheme="consistent"):
    return {"name": name, "kind": "ensemble", "L": L, "m0": m0, "batch": batch,
            "contrast": contrast, "precision": precision, "tol": tol, "scheme": scheme}


def draw(rng) -> dict:
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["ensemble", "ensemble", "plan", "study", "adjoint", "fem", "stiffness",
                       "stiffness", "precond", "precond", "dos", "cubes", "cubes"])
    n = 1 << rng.randint(5, 11)
    m0 = rng.choice([4, 8, 16])
    scheme = rng.choice(["consistent", "consistent", "lumped"])
    precision = rng.choice([FP64, MIXED])
    contrast = rng.choice([10.0, 100.0, 2.5, round(rng.uniform(2.0, 100.0), 2)])

    def batch(nodes):   # at most `nodes` grid nodes in all
        return log_int(1, max(1, min(2000, nodes // (n * n))))

    if kind == "ensemble":
        tol = rng.choice([1e-8, 1e-10])
        return {"kind": kind, "L": n // m0, "m0": m0,
                "batch": batch(1 << 20 if precision == FP64 else 1 << 23), "contrast": contrast,
                "precision": precision, "tol": tol, "scheme": scheme}
    if kind == "plan":
        return {"kind": kind, "batch": log_int(3, 250), "precision": MIXED, "tol": 1e-10}
    if kind == "study":
        L = rng.choice([8, 16, 32, 64])
        return {"kind": kind, "L": L, "batch": log_int(10, 24_000_000 // (16 * L * L)),
                "precision": MIXED, "tol": 1e-8}
    if kind == "adjoint":
        n = min(n, 1024)
        return {"kind": kind, "L": n // m0, "m0": m0, "batch": batch(1 << 20),
                "contrast": contrast, "tol": 1e-12, "scheme": scheme}
    if kind == "fem":
        n = min(n, 1024)
        L = rng.choice([2, 4, 8])
        return {"kind": kind, "L": L, "m0": n // L, "batch": batch(1 << 20), "contrast": contrast,
                "tol": 1e-10, "scheme": scheme}
    if kind == "stiffness":
        return {"kind": kind, "L": n // m0, "m0": m0, "batch": batch(20_000_000),
                "contrast": contrast, "precision": precision, "scheme": scheme,
                "coef": rng.random() < 0.5}
    if kind == "precond":
        return {"kind": kind, "L": n // m0, "m0": m0, "batch": batch(8_000_000),
                "contrast": contrast, "precision": precision,
                "delta": rng.choice([0.0, round(rng.uniform(0.01, 1.0), 3)])}
    if kind == "dos":
        return {"kind": kind, "L": rng.choice([4, 8, 16]), "m0": 8, "batch": log_int(1, 48),
                "K": rng.choice([128, 255, 512]), "scheme": rng.choice(["lumped", "consistent"])}
    n = 1 << rng.randint(5, 7 if precision == MIXED else 6)
    m0 = rng.choice([8, 16])
    most = (1 << 22) if precision == MIXED else (1 << 18)
    return {"kind": kind, "L": n // m0, "m0": m0,
            "batch": log_int(1, max(1, min(64, most // n ** 3))), "contrast": contrast,
            "precision": precision, "tol": rng.choice([1e-8, 1e-10]), "scheme": scheme}


def _scheme(case):
    return rve.LUMPED if case.get("scheme") == "lumped" else rve.CONSISTENT


def _precision(case):
    return rve.FP64 if case.get("precision", FP64) == FP64 else rve.MIXED


def _descs(case, seed):
    kind = case["kind"]
    if kind == "plan":   # sizes and contrasts are part of the workload's seed
        return workloads.config_batch("uneven_4096", seed=seed, count=case["batch"])
    if kind == "study":
        return studies.paper_descs(case["L"], case["batch"], seed=seed)
    if kind == "dos":
        return [workloads.realization(case["L"], case["m0"], 2.0, seed, 0, density=1.0,
                                      side_units=0.5, a_matrix=0.5)] * case["batch"]
    if kind == "cubes":
        return [workloads.realization3(case["L"], case["m0"], case["contrast"], seed, k)
                for k in range(case["batch"])]
    return workloads.batch(case["L"], case["m0"], case["contrast"], seed, case["batch"])


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _normal(count, comps, dtype, seed):
    return torch.randn(count, comps, dtype=dtype, device="cuda", generator=_gen(seed))


def _nodal_load(case, seed):
    """Two smooth nodal loads per realization (the FEM test's, with seeded weights)."""
    n, L, B = case["L"] * case["m0"], case["L"], case["batch"]
    x = torch.arange(n, dtype=torch.float64, device="cuda") / case["m0"]
    a = torch.outer(torch.sin(2 * np.pi * x / L), torch.cos(6 * np.pi * x / L))
    w = torch.rand(B, 2, dtype=torch.float64, device="cuda", generator=_gen(seed)) + 0.5
    g = torch.stack([a, a.t()], dim=-1).reshape(1, n * n, 2) * w[:, None, :]
    return g.reshape(B * n * n, 2).contiguous()


def _signs(case, seed):
    n, B = case["L"] * case["m0"], case["batch"]
    return torch.randint(0, 2, (B * n * n, 2), device="cuda", generator=_gen(seed)).double() * 2 - 1


def _weights(case, seed):
    """The gradient arriving at A_hom in the adjoint cases."""
    return torch.randn(case["batch"], 2, 2, dtype=torch.float64, device="cuda", generator=_gen(seed))


DOS_HI = 16.0 * 0.5 * 1.0 * (1.0 + 1e-9)   # Gershgorin bound, lumped weights, a_max = 1


# ------------------------------------------------------------ prepare / run --
def prepare(case, seed):
    kind = case["kind"]
    ds = _descs(case, seed)
    s = {"kind": kind, "scheme": _scheme(case), "precision": _precision(case)}
    if kind == "cubes":
        s["batch"] = rve3.Batch3(ds)
        s["tol"] = case["tol"]
        return s
    b = rve.Batch(ds)
    s["batch"] = b
    if kind == "ensemble":
        s["opts"] = rve.make_opts(scheme=s["scheme"], precision=s["precision"], tol=case["tol"])
        # the host pipeline's workspace, kept by a program that calls it again
        nb = rve.lib().rve_homogenize_workspace_size(b.ptr, b.count, rve.ctypes.byref(s["opts"]))
        s["ws"] = rve.workspace(nb)
    elif kind == "plan":
        s["plan"] = rve.Plan(b, rve.make_opts(precision=rve.MIXED, tol=case["tol"],
                                              path=rve.PATH_FUSED))
    elif kind == "study":
        s["opts"] = rve.make_opts(scheme=rve.LUMPED, precision=rve.MIXED, tol=case["tol"])
        s["ws"] = rve.workspace(rve.workspace_size(b, s["opts"]))
    elif kind == "adjoint":
        s["opts"] = rve.make_opts(scheme=s["scheme"], precision=rve.FP64, tol=case["tol"])
        s["coef"] = rve.coef_from_mask(b, rve.gen_field(b)).requires_grad_(True)
        s["G"] = _weights(case, seed)
    elif kind == "fem":
        s["opts"] = rve.make_opts(scheme=s["scheme"], precision=rve.FP64, tol=case["tol"])
        s["coef"] = rve.coef_from_mask(b, rve.gen_field(b))
        s["g"] = _nodal_load(case, seed)
    elif kind == "stiffness":
        mask = rve.gen_field(b)
        s["mask"] = None if case["coef"] else mask
        s["coef"] = rve.coef_from_mask(b, mask) if case["coef"] else None
        s["x"] = _normal(b.nodes, 2, torch.float64 if s["precision"] == rve.FP64 else torch.float32,
                         seed)
    elif kind == "precond":
        s["x"] = _normal(b.nodes, 2, torch.float64 if s["precision"] == rve.FP64 else torch.float32,
                         seed)
        s["delta"] = case["delta"]
    elif kind == "dos":
        words = rve.gen_field(b.descs[:1])
        s["mask"] = words.repeat(b.count)
        s["v"] = _signs(case, seed)
        s["K"] = case["K"]
    return s


def run(s):
    kind, b = s["kind"], s["batch"]
    if kind == "ensemble":
        A, infos = rve.homogenize_host(b, s["opts"], ws=s["ws"])
        return {"A": A, "status": np.array([i["status"] for i in infos])}
    if kind == "plan":
        A, info = s["plan"].execute()
        return {"A": A, "status": info.view(torch.int32).view(b.count, -1)[:, 2]}
    if kind == "study":
        mask = rve.gen_field(b)
        u, info = rve.solve(b, mask=mask, opts=s["opts"], ws=s["ws"])
        A = rve.a_hom(b, u, mask=mask, scheme=rve.LUMPED, precision=rve.MIXED, ws=s["ws"])
        return {"A": A, "status": info.view(torch.int32).view(b.count, -1)[:, 2]}
    if kind == "adjoint":
        A = rve.AHom.apply(s["coef"], b, s["opts"])
        (grad,) = torch.autograd.grad(A, s["coef"], s["G"])
        return {"A": A.detach(), "grad": grad}
    if kind == "fem":
        f = rve.apply_mass(b, s["g"], scheme=s["scheme"])
        u, info = rve.solve(b, coef=s["coef"], opts=s["opts"], f=f)
        return {"f": f, "u": u, "status": info.view(torch.int32).view(b.count, -1)[:, 2]}
    if kind == "stiffness":
        return rve.apply_stiffness(b, s["x"], mask=s["mask"], coef=s["coef"], scheme=s["scheme"])
    if kind == "precond":
        return rve.apply_precond(b, s["x"], delta=s["delta"])
    if kind == "dos":
        return rve.cheb_moments(b, s["v"], s["K"], 0.0, DOS_HI, mask=s["mask"], scheme=s["scheme"])
    A, infos = rve3.homogenize(b, scheme=s["scheme"], tol=s["tol"], precision=s["precision"])
    return {"A": A, "status": np.array([i["status"] for i in infos])}


# --------------------------------------------------------------------- work --
def work(case) -> dict:
    """Bytes and operations of one call.  A single application reads its
    inputs and writes its outputs once.  A solve moves, per CG step and
    vector, p, x and r once in and once out, the preconditioned residual once
    out and in, and what the row transforms hand to the column solves once
    out and in (10 vector passes); the number of steps is CG's bound
    sqrt(contrast) log(2/tol) / 2 with the factor 1.7 that the residual norm
    is seen to take on these fields."""
    kind = case["kind"]
    v = 16 if case.get("precision", FP64) == FP64 else 8   # bytes of a node's corrector pair

    def solve(nodes, n, contrast, tol, vb, pairs=1.0, dims=2):
        steps = math.ceil(0.85 * math.sqrt(contrast) * math.log(2.0 / tol))
        passes = 10 if dims == 2 else 14   # 3D: two more transforms between x and z
        per = (2 * (dims - 1) * 5 * math.log2(n) + (36 if dims == 2 else 108) + 30)
        return {"bytes": nodes * pairs * passes * vb * steps, "flops": nodes * pairs * per * steps}

    if kind == "plan":
        tot = {"bytes": 0.0, "flops": 0.0}
        for d in workloads.config_batch("uneven_4096", seed=0, count=case["batch"]):
            n = d["L"] * d["m0"]
            w = solve(n * n, n, d["a_incl"], case["tol"], 8)
            tot = {k: tot[k] + w[k] for k in tot}
        return tot
    if kind == "study":
        n = 4 * case["L"]
        return solve(case["batch"] * n * n, n, 2.5, case["tol"], 8)
    n = case["L"] * case["m0"]
    if kind == "cubes":
        return solve(case["batch"] * n ** 3, n, case["contrast"], case["tol"], v, pairs=1.5, dims=3)
    nodes = case["batch"] * n * n
    if kind == "ensemble":
        return solve(nodes, n, case["contrast"], case["tol"], v)
    if kind in ("adjoint", "fem"):
        w = solve(nodes, n, case["contrast"], case["tol"], 16)
        w["bytes"] += nodes * 40   # the gradient's, or the mass matrix's, vectors
        return w
    stencil = 36 if case.get("scheme", "consistent") == "consistent" else 20
    if kind == "stiffness":
        return {"bytes": nodes * (2 * v + (8 if case["coef"] else 0.125)), "flops": nodes * stencil}
    if kind == "precond":
        return {"bytes": nodes * 2 * v, "flops": nodes * (2 * 5 * math.log2(n) + 16)}
    # Chebyshev: two vectors per step, one in and one in and out; small grids
    # could stay on the chip, so only the start vectors have to be read
    return {"bytes": nodes * 16 + case["batch"] * 2 * case["K"] * 8,
            "flops": nodes * (stencil + 12) * ((case["K"] + 1) // 2)}


# -------------------------------------------------------------------- exact --
_M64 = (1 << 64) - 1
_GAMMA = 0x9E3779B97F4A7C15


def _mix(z):
    z = z.astype(np.uint64)
    with np.errstate(over="ignore"):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _corners(d, dim, n):
    """Lower corners [n_incl, dim] of the inclusions (SplitMix64 counters)."""
    key = int(_mix(np.array([(d["seed"] + (d["index"] + 1) * _GAMMA) & _M64], dtype=np.uint64))[0])
    ctr = np.arange(dim * d["n_incl"], dtype=np.uint64) + np.uint64((1 << 40) + 1)
    with np.errstate(over="ignore"):
        v = _mix(np.uint64(key) + ctr * np.uint64(_GAMMA))
    shift = 64 - int(n).bit_length() + 1   # n a power of two: the draw's high bits
    return (v >> np.uint64(shift)).astype(np.int64).reshape(-1, dim)


def _field(d, dim):
    """Cell values of one realization, [n] * dim, float64 on the GPU."""
    n, s = d["L"] * d["m0"], d["incl_cells"]
    c = torch.as_tensor(_corners(d, dim, n), device="cuda")
    cnt = torch.zeros((n,) * dim, dtype=torch.float64, device="cuda")
    if len(c):
        cnt.index_put_(tuple(c.t()), torch.ones(len(c), dtype=torch.float64, device="cuda"),
                       accumulate=True)
    for ax in range(dim):   # a cell is covered by a corner at most s - 1 cells below it
        cs = torch.cumsum(torch.cat([cnt, cnt], dim=ax), dim=ax)
        hi = cs.narrow(ax, n, n)
        cnt = hi - cs.narrow(ax, n - s, n)
    return torch.where(cnt > 0.5, d["a_incl"], d["a_matrix"]).double()


def _element(dim, h, scheme):
    m = h * np.array([[1 / 3, 1 / 6], [1 / 6, 1 / 3]]) if scheme == 0 else h * np.eye(2) / 2
    k = np.array([[1.0, -1.0], [-1.0, 1.0]]) / h
    E = np.zeros((2 ** dim, 2 ** dim))
    for ax in range(dim):
        t = np.ones((1, 1))
        for q in range(dim):
            t = np.kron(t, k if q == ax else m)
        E += t
    return E


class _Grid:
    """A batch of equal-size realizations: fields v[comp, batch, n, ...]."""

    def __init__(self, a, h, scheme):
        self.a, self.h = a, h
        self.dim = a.dim() - 1
        self.axes = list(range(-self.dim, 0))
        self.E = _element(self.dim, h, scheme)
        # the corner bits of the local order, first axis the slowest
        self.bits = [tuple((c >> (self.dim - 1 - q)) & 1 for q in range(self.dim))
                     for c in range(2 ** self.dim)]

    def at(self, v, bits):   # v at the cell's corner
        return torch.roll(v, [-b for b in bits], self.axes) if any(bits) else v

    def apply(self, v):      # A v, element by element
        loc = [self.at(v, b) for b in self.bits]
        out = torch.zeros_like(v)
        for r, br in enumerate(self.bits):
            t = torch.zeros_like(v)
            for c in range(len(self.bits)):
                if self.E[r, c]:
                    t += self.E[r, c] * loc[c]
            t *= self.a
            out += torch.roll(t, list(br), self.axes) if any(br) else t
        return out

    def loads(self):         # -A x_i, cell by cell (x_i = h times the corner bit)
        f = []
        for ax in range(self.dim):
            xi = self.h * np.array([b[ax] for b in self.bits])
            w = -(self.E @ xi)
            t = torch.zeros_like(self.a)
            for r, br in enumerate(self.bits):
                t += torch.roll(w[r] * self.a, list(br), self.axes) if any(br) else w[r] * self.a
            f.append(t)
        return torch.stack(f)

    def precond(self, c0, delta=0.0):
        n = self.a.shape[-1]
        dev = self.a.device
        lam = 4 * torch.sin(np.pi * torch.arange(n, dtype=torch.float64, device=dev) / n) ** 2
        half = lam[: n // 2 + 1]
        sym = lam[:, None] + half if self.dim == 2 else lam[:, None, None] + lam[:, None] + half
        sym = c0 * sym + delta
        inv = torch.where(sym > 0, 1.0 / torch.where(sym > 0, sym, 1.0), 0.0)
        return lambda r: torch.fft.irfftn(torch.fft.rfftn(r, dim=self.axes) * inv, s=(n,) * self.dim,
                                          dim=self.axes)

    def solve(self, f, c0, tol=1e-13, most=1500):
        """CG from 0, restarted once from the true residual."""
        B = self.precond(c0)
        dot = lambda x, y: (x * y).sum(dim=self.axes, keepdim=True)  # noqa: E731
        u = torch.zeros_like(f)
        fn = dot(f, f).sqrt().clamp_min(1e-300)
        for cycle in range(2):
            r = f - self.apply(u)
            z = B(r)
            p = z.clone()
            rho = dot(r, z)
            for it in range(most):
                q = self.apply(p)
                al = rho / dot(p, q).clamp_min(1e-300)
                u += al * p
                r -= al * q
                if it % 8 == 7 and float((dot(r, r).sqrt() / fn).max()) < (tol if not cycle else 0.1 * tol):
                    break
                z = B(r)
                new = dot(r, z)
                p = z + (new / rho.clamp_min(1e-300)) * p
                rho = new
        return u

    def local(self, u):      # v_i = xi_i + u_i at the corners of every cell
        out = []
        for ax in range(self.dim):
            out.append([self.at(u[ax], b) + self.h * b[ax] for b in self.bits])
        return out

    def energies(self, u):   # v_i^T E v_j per cell, from differences across the cell
        v = self.local(u)
        k = len(self.bits)
        e = {}
        for i in range(self.dim):
            for j in range(i, self.dim):
                t = torch.zeros_like(self.a)
                for c in range(k):
                    for q in range(c):
                        if self.E[c, q]:
                            t -= self.E[c, q] * (v[i][c] - v[i][q]) * (v[j][c] - v[j][q])
                e[i, j] = e[j, i] = t
        return e


def _grid_of(ds, scheme, dim=2):
    a = torch.stack([_field(d, dim) for d in ds])
    return _Grid(a, 1.0 / ds[0]["m0"], scheme)


def _c0(ds):
    return 0.5 * (ds[0]["a_matrix"] + ds[0]["a_incl"])


def _a_hom(g, u, L):
    e = g.energies(u)
    rows = [torch.stack([(g.a * e[i, j]).sum(dim=g.axes) for j in range(g.dim)], dim=-1)
            for i in range(g.dim)]
    return torch.stack(rows, dim=-2) / float(L) ** g.dim


def exact(case, seed):
    kind = case["kind"]
    scheme = 1 if kind == "study" or case.get("scheme") == "lumped" else 0
    ds = _descs(case, seed)
    if kind in ("ensemble", "study", "cubes", "plan"):
        dim = 3 if kind == "cubes" else 2
        A = torch.zeros(len(ds), dim, dim, dtype=torch.float64)
        groups = {}
        for k, d in enumerate(ds):
            groups.setdefault((d["L"] * d["m0"], d["a_incl"]), []).append(k)
        for (n, _), idx in groups.items():
            step = max(1, (1 << 25) // n ** dim)
            for s in range(0, len(idx), step):
                part = [ds[k] for k in idx[s:s + step]]
                g = _grid_of(part, scheme, dim)
                u = g.solve(g.loads(), _c0(part))
                A[idx[s:s + step]] = _a_hom(g, u, part[0]["L"]).cpu()
        return {"A": A, "status": None}
    n, B = case["L"] * case["m0"], case["batch"]

    def to_grid(x):   # [nodes, 2] -> [2, B, n, n]
        return x.double().reshape(B, n, n, 2).permute(3, 0, 1, 2).contiguous()

    def to_nodes(v):
        return v.permute(1, 2, 3, 0).reshape(B * n * n, 2)

    if kind == "adjoint":
        g = _grid_of(ds, scheme)
        u = g.solve(g.loads(), _c0(ds))
        e, G = g.energies(u), _weights(case, seed)[..., None, None]
        grad = sum(G[:, i, j] * e[i, j] for i in range(2) for j in range(2)) / float(case["L"]) ** 2
        return {"A": _a_hom(g, u, case["L"]), "grad": grad.reshape(-1)}
    if kind == "fem":
        h = 1.0 / case["m0"]
        x = to_grid(_nodal_load(case, seed))
        if scheme == 0:
            for ax in (-2, -1):
                x = (torch.roll(x, 1, ax) + 4 * x + torch.roll(x, -1, ax)) / 6
        f = h * h * x
        g = _grid_of(ds, scheme)
        u = g.solve(f, _c0(ds), tol=1e-12)
        return {"f": to_nodes(f), "u": to_nodes(u), "status": None}
    if kind == "stiffness":
        g = _grid_of(ds, scheme)
        x = _normal(B * n * n, 2, torch.float64 if case["precision"] == FP64 else torch.float32, seed)
        return to_nodes(g.apply(to_grid(x)))
    if kind == "precond":
        g = _Grid(torch.ones(1, n, n, dtype=torch.float64, device="cuda"), 1.0, 0)
        x = _normal(B * n * n, 2, torch.float64 if case["precision"] == FP64 else torch.float32, seed)
        return to_nodes(g.precond(_c0(ds), case["delta"])(to_grid(x)))
    # Chebyshev moments v^T T_k v of the operator mapped to [-1, 1]
    g = _grid_of(ds[:1], scheme)
    v = to_grid(_signs(case, seed))
    tilde = lambda w: (2.0 / DOS_HI) * g.apply(w) - w  # noqa: E731
    prev, cur = v, tilde(v)
    mu = torch.zeros(B, 2, case["K"], dtype=torch.float64, device="cuda")
    for k in range(case["K"]):
        w = prev if k == 0 else cur
        mu[:, :, k] = (v * w).sum(dim=(-2, -1)).t()
        if k:
            prev, cur = cur, 2 * tilde(cur) - prev
    return mu
