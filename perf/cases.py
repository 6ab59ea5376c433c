"""The timed cases of the library: what its callers run, from the smallest tangent apply to whole
linear and Newton solves, each through the public binding.

`listed()` holds the cases, `draw()` more of the same ranges, `prepare()` what a program has in
hand before the call (inputs on the GPU, the problem with its linearisation point, the network's
weights), `run()` one pass, `work()` the bytes and operations a pass cannot do without, and
`exact()` the same result in plain FP64 torch, without the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2505_15535_gb300 import nhmf

MU = 1.0
PRECISION = {"fp64": nhmf.NHMF_FP64, "fp32": nhmf.NHMF_FP32, "df64": nhmf.NHMF_DF64}
STRATEGY = {"on_the_fly": nhmf.NHMF_ON_THE_FLY, "cached": nhmf.NHMF_CACHED, "spatial": nhmf.NHMF_SPATIAL}
SOLVER = {"jacobi_cg": nhmf.NHMF_SOLVER_JACOBI_CG, "mixed_fcg": nhmf.NHMF_SOLVER_MIXED_FCG,
          "mixed_gmg": nhmf.NHMF_SOLVER_MIXED_GMG}
MODEL = {"compressible": nhmf.NHMF_MODEL_COMPRESSIBLE, "split": nhmf.NHMF_MODEL_SPLIT}
BC = {"none": nhmf.NHMF_BC_NONE, "clamp": nhmf.NHMF_BC_CLAMP_X0, "compression": nhmf.NHMF_BC_COMPRESSION}
LINEAR_RTOL = 1e-10   # of the timed solves: tight, so that the solution is defined to about this
NEWTON_RTOL = 1e-10
COMPRESSION = 0.01    # of the cube's height in one load step


def _tangent(name, n_el, degree, precision, strategy, lam, bc, model="compressible", inclusions=False):
    return {"name": name, "op": "tangent", "n_el": n_el, "degree": degree, "precision": precision,
            "strategy": strategy, "lam": lam, "bc": bc, "model": model, "inclusions": inclusions}


def listed():
    return [
        # a check or a coarse-level apply on the smallest mesh: latency and launches
        _tangent("tangent_q1_8_fp64", 8, 1, "fp64", "on_the_fly", 1.5, "clamp"),
        # the matrix-vector product of every FP64 Krylov iteration (the benchmark's headline)
        _tangent("tangent_q2_64_fp64_cached", 64, 2, "fp64", "cached", 1.5, "clamp"),
        # one-off products at a new state, where no point cache is worth building (Algorithm 1)
        _tangent("tangent_q4_32_fp64", 32, 4, "fp64", "on_the_fly", 1.5, "clamp"),
        # the smoother's and the inner CG's product on the fine level of the mixed solvers
        _tangent("tangent_q2_64_fp32_cached", 64, 2, "fp32", "cached", 1.5, "compression"),
        # the same on the largest mesh in use, 51 M DoFs
        _tangent("tangent_q4_64_fp32_cached", 64, 4, "fp32", "cached", 49.0, "compression"),
        # an odd mesh with stiff inclusions, FP32 on the fly (no memory for a cache)
        _tangent("tangent_q3_47_fp32", 47, 3, "fp32", "on_the_fly", 1.5, "clamp", inclusions=True),
        # the outer product of the mixed solvers in double-float arithmetic
        _tangent("tangent_q3_48_df64_cached", 48, 3, "df64", "cached", 49.0, "compression"),
        # what each Newton iterate needs before its linear solve, and the first smoothing product
        {"name": "setup_q3_48", "op": "setup", "n_el": 48, "degree": 3, "lam": 49.0, "bc": "compression",
         "inclusions": False},
        # the linear solve inside Newton at the size of the compression runs
        {"name": "solve_q2_64_gmg", "op": "solve", "n_el": 64, "degree": 2, "lam": 1.5, "bc": "compression",
         "solver": "mixed_gmg", "outer": "fp64", "inclusions": False},
        # high order, near-incompressible, double-float outer products
        {"name": "solve_q4_16_gmg_df64", "op": "solve", "n_el": 16, "degree": 4, "lam": 49.0, "bc": "compression",
         "solver": "mixed_gmg", "outer": "df64", "inclusions": False},
        # a whole load step on a small mesh: many short kernels and host reads
        {"name": "newton_q2_16_gmg", "op": "newton", "n_el": 16, "degree": 2, "lam": 1.5, "bc": "compression",
         "solver": "mixed_gmg", "outer": "fp64", "inclusions": False},
        # training the learned preconditioner on the nodal grid of the Q2 64^3 mesh
        {"name": "unet_grad_129", "op": "unet_grad", "n_el": 64, "degree": 2, "bc": "compression"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    op = rng.choice(["tangent"] * 6 + ["setup", "solve", "newton", "unet_grad", "unet_forward"])
    bc = rng.choice(["none", "clamp", "compression"])
    inclusions = rng.random() < 0.25
    if op == "tangent":
        degree = rng.choice([1, 2, 3, 4])
        precision, strategy = rng.choice([("fp64", "on_the_fly"), ("fp64", "cached"), ("fp64", "spatial"),
                                          ("fp32", "on_the_fly"), ("fp32", "cached"), ("fp32", "cached"),
                                          ("df64", "cached")])
        top = 200 if precision == "fp32" else 128   # nodes per direction
        model = "split" if strategy != "cached" and rng.random() < 0.3 else "compressible"
        return {"op": op, "n_el": _log_int(rng, 4, top // degree), "degree": degree, "precision": precision,
                "strategy": strategy, "lam": rng.choice([1.5, 5.0, 49.0]), "bc": bc, "model": model,
                "inclusions": inclusions}
    if op == "setup":
        degree = rng.choice([1, 2, 3, 4])
        return {"op": op, "n_el": _log_int(rng, 6, 128 // degree), "degree": degree, "lam": rng.choice([1.5, 49.0]),
                "bc": bc, "inclusions": inclusions}
    if op in ("solve", "newton"):
        degree = rng.choice([1, 2, 3, 4])
        solver = rng.choice(["mixed_gmg", "mixed_gmg", "mixed_gmg", "mixed_fcg", "jacobi_cg"])
        # multigrid halves even meshes; the Krylov solvers without it run the smaller ones
        top = {"newton": 32, "solve": 64}[op] if solver == "mixed_gmg" else {"newton": 20, "solve": 32}[op]
        n_el = _log_int(rng, 4, top // degree)
        if solver == "mixed_gmg":
            n_el += n_el % 2
        return {"op": op, "n_el": n_el, "degree": degree, "lam": 1.5, "bc": rng.choice(["clamp", "compression"])
                if op == "solve" else "compression", "solver": solver, "inclusions": inclusions and op == "solve",
                "outer": "fp64" if solver == "jacobi_cg" else rng.choice(["fp64", "df64"])}
    return {"op": op, "n_el": 2 * _log_int(rng, 4, 32), "degree": 2, "bc": bc}


# ------------------------------------------------------------------ inputs
def _uniform(seed, n, a, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (2 * a) - a).to(dtype)


def _normal(seed, n, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, generator=g, device="cuda", dtype=dtype)


def _constrained(case):
    """Boolean [3, M, M, M] (component, z, y, x) of the constrained DoFs."""
    M = case["degree"] * case["n_el"] + 1
    m = torch.zeros(3, M, M, M, dtype=torch.bool, device="cuda")
    if case["bc"] == "clamp":
        m[..., 0] = True
    elif case["bc"] == "compression":
        m[:, 0] = True
        m[2, M - 1] = True
    return m


def _state_u(case, seed, amp=0.05):
    """A deformed state with det F > 0: nodal difference quotients within +-amp."""
    M = case["degree"] * case["n_el"] + 1
    u = _uniform(seed, 3 * M ** 3, amp / (case["n_el"] * case["degree"]))
    return u.masked_fill_(_constrained(case).reshape(-1), 0.0)


def _compressed_u(case, seed):
    """A state as load steps reach it: 1 % compressed along the loaded axis and wider by half of that
    along the others (near-incompressible material keeps its volume), with small deviations."""
    M = case["degree"] * case["n_el"] + 1
    t, _, _ = _basis(case["degree"], nodes_only=True)
    e = torch.arange(case["n_el"], device="cuda", dtype=torch.float64)
    x = torch.cat([((e[:, None] + torch.from_numpy(t[:-1]).cuda()) / case["n_el"]).reshape(-1),
                   torch.ones(1, dtype=torch.float64, device="cuda")])
    u = _uniform(seed, 3 * M ** 3, 0.0002 / (case["n_el"] * case["degree"])).reshape(3, M, M, M)
    along = 0 if case["bc"] == "clamp" else 2
    for c, xc in enumerate((x, x[:, None], x[:, None, None])):
        u[c] += COMPRESSION * (-xc if c == along else 0.5 * xc)
    return u.reshape(-1)


def _factors(case):
    """Per-element factors of two spherical inclusions 100x stiffer than the matrix."""
    N = case["n_el"]
    x = (torch.arange(N, device="cuda", dtype=torch.float64) + 0.5) / N
    z, y, x = torch.meshgrid(x, x, x, indexing="ij")
    f = torch.ones(N, N, N, dtype=torch.float64, device="cuda")
    for cx in (0.3, 0.7):
        f[(x - cx) ** 2 + (y - 0.5) ** 2 + (z - 0.5) ** 2 <= 0.15 ** 2] = 100.0
    return f.reshape(-1)


def _problem(case):
    p = nhmf.Problem(case["n_el"], case["degree"], MU, case.get("lam", 1.5), BC[case["bc"]],
                     model=MODEL[case.get("model", "compressible")])
    if case.get("inclusions"):
        nhmf.nhmf_set_material_factors(p.ctx, _factors(case))
    return p


def _mask(case):
    """The point caches that the case's applies read."""
    op = case["op"]
    if op == "setup":
        return nhmf.NHMF_CACHE_FP64 | nhmf.NHMF_CACHE_FP32
    if op == "tangent":
        if case["strategy"] == "spatial":
            return nhmf.NHMF_CACHE_SPATIAL
        if case["strategy"] == "on_the_fly":
            return 0
        return {"fp64": nhmf.NHMF_CACHE_FP64, "fp32": nhmf.NHMF_CACHE_FP32, "df64": nhmf.NHMF_CACHE_DF64}[case["precision"]]
    mask = nhmf.NHMF_CACHE_FP64
    if case["solver"] != "jacobi_cg":
        mask |= nhmf.NHMF_CACHE_FP32
    if case["outer"] == "df64":
        mask |= nhmf.NHMF_CACHE_DF64
    return mask


def _unet_params(case, seed):
    """He-normal weights with small biases, in the layers' order."""
    rs = np.random.RandomState(seed)
    flat = []
    for _, kind, cin, cout in UNET:
        flat.append(rs.standard_normal(27 * cin * cout) * math.sqrt(2.0 / (27 * cin)))
        flat.append(0.05 * rs.standard_normal(cout))
    return np.concatenate(flat).astype(np.float32)


def _inputs(case, seed):
    """The case's tensors by name, from the seed alone."""
    M = case["degree"] * case["n_el"] + 1
    n = 3 * M ** 3
    op = case["op"]
    if op in ("unet_grad", "unet_forward"):
        return {"x": _normal(7 * seed + 1, n, torch.float32), "e": _normal(7 * seed + 2, n, torch.float32)}
    if op == "newton":
        # a state near the last converged one, and the next prescribed displacement
        return {"u": _state_u(case, 7 * seed + 1, amp=0.01)}
    d = {"u": (_compressed_u if op == "solve" else _state_u)(case, 7 * seed + 1)}
    dtype = torch.float32 if op == "setup" or case.get("precision") == "fp32" else torch.float64
    d["du"] = _normal(7 * seed + 2, n, dtype).masked_fill_(_constrained(case).reshape(-1), 0.0)
    return d


def prepare(case, seed):
    s = {"case": case, **_inputs(case, seed)}
    op = case["op"]
    p = s["problem"] = _problem(case)
    if op in ("unet_grad", "unet_forward"):
        nhmf.nhmf_unet_create(p.ctx)
        nhmf.nhmf_unet_set_params(p.ctx, _unet_params(case, seed % (1 << 31)))
        s["y"] = torch.empty_like(s["x"])
    elif op == "newton":
        s["sol"] = torch.empty_like(s["u"])
    elif op == "setup":
        s["r"], s["d"] = torch.empty_like(s["u"]), torch.empty_like(s["u"])
        s["v"] = torch.empty_like(s["du"])
    else:
        p.set_linearization(s["u"], _mask(case))
        s["v"] = torch.empty_like(s["du"])
    return s


def run(s):
    case, p = s["case"], s["problem"]
    op = case["op"]
    if op == "tangent":
        return p.apply(s["du"], s["v"], PRECISION[case["precision"]], STRATEGY[case["strategy"]])
    if op == "setup":
        p.residual(s["u"], s["r"])
        p.set_linearization(s["u"], _mask(case))
        p.diagonal(s["d"])
        p.apply(s["du"], s["v"], nhmf.NHMF_FP32, nhmf.NHMF_CACHED)
        return {"r": s["r"], "d": s["d"], "v": s["v"]}
    if op == "solve":
        p.linear_solve(s["du"], s["v"], solver=SOLVER[case["solver"]], linear_rtol=LINEAR_RTOL,
                       outer_apply=PRECISION[case["outer"]])
        return s["v"]
    if op == "newton":
        s["sol"].copy_(s["u"])
        p.solve(s["sol"], solver=SOLVER[case["solver"]], load_steps=1, compression=COMPRESSION,
                newton_rtol=NEWTON_RTOL, outer_apply=PRECISION[case["outer"]])
        return s["sol"]
    if op == "unet_grad":
        loss, grads = nhmf.nhmf_unet_loss_grad(p.ctx, s["x"], s["e"])
        return {"loss": np.float32(loss), "grads": grads}
    nhmf.nhmf_unet_forward(p.ctx, s["x"], s["y"])
    return s["y"]


# ------------------------------------------------------------------ work
UNET = [("in", "conv", 3, 16), ("e0", "conv", 16, 16), ("d1", "down", 16, 16), ("e1", "conv", 16, 16),
        ("d2", "down", 16, 16), ("m2", "conv", 16, 16), ("u1", "up", 16, 16), ("t1", "conv", 16, 16),
        ("u0", "up", 16, 16), ("t0", "conv", 16, 16), ("out", "conv", 16, 3)]
UNET_LEVEL = {"in": 0, "e0": 0, "d1": 1, "e1": 1, "d2": 2, "m2": 2, "u1": 1, "t1": 1, "u0": 0, "t0": 0, "out": 0}


def _tangent_work(N, p, size, cached, values=10):
    """One apply: du and v once, and u or the point values once; 2 n^4 operations per 1D pass and
    scalar field (18 passes each for u, du and back) and the point code."""
    n, M = p + 1, p * N + 1
    passes, point = (36, 150) if cached else (54, 230)
    by = 2 * size * 3 * M ** 3 + (values * size * N ** 3 * n ** 3 if cached else size * 3 * M ** 3)
    return by, N ** 3 * (passes * 2 * n ** 4 + point * n ** 3)


def work(case):
    N, p, op = case["n_el"], case["degree"], case["op"]
    n, M = p + 1, p * N + 1
    dofs = 3 * M ** 3
    if op == "tangent":
        by, fl = _tangent_work(N, p, 4 if case["precision"] == "fp32" else 8, case["strategy"] != "on_the_fly",
                               36 if case["strategy"] == "spatial" else 10)
    elif op == "setup":
        # u read; r, d, the FP64 and FP32 point values and v written; du and the FP32 values read
        tb, tf = _tangent_work(N, p, 4, True)
        by = 8 * 3 * dofs + 120 * N ** 3 * n ** 3 + tb
        fl = N ** 3 * (2 * (36 * 2 * n ** 4 + 150 * n ** 3) + 6 * 9 * 2 * n ** 4) + tf
    elif op in ("solve", "newton"):
        # a product per outer iteration in the outer precision, and for multigrid seven FP32
        # products on the fine level with 8/7 for the coarser meshes; about a dozen iterations a
        # solve (fifty for near-incompressible material), three solves a load step
        its = (12 if case["lam"] < 10 else 50) * (3 if op == "newton" else 1)
        ob, of = _tangent_work(N, p, 8, True)
        ib, if_ = _tangent_work(N, p, 4, True)
        inner = 8 if case["solver"] == "mixed_gmg" else (0 if case["solver"] == "jacobi_cg" else 30)
        if case["solver"] == "jacobi_cg":
            its *= M // 4 + 1
        by, fl = its * (ob + inner * ib), its * (of + inner * if_)
    else:
        by, fl = 2 * dofs * 4, 0
        sizes = [M, (M - 1) // 2 + 1, (M - 1) // 4 + 1]
        for name, kind, cin, cout in UNET:
            g = sizes[UNET_LEVEL[name] + (1 if kind == "up" else 0)]
            fl += 2 * 27 * cin * cout * g ** 3
            if op == "unet_grad":  # the activations the backward pass needs, kept in 16 bits
                by += 2 * 2 * cin * sizes[UNET_LEVEL[name]] ** 3
        fl *= 3 if op == "unet_grad" else 1
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ the same in plain FP64 torch
def _basis(p, nodes_only=False):
    """Values and derivatives of the Lagrange basis on the GLL nodes at the p + 1 Gauss points of [0, 1],
    and the weights; or the nodes."""
    legendre = np.polynomial.legendre
    inner = np.real(legendre.legroots(legendre.legder([0.0] * p + [1.0]))) if p > 1 else []
    nodes = (np.concatenate([[-1.0], np.sort(inner), [1.0]]) + 1) / 2
    if nodes_only:
        return nodes, None, None
    x, w = legendre.leggauss(p + 1)
    x, w = (x + 1) / 2, w / 2
    B, D = np.empty((p + 1, p + 1)), np.zeros((p + 1, p + 1))
    for i in range(p + 1):
        others = [m for m in range(p + 1) if m != i]
        scale = np.prod([nodes[i] - nodes[m] for m in others])
        B[:, i] = np.prod([x - nodes[m] for m in others], axis=0) / scale
        for j in others:
            D[:, i] += np.prod([x - nodes[m] for m in others if m != j] or [np.ones_like(x)], axis=0) / scale
    return B, D, w


class _Plain:
    """Residual, tangent product and diagonal by dense element matrices, slab by slab in z."""

    def __init__(self, case, points=1_500_000):
        self.N, self.p = case["n_el"], case["degree"]
        self.n, self.M = self.p + 1, self.p * self.N + 1
        self.n3 = self.n ** 3
        self.lam, self.split = case["lam"], case.get("model") == "split"
        B, D, w = _basis(self.p)
        h = 1.0 / self.N
        grads = [np.kron(B, np.kron(B, D)), np.kron(B, np.kron(D, B)), np.kron(D, np.kron(B, B))]
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        self.G = t(np.stack(grads) / h)                              # [3 (d), q, a]
        self.Gt = self.G.permute(2, 0, 1).reshape(self.n3, -1).contiguous()  # [a, (d, q)]
        self.wq = t(np.kron(w, np.kron(w, w)) * h ** 3)
        self.fixed = _constrained(case).reshape(-1)
        f = _factors(case) if case.get("inclusions") else torch.ones(self.N ** 3, dtype=torch.float64, device="cuda")
        self.factor = f.reshape(self.N, -1)
        layers = max(1, points // (self.N ** 2 * self.n3))
        self.slabs = [(z, min(self.N, z + layers)) for z in range(0, self.N, layers)]
        e = torch.arange(self.N, device="cuda") * self.p
        a = torch.arange(self.n, device="cuda")
        M = self.M
        line = e[:, None] + a                                         # [N, n]
        self.conn = lambda z0, z1: (line[None, None, :, None, None, :] + M * (
            line[None, :, None, None, :, None] + M * line[z0:z1, None, None, :, None, None])).reshape(-1, self.n3)

    def grad(self, vec, conn):
        """[3 (c), 3 (d), elements, points]."""
        v = vec.reshape(3, -1)[:, conn]                               # [3, E, a]
        return torch.matmul(v[:, None], self.G.transpose(1, 2)[None])

    def add(self, out, P, conn, z0, z1):
        """out += sum over points of P : Grad phi, P [3, 3, E, q]."""
        P = P * (self.wq * self.factor[z0:z1].reshape(-1, 1))
        fe = torch.matmul(P, self.G[None]).sum(dim=1)                 # [3, E, a]
        out.reshape(3, -1).index_add_(1, conn.reshape(-1), fe.reshape(3, -1))

    @staticmethod
    def inverse(F):
        cof = [[F[(j + 1) % 3][(i + 1) % 3] * F[(j + 2) % 3][(i + 2) % 3]
                - F[(j + 1) % 3][(i + 2) % 3] * F[(j + 2) % 3][(i + 1) % 3] for j in range(3)] for i in range(3)]
        J = F[0][0] * cof[0][0] + F[0][1] * cof[1][0] + F[0][2] * cof[2][0]
        return torch.stack([torch.stack(r) for r in cof]) / J, J

    def kinematics(self, u, conn):
        F = self.grad(u, conn)
        for c in range(3):
            F[c, c] += 1.0
        Fi, J = self.inverse(F)
        return F, Fi, J

    def piola(self, F, Fi, J):
        T = Fi.transpose(0, 1)
        if self.split:
            a, I1 = MU * J ** (-2.0 / 3.0), (F * F).sum((0, 1))
            return a * F + (self.lam / 2 * (J * J - 1) - a * I1 / 3) * T
        return MU * F + (2 * self.lam * torch.log(J) - MU) * T

    def stress(self, F, Fi, J, dH):
        """The derivative of piola() in the direction dH."""
        K = torch.einsum("abeq,bceq->aceq", Fi, dH)
        tr = K[0, 0] + K[1, 1] + K[2, 2]
        Q = torch.einsum("abeq,bceq->aceq", K, Fi).transpose(0, 1)    # F^-T dH^T F^-T
        T = Fi.transpose(0, 1)
        if self.split:
            a, I1, FdH = MU * J ** (-2.0 / 3.0), (F * F).sum((0, 1)), (F * dH).sum((0, 1))
            return (a * dH - 2.0 / 3.0 * a * tr * F + (2.0 / 9.0 * a * I1 * tr - 2.0 / 3.0 * a * FdH
                    + self.lam * J * J * tr) * T + (a * I1 / 3 - self.lam / 2 * (J * J - 1)) * Q)
        return MU * dH + (MU - 2 * self.lam * torch.log(J)) * Q + 2 * self.lam * tr * T

    def residual(self, u):
        r = torch.zeros_like(u)
        for z0, z1 in self.slabs:
            conn = self.conn(z0, z1)
            self.add(r, self.piola(*self.kinematics(u, conn)), conn, z0, z1)
        return r.masked_fill_(self.fixed, 0.0)

    def linearise(self, u, keep=False):
        """The tangent product at u; `keep`: the point values stay in memory."""
        kept = [(self.conn(z0, z1), self.kinematics(u, self.conn(z0, z1))) for z0, z1 in self.slabs] if keep else None

        def product(du, raw=False):
            d = du if raw else du.masked_fill(self.fixed, 0.0)
            v = torch.zeros_like(u)
            for k, (z0, z1) in enumerate(self.slabs):
                conn, kin = kept[k] if keep else (self.conn(z0, z1), None)
                kin = kin or self.kinematics(u, conn)
                self.add(v, self.stress(*kin, self.grad(d, conn)), conn, z0, z1)
            return v if raw else torch.where(self.fixed, du, v)

        return product

    def diagonal(self, u):
        out = torch.zeros_like(u)
        o = out.reshape(3, -1)
        for z0, z1 in self.slabs:
            conn = self.conn(z0, z1)
            F, Fi, J = self.kinematics(u, conn)
            s = self.wq * self.factor[z0:z1].reshape(-1, 1)
            for c in range(3):
                fe = 0.0
                for d in range(3):
                    for l in range(3):
                        dH = torch.zeros_like(F)
                        dH[c, l] = 1.0
                        L = self.stress(F, Fi, J, dH)[c, d]
                        fe = fe + torch.matmul(L * s, self.G[d] * self.G[l])
                o[c].index_add_(0, conn.reshape(-1), fe.reshape(-1))
        return out.masked_fill_(self.fixed, 1.0)

    def solve(self, product, diag, b, rtol, most=4000):
        """Conjugate gradients on the inverse diagonal; None where they take too long."""
        x, r = torch.zeros_like(b), b.clone()
        z = r / diag
        p, rz, stop = z.clone(), torch.dot(r, z), rtol * float(b.norm())
        for k in range(most):
            q = product(p)
            alpha = rz / torch.dot(p, q)
            x += alpha * p
            r -= alpha * q
            if k % 10 == 9 and float(r.norm()) <= stop:
                return x
            z = r / diag
            rz, old = torch.dot(r, z), rz
            p = z + (rz / old) * p
        return None


def _exact_newton(case, u):
    """Newton to the rounding of FP64 for one load step: the state u with K du = -R(u), u = g on the boundary."""
    m = _Plain(case)
    u = u.clone()
    g = torch.zeros_like(u)
    M = m.M
    g.reshape(3, M, M, M)[2, M - 1] = -COMPRESSION
    first = None
    for _ in range(12):
        lift = torch.where(m.fixed, g - u, torch.zeros_like(u))
        product = m.linearise(u, keep=True)
        b = torch.where(m.fixed, lift, -m.residual(u) - product(lift, raw=True))
        size = float(b.norm())
        first = first or size
        if size <= 1e-13 * first:
            break
        du = m.solve(product, m.diagonal(u), b, 1e-9)
        if du is None:
            return None
        u += du
        u = torch.where(m.fixed, g, u)
    return u


def _conv(x, W, b, stride=1):
    """3x3x3 cross-correlation with zero padding of [c, z, y, x] by 27 matrix products."""
    m = x.shape[1]
    om = m if stride == 1 else (m - 1) // 2 + 1
    xp = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    out = b[:, None].expand(-1, om ** 3)
    cut = lambda d: slice(d, d + stride * (om - 1) + 1, stride)
    for dz in range(3):
        for dy in range(3):
            for dx in range(3):
                out = out + W[:, :, dz, dy, dx] @ xp[:, cut(dz), cut(dy), cut(dx)].reshape(x.shape[0], -1)
    return out.reshape(-1, om, om, om)


def _up(y, U, b, om):
    """The adjoint of the stride-2 convolution, onto om points per direction."""
    ym, co = y.shape[1], U.shape[1]
    out = torch.zeros(co, om + 2, om + 2, om + 2, dtype=y.dtype, device=y.device)
    cut = lambda d: slice(d, d + 2 * (ym - 1) + 1, 2)
    for dz in range(3):
        for dy in range(3):
            for dx in range(3):
                t = (U[:, :, dz, dy, dx].T @ y.reshape(y.shape[0], -1)).reshape(co, ym, ym, ym)
                part = torch.zeros_like(out)
                part[:, cut(dz), cut(dy), cut(dx)] = t
                out = out + part
    return out[:, 1:-1, 1:-1, 1:-1] + b[:, None, None, None]


def _exact_unet(case, seed, inputs):
    M = case["degree"] * case["n_el"] + 1
    flat = torch.from_numpy(_unet_params(case, seed % (1 << 31))).cuda().double().requires_grad_(case["op"] == "unet_grad")
    P, at = {}, 0
    for name, kind, cin, cout in UNET:
        shape = (cin, cout, 3, 3, 3) if kind == "up" else (cout, cin, 3, 3, 3)
        P[name] = (flat[at:at + 27 * cin * cout].reshape(shape), flat[at + 27 * cin * cout:at + 27 * cin * cout + cout])
        at += 27 * cin * cout + cout
    relu = torch.relu
    with torch.set_grad_enabled(case["op"] == "unet_grad"):
        x = inputs["x"].double().reshape(3, M, M, M)
        s0 = relu(_conv(relu(_conv(x, *P["in"])), *P["e0"]))
        s1 = relu(_conv(relu(_conv(s0, *P["d1"], 2)), *P["e1"]))
        m2 = relu(_conv(relu(_conv(s1, *P["d2"], 2)), *P["m2"]))
        t1 = relu(_conv(relu(_up(m2, *P["u1"], s1.shape[1]) + s1), *P["t1"]))
        t0 = relu(_conv(relu(_up(t1, *P["u0"], M) + s0), *P["t0"]))
        y = _conv(t0, *P["out"]).reshape(-1)
        if case["op"] == "unet_forward":
            return y
        e = inputs["e"].double()
        free = (~_constrained(case).reshape(-1)).double()
        loss = ((free * (y - e)) ** 2).sum() / ((free * e) ** 2).sum()
        loss.backward()
    return {"loss": loss.detach(), "grads": flat.grad}


def exact(case, seed):
    s, op = _inputs(case, seed), case["op"]
    if op in ("unet_grad", "unet_forward"):
        return _exact_unet(case, seed, s)
    if op == "newton":
        return _exact_newton(case, s["u"])
    m = _Plain(case)
    if op == "tangent":
        return m.linearise(s["u"])(s["du"].double())
    if op == "setup":
        return {"r": m.residual(s["u"]), "d": m.diagonal(s["u"]), "v": m.linearise(s["u"])(s["du"].double())}
    if case["lam"] > 10 or case["n_el"] * case["degree"] > 72 or case["inclusions"]:
        return None  # thousands of plain conjugate-gradient iterations, or each of them long
    return m.solve(m.linearise(s["u"], keep=True), m.diagonal(s["u"]), s["du"], 1e-13)
