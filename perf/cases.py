"""Timed cases of the eHDG library, through its public Python entry points.

A case is one problem as a user's program poses it: a mesh, a degree, a scheme,
a precision. `prepare` makes the solver (local operators factored, the handle a
program keeps) and the fields on the GPU; `run` uploads boundary data and
initial state, advances the steps and fetches the volume and trace solutions.

`exact` solves the same problem in plain float64 torch, from the weak form
alone: assembly by quadrature, a dense inverse, Algorithm 1 to the same
tolerance.
"""
import math

import numpy as np
import torch

from paper_1601_06681_gb300 import ehdg

# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------


def _solve(name, kind, n, p, steps, dt, scheme="be", precision="fp64", inner=0, outer=False,
           tol=1e-10):
    n = tuple(n) + (0,) * (3 - len(n))
    return {"name": name, "kind": kind, "n0": n[0], "n1": n[1], "n2": n[2], "p": p, "steps": steps,
            "dt": dt, "scheme": scheme, "precision": precision, "inner": inner, "outer": outer,
            "tol": tol}


def _batch(name, count, mix, steps, precision, inner=0):
    return {"name": name, "kind": "batch", "count": count, "mix": mix, "steps": steps,
            "precision": precision, "inner": inner}


def listed():
    return [
        # the smallest call a program makes: a coarse 2D run, ten steps
        _solve("transport2d_16_p2", "transport", (16, 16), 2, 10, 0.01),
        # an ordinary 2D run on a ragged mesh, one velocity for all elements
        _solve("transport2d_253x187_p4_cn", "transport", (253, 187), 4, 10, 2e-3, scheme="cn"),
        # the 2D variable-velocity benchmark: one local operator per element
        _solve("varbeta2d_256_p4_cn", "varbeta", (256, 256), 4, 10, 2e-3, scheme="cn"),
        # a steady solve with per-element operators, BF16 corrections
        _solve("steady2d_160_p4_bf16", "steady", (160, 160), 4, 1, 1.0, scheme="steady",
               precision="bf16", inner=8),
        # the shallow-water benchmark in FP64
        _solve("sw2d_512_p3", "sw", (512, 512), 3, 10, 2.5e-5),
        # shallow water on a ragged mesh, mixed precision
        _solve("sw2d_301x170_p2_tf32", "sw", (301, 170), 2, 10, 7e-5, precision="tf32", inner=3,
               outer=True),
        # the headline: 3D transport in FP64
        _solve("transport3d_64_p3", "transport", (64, 64, 64), 3, 2, 5e-3),
        # a small odd 3D run, Crank-Nicolson
        _solve("transport3d_17x12x9_p2_cn", "transport", (17, 12, 9), 2, 4, 1e-2, scheme="cn"),
        # the headline's mixed-precision form, at the tolerance of matched accuracy
        _solve("transport3d_64_p3_tf32", "transport", (64, 64, 64), 3, 4, 5e-3, precision="tf32",
               inner=14, outer=True, tol=3e-12),
        # FP64-accurate products on the tensor cores, ragged 3D mesh
        _solve("transport3d_37x29x31_p3_emulated", "transport", (37, 29, 31), 3, 2, 5e-3,
               precision="fp64_emulated"),
        # many small independent problems served together
        _batch("batch_48_fp64", 48, 11, 4, "fp64"),
        _batch("batch_48_tf32", 48, 12, 4, "tf32", 8),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["transport2", "transport2", "transport3", "transport3", "transport3", "varbeta",
                       "steady", "sw", "sw", "batch"])
    scheme = rng.choice(["be", "cn"])
    if kind == "transport2":
        n = (_log_int(rng, 8, 300), _log_int(rng, 8, 300))
        c = _solve("", "transport", n, rng.randint(1, 6), rng.randint(2, 10), rng.uniform(1e-3, 1e-2),
                   scheme=scheme, precision=rng.choice(["fp64", "fp64", "fp32", "tf32"]))
        c["inner"] = 0 if c["precision"] == "fp64" else rng.choice([4, 8])
    elif kind == "transport3":
        n = [_log_int(rng, 4, 56) for _ in range(3)]
        pr = rng.choice(["fp64", "fp64", "tf32", "bf16", "fp64_emulated"])
        mixed = pr in ("tf32", "bf16")
        c = _solve("", "transport", n, rng.randint(1, 3), 2, rng.uniform(2e-3, 1e-2), scheme=scheme,
                   precision=pr, inner=rng.choice([8, 12]) if mixed else 0, outer=mixed)
    elif kind == "varbeta":
        n = (_log_int(rng, 12, 256), _log_int(rng, 12, 256))
        c = _solve("", "varbeta", n, rng.randint(1, 5), rng.randint(2, 8), rng.uniform(1e-3, 4e-3),
                   scheme=scheme, precision=rng.choice(["fp64", "fp64", "bf16"]))
        c["inner"] = 0 if c["precision"] == "fp64" else 8
    elif kind == "steady":
        n = (_log_int(rng, 12, 160), _log_int(rng, 12, 160))
        c = _solve("", "steady", n, rng.randint(1, 4), 1, 1.0, scheme="steady",
                   precision=rng.choice(["fp64", "bf16"]))
        c["inner"] = 0 if c["precision"] == "fp64" else 8
    elif kind == "sw":
        n = (_log_int(rng, 12, 480), _log_int(rng, 12, 480))
        p = rng.randint(1, 5)
        dt = 1.0 / (max(n) * (p + 1) * (p + 2) * rng.uniform(3.0, 6.0))
        c = _solve("", "sw", n, p, rng.randint(2, 8), dt, scheme="be",
                   precision=rng.choice(["fp64", "fp64", "tf32", "fp64_emulated"]))
        if c["precision"] == "tf32":
            c["inner"], c["outer"] = 3, True
    else:
        c = _batch("", rng.randint(8, 48), rng.randint(1, 1 << 20), 4,
                   rng.choice(["fp64", "fp32", "tf32"]))
        c["inner"] = 0 if c["precision"] == "fp64" else 8
    del c["name"]
    return c


# --------------------------------------------------------------------------
# meshes, nodes and fields
# --------------------------------------------------------------------------


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gll(p):
    P = np.polynomial.legendre.Legendre.basis(p)
    x = np.concatenate(([-1.0], np.sort(np.real(P.deriv().roots())) if p > 1 else [], [1.0]))
    for _ in range(4 if p > 1 else 0):
        x[1:-1] -= P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1])
    return x


def _points(case):
    p = case["p"]
    return (3 * p + 1) // 2 + 1 if case["kind"] in ("varbeta", "steady") else p + 1


def _sizes(case):
    return tuple(v for v in (case["n0"], case["n1"], case["n2"]) if v)


def _tensor_points(r, dim):
    """[len(r)^dim, dim], axis 0 fastest."""
    g = np.meshgrid(*([r] * dim), indexing="ij")
    return np.stack([v.reshape(-1, order="F") for v in g], -1)


class _Grid:
    """Connectivity and geometry of the structured mesh of the unit box, with
    the library's numbering: elements and, axis by axis, faces, axis 0 fastest."""

    def __init__(self, n, dev):
        self.n, self.dim, self.dev = n, len(n), dev
        d = self.dim
        self.nel = int(np.prod(n))
        self.h = [1.0 / v for v in n]
        e = torch.arange(self.nel, device=dev)
        idx, rem = [], e
        for a in range(d):
            idx.append(rem % n[a])
            rem = rem // n[a]
        self.lo = torch.stack([idx[a].double() * self.h[a] for a in range(d)], -1)
        self.elem_face = torch.empty((self.nel, 2 * d), dtype=torch.int64, device=dev)
        base = 0
        for ax in range(d):
            shape = [n[a] + (a == ax) for a in range(d)]
            for side in (0, 1):
                f, stride = 0, 1
                for a in range(d):
                    f = f + (idx[a] + (side if a == ax else 0)) * stride
                    stride *= shape[a]
                self.elem_face[:, 2 * ax + side] = base + f
            base += int(np.prod(shape))
        self.nface = base
        # the element and local face on the minus (low) side, and on the plus side
        self.minus = torch.full((base,), -1, dtype=torch.int64, device=dev)
        self.plus = torch.full((base,), -1, dtype=torch.int64, device=dev)
        for ax in range(d):
            self.minus[self.elem_face[:, 2 * ax + 1]] = e * 2 * d + 2 * ax + 1
            self.plus[self.elem_face[:, 2 * ax]] = e * 2 * d + 2 * ax
        only = self.minus < 0
        self.minus[only] = self.plus[only]
        self.plus[only] = -1

    def nodes(self, p):
        r = torch.from_numpy((_tensor_points(_gll(p), self.dim) + 1.0) / 2.0).to(self.dev)
        return self.lo[:, None, :] + torch.tensor(self.h, dtype=torch.float64, device=self.dev) * r

    def face_points(self, q):
        d, xi = self.dim, np.polynomial.legendre.leggauss(q)[0]
        el, lf = self.minus // (2 * d), self.minus % (2 * d)
        t = _tensor_points(xi, d - 1)
        ref = np.empty((2 * d, t.shape[0], d))
        for f in range(2 * d):
            ax, side = divmod(f, 2)
            ref[f, :, [a for a in range(d) if a != ax]] = t.T
            ref[f, :, ax] = 2.0 * side - 1.0
        ref = torch.from_numpy((ref + 1.0) / 2.0).to(self.dev)
        return self.lo[el][:, None, :] + torch.tensor(self.h, dtype=torch.float64, device=self.dev) * ref[lf]


def _gaussian(x, c, s):
    c = torch.as_tensor(np.asarray(c), dtype=torch.float64, device=x.device)
    return torch.exp(-((x - c) ** 2).sum(-1) / (2.0 * s * s))


def _velocity(x, rng):
    """0.5 (cos 2 pi y, sin 2 pi x) plus eight small random Fourier modes per component."""
    out = torch.stack([0.5 * torch.cos(2 * math.pi * x[..., 1]), 0.5 * torch.sin(2 * math.pi * x[..., 0])], -1)
    for c in range(2):
        for _ in range(8):
            k, th = rng.integers(1, 5, 2), rng.uniform(0, 2 * math.pi)
            out[..., c] += 0.05 / 8 * torch.cos(2 * math.pi * (k[0] * x[..., 0] + k[1] * x[..., 1]) + th)
    return out


def _problem(case, seed, dev):
    """The fields of one problem: dict(grid, u0, g, beta, beta_nodes, force)."""
    rng = np.random.default_rng(seed)
    grid = _Grid(_sizes(case), dev)
    d, kind = grid.dim, case["kind"]
    x, xf = grid.nodes(case["p"]), grid.face_points(_points(case))
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) + 7919)
    out = {"grid": grid, "beta": None, "beta_nodes": None, "force": None}
    if kind == "sw":
        u0 = torch.zeros((grid.nel, 3, x.shape[1]), dtype=torch.float64, device=dev)
        for _ in range(16):
            amp = math.cos(rng.uniform(0, 2 * math.pi))
            u0[:, 0] += amp * _gaussian(x, rng.uniform(0.1, 0.9, 2), rng.uniform(0.02, 0.08))
        g = torch.zeros(xf.shape[:-1], dtype=torch.float64, device=dev)
    elif kind == "steady":
        u0 = torch.zeros((grid.nel, 1, x.shape[1]), dtype=torch.float64, device=dev)
        a = math.pi * rng.uniform(0.9, 1.1)
        g = torch.sin(a * xf[..., 0]) * torch.cos(a * xf[..., 1]) / a
        out["force"] = (x[..., 1] * torch.cos(a * x[..., 0]) * torch.cos(a * x[..., 1])
                        - x[..., 0] * torch.sin(a * x[..., 0]) * torch.sin(a * x[..., 1]))[:, None, :].contiguous()
        out["beta_nodes"] = torch.stack([x[..., 1], x[..., 0]], 1).contiguous()
    else:
        c, s = rng.uniform(0.2, 0.6, d), rng.uniform(0.07, 0.13)
        noise = 1e-3 * (2.0 * torch.rand(x.shape[:-1], generator=gen, dtype=torch.float64, device=dev) - 1.0)
        u0 = (_gaussian(x, c, s) + noise)[:, None, :].contiguous()
        g = _gaussian(xf, c, s)
        if kind == "varbeta":
            out["beta_nodes"] = _velocity(x, rng).transpose(1, 2).contiguous()
        else:
            # a random direction without a vanishing component
            b = rng.uniform(0.3, 1.0, d) * rng.choice([-1.0, 1.0], d)
            out["beta"] = rng.uniform(0.8, 1.2) * b / np.linalg.norm(b)
    out["u0"], out["g"] = u0, g.contiguous()
    return out


def _instances(case):
    """The batch's problems as single cases: sides 8..128 (log-uniform), p 1..5."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["count"]):
        n, p = int(round(8 * 16 ** rng.uniform())), int(rng.integers(1, 6))
        c = _solve("", "transport", (n, n), p, case["steps"], 0.01, precision=case["precision"],
                   inner=case["inner"])
        out.append(c)
    return out


def _solver_args(case, f):
    kw = dict(p=case["p"], pde="sw" if case["kind"] == "sw" else "transport", scheme=case["scheme"],
              dt=case["dt"], tol=case["tol"], max_iter=2000, precision=case["precision"],
              inner_sweeps=case["inner"], emulated_outer=case["outer"])
    if f["beta"] is not None:
        kw["beta_const"] = f["beta"]
    if f["beta_nodes"] is not None:
        kw["beta_nodes"] = f["beta_nodes"].cpu().numpy()
    kw["mesh"] = ehdg.ehdg_mesh_structured(
        _sizes(case), boundary_tag=ehdg.FACE_WALL if case["kind"] == "sw" else ehdg.FACE_DIRICHLET)
    return kw


def prepare(case, seed):
    dev = _dev()
    if case["kind"] == "batch":
        fields, problems = [], []
        for i, c in enumerate(_instances(case)):
            f = _problem(c, seed * 1000 + i, dev)
            problems.append(_solver_args(c, f))
            fields.append((f["u0"], f["g"]))
        b = ehdg.Batch(problems)
        sizes = [(s.info["state_len"], s.info["trace_len"]) for s in b.instances]
        u = torch.empty(sum(v[0] for v in sizes), dtype=torch.float64, device=dev)
        uh = torch.empty(sum(v[1] for v in sizes), dtype=torch.float64, device=dev)
        outs, i, j = [], 0, 0
        for s, t in sizes:
            outs.append((u[i:i + s], uh[j:j + t]))
            i, j = i + s, j + t
        return {"case": case, "batch": b, "fields": fields, "outs": outs, "u": u, "uhat": uh}
    f = _problem(case, seed, dev)
    kw = _solver_args(case, f)
    sol = ehdg.Solver(kw.pop("mesh"), **kw)
    return {"case": case, "solver": sol, "u0": f["u0"], "g": f["g"], "force": f["force"],
            "u": torch.empty(sol.state_shape, dtype=torch.float64, device=dev),
            "uhat": torch.empty(sol.trace_shape, dtype=torch.float64, device=dev)}


def run(state):
    case = state["case"]
    if "batch" in state:
        b = state["batch"]
        for s, (u0, g) in zip(b.instances, state["fields"]):
            s.set_boundary(g)
            s.set_state(u0)
        iters, _ = b.run(case["steps"])
        for s, (u, uh) in zip(b.instances, state["outs"]):
            s.get_state(u, uh)
        return {"u": state["u"], "uhat": state["uhat"], "iterations": iters}
    sol = state["solver"]
    sol.set_boundary(state["g"])
    if state["force"] is not None:
        sol.set_forcing(state["force"])
    sol.set_state(state["u0"])
    iters = sol.run(case["steps"])
    sol.get_state(state["u"], state["uhat"])
    return {"u": state["u"], "uhat": state["uhat"], "iterations": np.asarray(iters, dtype=np.int64)}


def work(case):
    """Bytes: the state in and out, the boundary data of the box's faces in and
    the trace out. Operations: one element solve per step at the least, on the
    tensor-product space (p + 2 products per volume value and axis)."""
    if case["kind"] == "batch":
        ws = [work(c) for c in _instances(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    n, p, q = _sizes(case), case["p"], _points(case)
    d, nel = len(n), int(np.prod(n))
    nf = 3 if case["kind"] == "sw" else 1
    nface = sum(nel // n[a] * (n[a] + 1) for a in range(d))
    bface = sum(2 * nel // n[a] for a in range(d))
    values, points = nel * nf * (p + 1) ** d, q ** (d - 1)
    nbytes = 8 * (2 * values + nface * points + bface * points)
    if case["kind"] in ("varbeta", "steady"):
        nbytes += 8 * nel * d * (p + 1) ** d
    return {"bytes": nbytes, "flops": 2 * case["steps"] * values * d * (p + 2)}


# --------------------------------------------------------------------------
# the same problems in plain float64 torch
# --------------------------------------------------------------------------


def _kron(mats):
    out = mats[0]
    for m in mats[1:]:
        out = np.einsum("ga,hb->hgba", out, m).reshape(out.shape[0] * m.shape[0], -1)
    return out


def _lagrange(r, x):
    L, D = np.ones((len(x), len(r))), np.zeros((len(x), len(r)))
    for a in range(len(r)):
        for b in range(len(r)):
            if b != a:
                L[:, a] *= (x - r[b]) / (r[a] - r[b])
        for m in range(len(r)):
            if m != a:
                t = np.full(len(x), 1.0 / (r[a] - r[m]))
                for b in range(len(r)):
                    if b not in (a, m):
                        t = t * (x - r[b]) / (r[a] - r[b])
                D[:, a] += t
    return L, D


def _operators(case, f):
    """(P, H, E, Hy, weights): u = P w + H uhat for one element (or a batch of
    them), E the face-point values the trace formula reads, Hy = E H."""
    grid, p, q, kind = f["grid"], case["p"], _points(case), case["kind"]
    d, dev = grid.dim, grid.dev
    r, (xi, om) = _gll(p), np.polynomial.legendre.leggauss(q)
    L, D = _lagrange(r, xi)
    ends = [np.eye(1, p + 1, 0), np.eye(1, p + 1, p)]
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    phi = _kron([L] * d)
    W = _kron([om[:, None]] * d)[:, 0] * np.prod([h / 2 for h in grid.h])
    grads = [_kron([D if a == ax else L for a in range(d)]) * 2.0 / grid.h[ax] for ax in range(d)]
    fphi, fw = [], []
    for k in range(2 * d):
        ax, side = divmod(k, 2)
        fphi.append(_kron([ends[side] if a == ax else L for a in range(d)]))
        fw.append(_kron([om[:, None]] * (d - 1))[:, 0] * np.prod([grid.h[a] / 2 for a in range(d) if a != ax]))
    M = phi.T @ (W[:, None] * phi)
    Np, coef = phi.shape[1], 0.0
    if case["scheme"] != "steady":
        coef = 1.0 / (case["dt"] * (0.5 if case["scheme"] == "cn" else 1.0))
    if kind == "sw":
        Z = np.zeros_like(M)
        G = [g.T @ (W[:, None] * phi) for g in grads]
        Mb = np.block([[M, Z, Z], [Z, M, Z], [Z, Z, M]])
        A = coef * Mb + np.block([[Z, -G[0], -G[1]], [-G[0], Z, Z], [-G[1], Z, Z]])
        B, E = [], []
        for k in range(4):
            ax, s = k // 2, 2.0 * (k % 2) - 1.0
            Ef, Bf = fphi[k].T @ (fw[k][:, None] * fphi[k]), fphi[k].T * fw[k]
            A[:Np, :Np] += Ef
            A[:Np, (1 + ax) * Np:(2 + ax) * Np] += s * Ef
            col = [Bf, np.zeros_like(Bf), np.zeros_like(Bf)]
            col[1 + ax] = -s * Bf
            B.append(np.concatenate(col, 0))
            row = [0.5 * fphi[k], np.zeros_like(fphi[k]), np.zeros_like(fphi[k])]
            row[1 + ax] = 0.5 * s * fphi[k]
            E.append(np.concatenate(row, 1))
        A, B, E = T(A), T(np.concatenate(B, 1)), T(np.concatenate(E, 0))
        M = T(Mb)
    else:
        E = T(np.concatenate(fphi, 0))
        if f["beta"] is not None:
            b = torch.as_tensor(f["beta"], dtype=torch.float64, device=dev)
            beta = b[None, :, None].expand(1, d, Np)
        else:
            beta = f["beta_nodes"]
        A = coef * T(M)[None].repeat(beta.shape[0], 1, 1)
        B = torch.zeros((beta.shape[0], Np, 2 * d * fphi[0].shape[0]), dtype=torch.float64, device=dev)
        pp = T(np.einsum("qi,qj->qij", phi, phi).reshape(len(W), -1))
        for ax in range(d):
            gp = T(np.einsum("qi,qj->qij", grads[ax], phi).reshape(len(W), -1))
            bq, dbq = beta[:, ax] @ T(phi).T, beta[:, ax] @ T(grads[ax]).T
            A -= ((bq * T(W)) @ gp + (dbq * T(W)) @ pp).view_as(A)
        nq = fphi[0].shape[0]
        for k in range(2 * d):
            ax, s = k // 2, 2.0 * (k % 2) - 1.0
            bn = s * (beta[:, ax] @ T(fphi[k]).T)
            ff = T(np.einsum("qi,qj->qij", fphi[k], fphi[k]).reshape(nq, -1))
            A += (((bn + bn.abs()) * T(fw[k])) @ ff).view_as(A)
            B[:, :, k * nq:(k + 1) * nq] = T(fphi[k]).T[None] * (bn.abs() * T(fw[k]))[:, None, :]
        M = T(M)[None]
        if A.shape[0] == 1:
            A, B, M = A[0], B[0], M[0]
    P, H = torch.linalg.solve(A, M.expand_as(A)), torch.linalg.solve(A, B)
    return P, H, E, E @ H, coef, [T(w) for w in fw]


def _exact(case, f):
    grid, kind, cn = f["grid"], case["kind"], case["scheme"] == "cn"
    d, F = grid.dim, 2 * grid.dim
    P, H, E, Hy, coef, fw = _operators(case, f)
    many = P.dim() == 3
    mul = (lambda A, x: torch.bmm(A, x[..., None])[..., 0]) if many else (lambda A, x: x @ A.T)
    nq, inner = E.shape[0] // F, grid.plus >= 0
    lf = grid.minus % F
    w = torch.stack(fw)[lf]
    minus, plus = grid.minus, grid.plus.clamp(min=0)
    if kind != "sw":
        if f["beta"] is not None:
            bn = torch.as_tensor(f["beta"], device=grid.dev)[lf // 2] * (2.0 * (lf % 2) - 1.0)
            bn = bn[:, None].expand(-1, nq)
        else:
            bp = torch.stack([f["beta_nodes"][:, k // 2] @ E[k * nq:(k + 1) * nq].T * (2.0 * (k % 2) - 1.0)
                              for k in range(F)], 1).reshape(-1, nq)
            bn = bp[minus]
        up = torch.where(bn > 0, 1.0, torch.where(bn < 0, 0.0, 0.5)).double()
    g = f["g"]

    def trace(Y):
        Y = Y.reshape(-1, nq)
        m = Y[minus]
        if kind == "sw":
            return m + torch.where(inner[:, None], Y[plus], m)
        return up * m + (1.0 - up) * torch.where(inner[:, None], Y[plus], g)

    gather = lambda uh: uh[grid.elem_face].reshape(grid.nel, F * nq)  # noqa: E731
    u = f["u0"].reshape(grid.nel, -1)
    uh_n = trace(u @ E.T)
    tol = case["tol"] if case["precision"] in ("fp64", "fp64_emulated") else case["tol"] / 30.0
    iters = []
    for _ in range(case["steps"]):
        rhs = coef * u + (0.0 if f["force"] is None else f["force"].reshape(grid.nel, -1))
        G = mul(P, rhs)
        Gy, uh, k = G @ E.T, trace(u @ E.T), 0
        while True:
            last = gather(uh)
            new = trace(Gy + mul(Hy, last))
            res = float(((new - uh) ** 2 * w).sum().sqrt()) * (2.0 if cn else 1.0)
            uh, k = new, k + 1
            if not res >= tol or k >= 2000:
                break
        v = G + mul(H, last)
        u, uh_n = (2 * v - u, 2 * uh - uh_n) if cn else (v, uh)
        iters.append(k)
    same = case["precision"] in ("fp64", "fp64_emulated")
    return u.reshape(f["u0"].shape), uh_n, torch.tensor(iters) if same else None


def exact(case, seed):
    dev = _dev()
    if case["kind"] == "batch":
        got = [_exact(c, _problem(c, seed * 1000 + i, dev)) for i, c in enumerate(_instances(case))]
        same = case["precision"] == "fp64"
        return {"u": torch.cat([v[0].reshape(-1) for v in got]), "uhat": torch.cat([v[1].reshape(-1) for v in got]),
                "iterations": torch.stack([v[2] for v in got]).int() if same else None}
    if case["kind"] == "varbeta" and case["p"] >= 5 and case["n0"] * case["n1"] > 40000:
        return None
    u, uh, it = _exact(case, _problem(case, seed, dev))
    return {"u": u, "uhat": uh, "iterations": it}
