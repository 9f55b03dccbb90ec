"""The workloads whose speed is followed: what a user of this library has it do.

Each case is one pass through the public entry points of
``paper_2202_12477_gb300.hb``: the operator ``Mesh.apply_A``, the solvers
``Mesh.cg``, building a ``Mesh``, and the solver ``Server``. Sizes are those of
this repository's benchmark and tests: the small cube of 4x4x4 elements, the
degree sweep (about 1.28e8 element-local nodes per mesh), the mixed-precision
cube of 24x24x24 elements and the serving stream (cubes of 2..16 elements per
axis, odd degrees 3..11).

``exact`` evaluates the same operator in plain torch and numpy, FP64, from the
definitions (GLL basis, trilinear elements, Z^T S_L Z + lambda).
"""
import os

import numpy as np
import torch

from paper_2202_12477_gb300 import hb

# the server asks for it (two streams per slot); read when the CUDA context is made
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

PRECS = {"f64": hb.HB_F64, "f32": hb.HB_F32, "f64x": hb.HB_F64X, "mixed": hb.HB_MIXED}
LOCAL_MAX = 1.28e8  # element-local nodes of the degree sweep's meshes


def _case(op, dims, N, **kw):
    c = dict(op=op, ex=dims[0], ey=dims[1], ez=dims[2], N=N, prec="f64", screen=0, lam=0.1, faces=0x3F,
             perturb=0.1, tuned=False, its=0, precond=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one operator application on the latency-bound cube, as an outer solver makes it
        _case("apply", (4, 4, 4), 7, name="ax_f64_n7_cube4"),
        # the degree sweep, FP64, kernels chosen by the autotuner as the benchmark does: lowest and highest
        # degree of the figures, the second with mass screening
        _case("apply", (128, 128, 122), 3, name="ax_f64_n3_sweep", tuned=True),
        _case("apply", (64, 64, 61), 7, name="ax_f64_n7_sweep", tuned=True),
        _case("apply", (32, 32, 30), 15, name="ax_f64_n15_sweep", tuned=True, screen=1),
        # the FP32 operator inside the mixed-precision solver, full size
        _case("apply", (64, 64, 61), 7, name="ax_f32_n7_sweep", prec="f32", tuned=True),
        # the same on an uneven box, odd line length, Dirichlet conditions on three faces, no tuning
        _case("apply", (23, 17, 19), 10, name="ax_f32_n10_ragged", prec="f32", screen=1, faces=0x15),
        # the double-float operator in a middling size
        _case("apply", (24, 25, 23), 11, name="ax_f64x_n11", prec="f64x"),
        # 100 iterations on the small cube: the solver's latency
        _case("cg", (4, 4, 4), 7, name="cg_f64_n7_cube4", its=100),
        # the headline benchmark: CG iterations on the sweep's box at N = 7
        _case("cg", (64, 64, 61), 7, name="cg_f64_n7_sweep", its=10, tuned=True),
        # a whole mixed-precision solve to a true residual of 1e-10, with the Jacobi preconditioner
        _case("cg", (24, 24, 24), 15, name="solve_mixed_n15_cube24", prec="mixed", precond=1),
        # a new mesh at full set-up cost, as every served request and every remeshing program pays it
        _case("mesh", (32, 32, 31), 11, name="mesh_n11"),
        # a burst of requests through the server
        _case("serve", (2, 16, 24), 0, name="serve_24", prec="mixed"),
    ]


def _dims(rng, N, lo, hi):
    """A box of about lo..hi local nodes (log-uniform), its axes up to a factor 1.4 apart, at least 2 each."""
    E = max(8.0, float(np.exp(rng.uniform(np.log(lo), np.log(hi)))) / (N + 1) ** 3)
    a, b = rng.uniform(0.85, 1.18), rng.uniform(0.85, 1.18)
    side = E ** (1.0 / 3.0)
    ex, ey = max(2, round(side * a)), max(2, round(side * b))
    return ex, ey, max(2, int(E / (ex * ey)))


def draw(rng):
    op = rng.choice(["apply", "apply", "apply", "apply", "cg", "cg", "cg", "mesh", "serve"])
    N = rng.choice([3, 5, 7, 7, 9, 11, 15, rng.randint(1, 15)])
    kw = dict(screen=rng.choice([0, 0, 1]), faces=rng.choice([0x3F, 0x3F, 0x15, 0x07]),
              lam=rng.choice([0.1, 0.7, 10.0]), perturb=rng.choice([0.05, 0.1, 0.15]))
    if op == "apply":
        prec = rng.choice(["f64", "f64", "f32", "f32", "f64x"])
        dims = _dims(rng, N, 2e3, LOCAL_MAX)
        # a program that applies the operator often to a mesh of size tunes it
        big = dims[0] * dims[1] * dims[2] * (N + 1) ** 3 > 4e6
        return _case("apply", dims, N, prec=prec, tuned=big and rng.random() < 0.7, **kw)
    if op == "cg":
        if rng.random() < 0.5:
            return _case("cg", _dims(rng, N, 2e3, 3e7), N, its=rng.randint(10, 40), precond=rng.choice([0, 0, 1]),
                         tuned=rng.random() < 0.5, **kw)
        return _case("cg", _dims(rng, N, 2e4, 5e7), N, prec="mixed", precond=rng.choice([0, 1]), **kw)
    if op == "mesh":
        return _case("mesh", _dims(rng, N, 2e4, 6e7), N, **{**kw, "prec": rng.choice(["f64", "f32"])})
    return _case("serve", (2, rng.randint(6, 16), rng.randint(4, 24)), 0, prec="mixed", lam=0.1)


# ---------------------------------------------------------------- what a program holds, and one pass


def _vector(n, seed, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(seed * 7919 + 13)
    return torch.rand(n, dtype=dtype, device="cuda", generator=g).mul_(2.0).sub_(1.0)


def _requests(case, seed):
    """The burst of a "serve" case: ez cubes of ex..ey elements per axis, odd degrees 3..11."""
    r = np.random.Generator(np.random.PCG64([case["ex"], case["ey"], case["ez"]]))
    return [dict(ek=int(r.integers(case["ex"], case["ey"] + 1)), N=int(r.choice([3, 5, 7, 9, 11])),
                 seed=(seed * 1000 + i) % (1 << 40)) for i in range(case["ez"])]


def _mesh(case, seed):
    return hb.Mesh(case["ex"], case["ey"], case["ez"], case["N"], perturb=case["perturb"], seed=seed,
                   faces=case["faces"], fp32=case["prec"] in ("f32", "mixed"))


def prepare(case, seed):
    if case["op"] == "mesh":
        return {"case": case, "seed": seed}
    if case["op"] == "serve":
        return {"case": case, "requests": _requests(case, seed),
                "server": hb.Server(16 << 30, max_slots=16, iters_per_launch=16)}
    m = _mesh(case, seed)
    prec = PRECS[case["prec"]]
    if case["tuned"]:
        hb.hb_autotune(m.handle, prec, case["screen"], case["lam"], reps=2)
    x = _vector(m.n_global, seed, torch.float32 if prec == hb.HB_F32 else torch.float64)
    s = {"case": case, "mesh": m, "x": x, "prec": prec}
    s["y"] = torch.empty_like(x)  # A x, or the solution
    return s


class _View:
    """An array of a mesh as torch sees it; the mesh lives as long as its views."""

    def __init__(self, mesh, ptr, n, kind):
        self.mesh = mesh
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": kind, "data": (ptr, False), "version": 2}


def _mesh_arrays(m):
    def view(ptr, n, kind):
        return torch.as_tensor(_View(m, ptr, n, kind), device="cuda")
    i = m.info
    out = {"l2g": view(i.l2g, i.n_local, "<i4"), "geo": view(i.geo, 7 * i.n_local, "<f8"),
           "rowptr": view(i.csr_rowptr, i.n_global + 1, "<i4"), "cols": view(i.csr_cols, i.nnz, "<i4")}
    if i.geo32:
        out["geo32"] = view(i.geo32, 7 * i.n_local, "<f4")
    return out


def run(state):
    c = state["case"]
    if c["op"] == "apply":
        return state["mesh"].apply_A(state["x"], state["y"], lam=c["lam"], screen=c["screen"], prec=state["prec"])
    if c["op"] == "cg":
        x = state["y"].zero_()
        tol = 1e-10 if c["prec"] == "mixed" else 0.0
        state["mesh"].cg(state["x"], x, lam=c["lam"], rtol=tol, max_it=c["its"] or 5000, prec=state["prec"],
                         screen=c["screen"], precond=c["precond"])
        return x
    if c["op"] == "mesh":
        return _mesh_arrays(_mesh(c, state["seed"]))
    srv = state["server"]
    tickets = [srv.submit(q["ek"], q["ek"], q["ek"], q["N"], perturb=c["perturb"], seed=q["seed"],
                          rhs_seed=q["seed"], lam=c["lam"], rtol=1e-10, keep_x=True) for q in state["requests"]]
    return [srv.wait(t, (q["N"] * q["ek"] - 1) ** 3, interval=0.0001)[1]
            for t, q in zip(tickets, state["requests"])]


# ---------------------------------------------------------------- what a pass cannot do without


def _counts(c):
    f, N = c["faces"], c["N"]
    E = c["ex"] * c["ey"] * c["ez"]
    ng = 1
    for ax, e in enumerate((c["ex"], c["ey"], c["ez"])):
        ng *= N * e + 1 - ((f >> (2 * ax)) & 1) - ((f >> (2 * ax + 1)) & 1)
    return E, E * (N + 1) ** 3, ng


def work(case):
    """Bytes: factors and node map read once per application, x read and y written once; a CG iteration also
    reads and writes its three other vectors once (x, r, p; A p is used up). Flops: 12 n^4 + 18 n^3 per element
    and application (contractions, metric, gather), 10 per DOF and iteration."""
    if case["op"] == "serve":
        t = [work(dict(case, op="cg", ex=q["ek"], ey=q["ek"], ez=q["ek"], N=q["N"])) for q in _requests(case, 0)]
        return {k: sum(w[k] for w in t) for k in ("bytes", "flops")}
    E, nl, ng = _counts(case)
    n = case["N"] + 1
    if case["op"] == "mesh":
        # node map, factors (and their FP32 copy), gather rows written once; 70 operations per node
        return {"bytes": nl * (4 + 56 + (28 if case["prec"] == "f32" else 0) + 4) + 4.0 * ng, "flops": 70.0 * nl}
    esz = 4 if case["prec"] in ("f32", "mixed") else 8
    op_b = nl * (4 + esz * (7 if case["screen"] else 6)) + 2 * esz * ng
    op_f = E * (12.0 * n ** 4 + 18.0 * n ** 3)
    if case["op"] == "apply":
        return {"bytes": op_b, "flops": op_f}
    its = case["its"] or 30  # a solve at these screenings takes some tens of iterations
    return {"bytes": its * (op_b + 6.0 * esz * ng), "flops": its * (op_f + 10.0 * ng)}


# ---------------------------------------------------------------- the same in plain FP64 torch


def _u01(seed, stream, idx):
    """splitmix64 of (seed ^ stream G) + idx as a uniform number in [0, 1)."""
    G = 0x9E3779B97F4A7C15
    with np.errstate(over="ignore"):
        z = np.asarray(idx, dtype=np.uint64) + np.uint64((seed ^ (stream * G % (1 << 64))) % (1 << 64)) + np.uint64(G)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _gll(N):
    L = np.polynomial.legendre.Legendre.basis(N)
    inner = np.sort(L.deriv().roots().real) if N > 1 else np.zeros(0)
    for _ in range(3):
        if N > 1:
            inner = inner - L.deriv()(inner) / L.deriv(2)(inner)
    xi = np.concatenate([[-1.0], inner, [1.0]])
    xi = 0.5 * (xi - xi[::-1])
    P = L(xi)
    w = 2.0 / (N * (N + 1) * P * P)
    D = np.zeros((N + 1, N + 1))
    for i in range(N + 1):
        for j in range(N + 1):
            if i != j:
                D[i, j] = P[i] / (P[j] * (xi[i] - xi[j]))
    D[0, 0], D[N, N] = -N * (N + 1) / 4.0, N * (N + 1) / 4.0
    return xi, w, D


class _Plain:
    """Node map, factors and operator of a box mesh, element chunks at a time."""

    def __init__(self, ex, ey, ez, N, perturb, seed, faces, keep=True):
        dev, n = "cuda", N + 1
        self.N, self.n, self.E, self.dims = N, n, ex * ey * ez, (ex, ey, ez)
        xi, w, D = _gll(N)
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.D, self.w = t(D), t(w)
        self.phi = t(np.stack([(1 - xi) / 2, (1 + xi) / 2]))  # [2][n]
        vz, vy, vx = np.meshgrid(np.arange(ez + 1), np.arange(ey + 1), np.arange(ex + 1), indexing="ij")
        inside = (vx > 0) & (vx < ex) & (vy > 0) & (vy < ey) & (vz > 0) & (vz < ez)
        V = np.empty(vx.shape + (3,))
        vid = vx + (ex + 1) * (vy + (ey + 1) * vz)
        for ax, (q, e) in enumerate(((vx, ex), (vy, ey), (vz, ez))):
            move = (2.0 * _u01(seed, 1, 3 * vid + ax) - 1.0) * perturb / e
            V[..., ax] = q / e + np.where(inside, move, 0.0)
        self.V = t(V)
        lo = [(faces >> (2 * a)) & 1 for a in range(3)]
        hi = [(faces >> (2 * a + 1)) & 1 for a in range(3)]
        self.lo, self.nu = lo, [N * e + 1 - lo[a] - hi[a] for a, e in enumerate(self.dims)]
        self.ng = self.nu[0] * self.nu[1] * self.nu[2]
        self.step = max(1, (1 << 22) // n ** 3)
        self.parts = [self.part(e0) for e0 in range(0, self.E, self.step)] if keep else None

    def part(self, e0):
        """(l2g [e,k,j,i], factors [e,k,7,j,i]) of the elements from e0."""
        n, N = self.n, self.N
        e = torch.arange(e0, min(e0 + self.step, self.E), device="cuda")
        pos = (e % self.dims[0], e // self.dims[0] % self.dims[1], e // (self.dims[0] * self.dims[1]))
        i = torch.arange(n, device="cuda")
        at, ok = [], []
        for a in range(3):
            g = N * pos[a][:, None] + i - self.lo[a]
            ok.append((g >= 0) & (g < self.nu[a]))
            at.append(g)
        l2g = at[0][:, None, None, :] + self.nu[0] * (at[1][:, None, :, None] + self.nu[1] * at[2][:, :, None, None])
        good = ok[0][:, None, None, :] & ok[1][:, None, :, None] & ok[2][:, :, None, None]
        l2g = torch.where(good, l2g, -1)
        C = torch.stack([torch.stack([torch.stack([self.V[pos[2] + c, pos[1] + b, pos[0] + a] for a in (0, 1)], 1)
                                      for b in (0, 1)], 1) for c in (0, 1)], 1)  # [e][c][b][a][3]
        ph = self.phi
        shape = (len(e), n, n, n, 3)
        jr = torch.einsum("ecbx,ck,bj->ekjx", (C[:, :, :, 1] - C[:, :, :, 0]) / 2, ph, ph)[:, :, :, None].expand(shape)
        js = torch.einsum("ecax,ck,ai->ekix", (C[:, :, 1] - C[:, :, 0]) / 2, ph, ph)[:, :, None].expand(shape)
        jt = torch.einsum("ebax,bj,ai->ejix", (C[:, 1] - C[:, 0]) / 2, ph, ph)[:, None].expand(shape)
        rows = [torch.linalg.cross(js, jt), torch.linalg.cross(jt, jr), torch.linalg.cross(jr, js)]
        det = (jr * rows[0]).sum(-1)
        w3 = self.w[:, None, None] * self.w[:, None] * self.w
        f = w3 / det
        geo = [f * (rows[a] * rows[b]).sum(-1) for a, b in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))]
        return l2g, torch.stack(geo + [w3 * det], 2)

    def apply(self, x, lam, screen):
        y = torch.zeros(self.ng + 1, dtype=torch.float64, device="cuda")  # the last: masked nodes
        xm = torch.cat([x.double(), x.new_zeros(1, dtype=torch.float64)])
        for p in range(-(-self.E // self.step)):
            l2g, g = self.parts[p] if self.parts is not None else self.part(p * self.step)
            u = xm[l2g]
            ur, us, ut = (torch.einsum(s, self.D, u) for s in ("im,ekjm->ekji", "jm,ekmi->ekji", "km,emji->ekji"))
            vr = g[:, :, 0] * ur + g[:, :, 1] * us + g[:, :, 2] * ut
            vs = g[:, :, 1] * ur + g[:, :, 3] * us + g[:, :, 4] * ut
            vt = g[:, :, 2] * ur + g[:, :, 4] * us + g[:, :, 5] * ut
            yl = torch.einsum("mi,ekjm->ekji", self.D, vr)
            yl += torch.einsum("mj,ekmi->ekji", self.D, vs)
            yl += torch.einsum("mk,emji->ekji", self.D, vt)
            if screen:
                yl += lam * g[:, :, 6] * u
            y.index_add_(0, torch.where(l2g < 0, self.ng, l2g).reshape(-1), yl.reshape(-1))
        return y[:-1] if screen else y[:-1] + lam * x

    def cg(self, b, lam, screen, its=0, tol=0.0, inv_d=None):
        x = torch.zeros_like(b)
        r = b.clone()
        z = r * inv_d if inv_d is not None else r
        p = z.clone()
        rz, bb = torch.dot(r, z), torch.dot(b, b)
        for _ in range(its or 400):
            Ap = self.apply(p, lam, screen)
            alpha = rz / torch.dot(p, Ap)
            x = x + alpha * p
            r = r - alpha * Ap
            z = r * inv_d if inv_d is not None else r
            new = torch.dot(r, z)
            p = z + (new / rz) * p
            rz = new
            if tol and torch.dot(r, r) <= tol * tol * bb:
                break
        return x

    def diag(self, lam, screen):
        """diag(A): per node the squares of D's columns against the diagonal factors, and D's own diagonal
        against the mixed ones."""
        D2, d = self.D * self.D, torch.diagonal(self.D)
        out = torch.zeros(self.ng + 1, dtype=torch.float64, device="cuda")
        for p in range(-(-self.E // self.step)):
            l2g, g = self.parts[p] if self.parts is not None else self.part(p * self.step)
            q = torch.einsum("mi,ekjm->ekji", D2, g[:, :, 0]) + torch.einsum("mj,ekmi->ekji", D2, g[:, :, 3])
            q += torch.einsum("mk,emji->ekji", D2, g[:, :, 5])
            di, dj, dk = d, d[:, None], d[:, None, None]
            q += 2.0 * (g[:, :, 1] * di * dj + g[:, :, 2] * di * dk + g[:, :, 4] * dj * dk)
            if screen:
                q += lam * g[:, :, 6]
            out.index_add_(0, torch.where(l2g < 0, self.ng, l2g).reshape(-1), q.reshape(-1))
        return out[:-1] if screen else out[:-1] + lam


def exact(case, seed):
    c = case
    if c["op"] == "serve":
        out = []
        for q in _requests(c, seed):
            P = _Plain(q["ek"], q["ek"], q["ek"], q["N"], c["perturb"], q["seed"], 0x3F)
            L = q["N"] * q["ek"] + 1
            k, j, i = np.meshgrid(*[np.arange(1, L - 1)] * 3, indexing="ij")
            b = torch.as_tensor(2.0 * _u01(q["seed"], 2, (i + L * (j + L * k)).reshape(-1)) - 1.0, device="cuda")
            out.append(P.cg(b, c["lam"], 0, tol=1e-14).cpu().numpy())
        return out
    P = _Plain(c["ex"], c["ey"], c["ez"], c["N"], c["perturb"], seed, c["faces"], keep=c["op"] == "cg")
    if c["op"] == "mesh":
        # the rows of Z^T list the copies of each DOF, ascending
        l2g, geo = [], []
        for p in range(-(-P.E // P.step)):
            a, g = P.part(p * P.step)
            l2g.append(a.reshape(-1).int())
            geo.append(g.reshape(-1))
        l2g, geo = torch.cat(l2g), torch.cat(geo)
        at = torch.nonzero(l2g >= 0).reshape(-1)
        rowptr = torch.zeros(P.ng + 1, dtype=torch.int64, device="cuda")
        rowptr[1:] = torch.bincount(l2g[at], minlength=P.ng).cumsum(0)
        out = {"l2g": l2g, "geo": geo, "rowptr": rowptr.int(), "cols": at[torch.sort(l2g[at], stable=True)[1]].int()}
        if c["prec"] == "f32":
            out["geo32"] = geo
        return out
    x = _vector(P.ng, seed, torch.float32 if c["prec"] == "f32" else torch.float64)
    if c["op"] == "apply":
        return P.apply(x.double(), c["lam"], c["screen"])
    inv_d = 1.0 / P.diag(c["lam"], c["screen"]) if c["precond"] else None
    if c["prec"] == "mixed":
        return P.cg(x, c["lam"], c["screen"], tol=1e-14, inv_d=1.0 / P.diag(c["lam"], c["screen"]))
    return P.cg(x, c["lam"], c["screen"], its=c["its"], inv_d=inv_d)
