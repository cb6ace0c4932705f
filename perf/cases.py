"""The work that a program using this library has it do, as measurable cases.

Every case goes through the library's public entry points (the binding of include/mf.h):
operator applies over the degrees, maps, precisions and mesh sizes of the library's own
configurations, CG iterations, mixed-precision solves, and a burst of served solve requests.

A case is a dict of plain values; ``prepare`` builds what a program holds before the call (the
operator with its workspace, the vectors, or a running server), ``run`` makes one pass, and
``exact`` computes the same outputs in 64-bit torch arithmetic without the library.
"""
import math

import numpy as np
import torch

import paper_2609_04534_gb300 as mf

AMP = 0.1  # curved meshes: x + AMP sin(pi x) sin(pi y) sin(pi z) on every coordinate
SHEAR = [1.0, 0.3, 0.0, 0.1, 1.2, -0.2, 0.0, 0.25, 0.9, 0.1, -0.2, 0.3]
PREC = {"fp64": mf.MF_FP64, "fp32": mf.MF_FP32, "mixed": mf.MF_MIXED}
KIND = {"laplace": mf.MF_LAPLACE, "helmholtz": mf.MF_HELMHOLTZ}


def _apply(name, nx, ny, nz, k, geom, prec, kind, bc, tune=False):
    return {"name": name, "what": "apply", "nx": nx, "ny": ny, "nz": nz, "degree": k, "geometry": geom,
            "precision": prec, "kind": kind, "dirichlet": bc, "autotune": tune}


def _cg(name, n, k, geom, its):
    return {"name": name, "what": "cg", "nx": n, "ny": n, "nz": n, "degree": k, "geometry": geom, "precision": "fp64",
            "kind": "laplace", "dirichlet": True, "iterations": its}


def listed():
    return [
        # The smallest configuration: an 8^3 mesh, where launches and latency are all there is.
        _apply("apply Q2 affine 8^3", 8, 8, 8, 2, "cart", "fp64", "laplace", True),
        # The same configuration's solver run: 50 CG iterations, as an application's inner solve.
        _cg("cg50 Q2 affine 8^3", 8, 2, "cart", 50),
        # Curved 64^3 mesh with per-point Jacobians: the residual evaluation of a production
        # mesh in FP64 (degree 3), and in FP32 (degree 4), as a mixed-precision solver runs it.
        _apply("apply Q3 curved 64^3", 64, 64, 64, 3, "curved", "fp64", "laplace", False),
        _apply("apply Q4 curved 64^3 fp32", 64, 64, 64, 4, "curved", "fp32", "laplace", False),
        # The benchmark's default workload: FP64 CG iterations of degree 4 on that mesh.
        _cg("cg20 Q4 curved 64^3", 64, 4, "curved", 20),
        # The degree sweep at about 50M cell-wise DoFs, Helmholtz on a Cartesian mesh, launch
        # configuration autotuned as the benchmark does: low, middle and high degree.
        _apply("apply Q2 cart 123^3", 123, 123, 123, 2, "cart", "fp64", "helmholtz", False, True),
        _apply("apply Q4 cart 74^3", 74, 74, 74, 4, "cart", "fp64", "helmholtz", False, True),
        _apply("apply Q7 cart 46^3", 46, 46, 46, 7, "cart", "fp64", "helmholtz", False, True),
        # A mid-size sheared (affine, full metric) mesh with ragged tiles and Dirichlet nodes, as
        # a program calls it that does not autotune.
        _apply("apply Q5 shear 27x22x19", 27, 22, 19, 5, "shear", "fp64", "helmholtz", True),
        # An ordinary FP32 call on an odd Cartesian mesh.
        _apply("apply Q6 cart 21x17x25 fp32", 21, 17, 25, 6, "cart", "fp32", "helmholtz", True),
        # Mixed-precision Poisson solve on a curved mesh (FP32 inner CG in FP64 refinement) of a
        # smooth right-hand side.
        {"name": "mixed solve Q4 curved 24^3", "what": "mixed", "nx": 24, "ny": 24, "nz": 24, "degree": 4,
         "geometry": "curved", "precision": "mixed", "kind": "laplace", "dirichlet": True, "rtol": 1e-12},
        # The serving stream's small requests (mesh 4^3..12^3, degrees 2..6, affine and curved
        # half and half): a burst submitted at once to a running server, all solutions returned.
        {"name": "serve 12 requests 4^3..12^3", "what": "serve", "requests": 12, "nmin": 4, "nmax": 12,
         "mesh_seed": 4, "rtol": 1e-12},
    ]


def _dims(rng, cells):
    """Three cell counts around the cube root of `cells`, odd and unequal ones among them."""
    f = [math.exp(rng.uniform(-0.35, 0.35)) for _ in range(2)]
    f.append(1.0 / (f[0] * f[1]))
    return [max(2, int(round(cells ** (1.0 / 3.0) * x))) for x in f]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    what = rng.choice(["apply", "apply", "apply", "cg", "mixed"])
    if what == "apply":
        k = rng.randint(1, 8)
        prec = rng.choice(["fp64", "fp64", "fp32"])
        nx, ny, nz = _dims(rng, _log(rng, 1.4e4, 4.5e7) / (k + 1) ** 3)
        return {"what": "apply", "nx": nx, "ny": ny, "nz": nz, "degree": k,
                "geometry": rng.choice(["cart", "curved", "shear", "cart", "curved"]), "precision": prec,
                "kind": rng.choice(["laplace", "helmholtz"]), "dirichlet": rng.random() < 0.5,
                "autotune": rng.random() < 0.3}
    k = rng.randint(2, 6)
    if what == "cg":
        nx, ny, nz = _dims(rng, _log(rng, 1.4e4, 1.5e7) / (k + 1) ** 3)
        return {"what": "cg", "nx": nx, "ny": ny, "nz": nz, "degree": k,
                "geometry": rng.choice(["cart", "curved", "shear"]), "precision": "fp64",
                "kind": rng.choice(["laplace", "helmholtz"]), "dirichlet": True, "iterations": rng.randint(10, 20)}
    nx, ny, nz = _dims(rng, _log(rng, 1.4e4, 6e5) / (k + 1) ** 3)
    return {"what": "mixed", "nx": nx, "ny": ny, "nz": nz, "degree": k, "geometry": rng.choice(["cart", "curved"]),
            "precision": "mixed", "kind": "laplace", "dirichlet": True, "rtol": 1e-12}


# ------------------------------------------------------------------ the program's side
class _State:
    """An operator (or server) and the device memory a program keeps with it."""

    def __init__(self):
        self.op = self.mesh = self.server = None

    def __del__(self):
        if self.server is not None:
            mf.mf_server_destroy(self.server)
        if self.op is not None:
            mf.mf_operator_destroy(self.op)
            mf.mf_mesh_destroy(self.mesh)


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def _unique_count(c):
    k = c["degree"]
    return (c["nx"] * k + 1) * (c["ny"] * k + 1) * (c["nz"] * k + 1)


def _random_unique(c, seed):
    """Values on the global nodes, uniform on [-1, 1), in the case's vector type."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand(_unique_count(c), dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    return u.float() if c["precision"] == "fp32" else u


def _rhs_weights(seed):
    """Weights of the manufactured right-hand sides of frequency 1, 2 and 3 in a smooth load."""
    return [float(w) for w in np.random.RandomState(seed % (1 << 32)).uniform(0.5, 1.5, 3)]


def _requests(c, seed):
    """The served requests: meshes and degrees from the case, right-hand sides from the seed."""
    r = np.random.RandomState(c["mesh_seed"])
    out = []
    for i in range(c["requests"]):
        n = int(round(math.exp(r.uniform(math.log(c["nmin"]), math.log(c["nmax"])))))
        out.append({"nx": n, "ny": n, "nz": n, "degree": int(r.randint(2, 7)),
                    "geometry": "curved" if r.randint(2) else "cart", "kind": "laplace", "dirichlet": True,
                    "seed": int(seed) * 1000 + i})
    return out


def prepare(case, seed):
    c, s = case, _State()
    s.case = c
    if c["what"] == "serve":
        s.arena = _bytes(2 << 30)
        s.server = mf.mf_server_create(s.arena.data_ptr(), s.arena.numel(), max_slots=16)
        s.x, s.req = [], []
        for q in _requests(c, seed):
            x = np.zeros(_unique_count(q))
            s.x.append(x)
            s.req.append(mf.make_request(
                q["nx"], q["ny"], q["nz"], q["degree"], geometry=mf.MF_CURVED_SIN if q["geometry"] == "curved" else
                mf.MF_AFFINE, curve_amp=AMP, rhs=mf.MF_RHS_RANDOM, seed=q["seed"], rtol=c["rtol"], mixed=1,
                x_out_ptr=x.ctypes.data))
        return s
    stream = torch.cuda.current_stream().cuda_stream
    s.mesh = mf.mf_mesh_create(c["nx"], c["ny"], c["nz"], mf.MF_CURVED_SIN if c["geometry"] == "curved" else
                               mf.MF_AFFINE, SHEAR if c["geometry"] == "shear" else None, AMP)
    s.op = mf.mf_operator_create(s.mesh, c["degree"], KIND[c["kind"]], 1.0, PREC[c["precision"]],
                                 mf.MF_BC_DIRICHLET0 if c["dirichlet"] else mf.MF_BC_NONE)
    info = mf.mf_operator_info(s.op)
    s.ws = _bytes(info["workspace_bytes"])
    mf.mf_operator_setup(s.op, s.ws.data_ptr(), s.ws.numel(), stream)
    dtype = torch.float32 if c["precision"] == "fp32" else torch.float64
    s.a = torch.empty(info["n_native"], dtype=dtype, device="cuda")  # the input (x or b)
    s.y = torch.zeros_like(s.a)                                      # the output
    if c["what"] == "mixed":
        scratch = _bytes(mf.mf_manufactured_workspace_bytes(s.op))
        part, s.a[:] = torch.empty_like(s.a), 0.0
        for f, w in enumerate(_rhs_weights(seed)):
            mf.mf_rhs_manufactured(s.op, float(f + 1), part.data_ptr(), scratch.data_ptr(), scratch.numel(), stream)
            s.a.add_(part, alpha=w)
        del part, scratch
    else:
        u = _random_unique(c, seed)
        mf.mf_scatter_unique(s.op, u.data_ptr(), s.a.data_ptr(), stream)
        del u
    if c["what"] != "apply":
        s.cws = _bytes(mf.mf_cg_workspace_bytes(s.op, int(c["what"] == "mixed")))
    elif c.get("autotune"):
        mf.mf_operator_autotune(s.op, s.a.data_ptr(), s.y.data_ptr(), 3, stream)
    return s


def run(state):
    s, c = state, state.case
    if c["what"] == "serve":
        tickets = [mf.mf_batch_submit(s.server, r) for r in s.req]
        mf.mf_server_drain(s.server, 60.0)
        for t in tickets:
            r = mf.mf_batch_poll(s.server, t)
            if r is None or r["status"] != mf.MF_OK:
                raise RuntimeError(f"request not solved: {r}")
        return s.x
    stream = torch.cuda.current_stream().cuda_stream
    if c["what"] == "apply":
        mf.mf_apply(s.op, s.a.data_ptr(), s.y.data_ptr(), stream)
    elif c["what"] == "cg":
        mf.mf_cg_solve(s.op, s.a.data_ptr(), s.y.data_ptr(), 0.0, c["iterations"], 0, s.cws.data_ptr(), s.cws.numel(),
                       stream, allow_not_converged=True)
    else:
        mf.mf_cg_solve(s.op, s.a.data_ptr(), s.y.data_ptr(), c["rtol"], 100000, 1, s.cws.data_ptr(), s.cws.numel(),
                       stream)
    return s.y


def _solve_iterations(c):
    """About what CG needs on such a mesh (the iteration count grows with cells x degree per axis)."""
    return max(10, 7 * max(c["nx"], c["ny"], c["nz"]) * c["degree"])


def work(case):
    """Bytes: the vectors once (per CG iteration x, r and p read and written once).  Operations:
    sum factorisation per cell-wise DoF (six folded sweeps on Cartesian cells, twelve and the
    metric on others)."""
    c = case
    if c["what"] == "serve":
        parts = [work(dict(q, what="mixed", precision="mixed")) for q in _requests(c, 0)]
        return {m: sum(p[m] for p in parts) for m in ("bytes", "flops")}
    n = c["degree"] + 1
    dofs = c["nx"] * c["ny"] * c["nz"] * n ** 3
    flops = dofs * (12 * n + 3 if c["geometry"] == "cart" else 24 * n + 15)
    if c["what"] == "apply":
        return {"bytes": dofs * (8 if c["precision"] == "fp32" else 16), "flops": flops}
    its = c["iterations"] if c["what"] == "cg" else _solve_iterations(c)
    return {"bytes": its * dofs * (48 if c["what"] == "cg" else 24), "flops": its * (flops + 12 * dofs)}


# ------------------------------------------------------------------ the same in 64 bits
def _gll(n):
    """Gauss-Lobatto-Legendre nodes on [0, 1]."""
    inner = np.polynomial.legendre.Legendre.basis(n - 1).deriv().roots().real if n > 2 else np.zeros(0)
    return (np.concatenate([[-1.0], np.sort(inner), [1.0]]) + 1) / 2


def _tables(n):
    """Values and derivatives of the nodal basis at the Gauss points of [0, 1], and the rule."""
    x = _gll(n)
    q, w = np.polynomial.legendre.leggauss(n)
    q, w = (q + 1) / 2, w / 2
    S, D = np.ones((n, n)), np.zeros((n, n))
    for i in range(n):
        for j in range(n):
            if j == i:
                continue
            S[:, i] *= (q - x[j]) / (x[i] - x[j])
            term = np.full(n, 1.0 / (x[i] - x[j]))
            for m in range(n):
                if m not in (i, j):
                    term *= (q - x[m]) / (x[i] - x[m])
            D[:, i] += term
    return S, D, q, w


class _Exact:
    """The operator by quadrature on global nodes, in FP64 torch."""

    def __init__(self, c):
        self.c, k = c, c["degree"]
        self.n = n = k + 1
        S, D, q, w = _tables(n)
        self.S, self.D = (torch.as_tensor(a, device="cuda") for a in (S, D))
        nx, ny, nz = c["nx"], c["ny"], c["nz"]
        self.shape = (nz, ny, nx, n, n, n)
        ax = [torch.arange(m, device="cuda")[:, None] * k + torch.arange(n, device="cuda") for m in (nx, ny, nz)]
        NX, NY, NZ = nx * k + 1, ny * k + 1, nz * k + 1
        self.nodes = NX * NY * NZ
        self.dofs = (ax[0][None, None, :, None, None, :] + NX * (ax[1][None, :, None, None, :, None] + NY *
                     ax[2][:, None, None, :, None, None])).reshape(-1).to(torch.int32)
        self.mask = None
        if c["dirichlet"]:
            m = torch.zeros((NZ, NY, NX), dtype=torch.bool, device="cuda")
            m[1:-1, 1:-1, 1:-1] = True
            self.mask = m.reshape(-1)
        # reference coordinates of the points per axis, as factors broadcast over the shape
        self.t = []
        for d, m in enumerate((nx, ny, nz)):
            v = (torch.arange(m, device="cuda", dtype=torch.float64)[:, None] + torch.as_tensor(q, device="cuda")) / m
            view = [1] * 6
            view[2 - d], view[5 - d] = m, n
            self.t.append(v.reshape(view))
        W = torch.as_tensor(w, device="cuda")
        self.w = W[:, None, None] * W[:, None] * W
        self.h = (1.0 / nx, 1.0 / ny, 1.0 / nz)
        self.mass = 1.0 if c["kind"] == "helmholtz" else 0.0

    def slab(self, z0, z1):
        """The metric of the cell layers z0..z1: G (6 entries), mass and det J, at every point."""
        h = self.h
        if self.c["geometry"] != "curved":
            A = np.array(SHEAR[:9]).reshape(3, 3) if self.c["geometry"] == "shear" else np.eye(3)
            J = A * np.array(h)
            Ji, det = np.linalg.inv(J), abs(np.linalg.det(J))
            G = Ji @ Ji.T
            return [self.w * float(det * G[i, j]) for i, j in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))], \
                self.w * (self.mass * det), self.w * det
        x, y, z = self.t[0], self.t[1], self.t[2][z0:z1]
        sx, sy, sz = (torch.sin(math.pi * v) for v in (x, y, z))
        v = [math.pi * torch.cos(math.pi * x) * sy * sz, math.pi * sx * torch.cos(math.pi * y) * sz,
             math.pi * sx * sy * torch.cos(math.pi * z)]
        # J = (I + AMP 1 v^T) diag(h): det and inverse of the rank-one update in closed form
        b = 1.0 + AMP * (v[0] + v[1] + v[2])
        a = AMP / b
        vv = a * a * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
        wd = self.w * (h[0] * h[1] * h[2]) * b.abs()
        G = [wd / (h[i] * h[j]) * ((1.0 if i == j else 0.0) - a * (v[i] + v[j]) + vv)
             for i, j in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))]
        return G, wd * self.mass, wd

    def _along(self, M, u, d):
        """M applied along local direction d (0 = x, the last axis)."""
        return torch.movedim(torch.matmul(torch.movedim(u, 5 - d, -1), M.T), -1, 5 - d)

    def cells(self, xu):
        """Local results A_K x_K of every cell, from global node values."""
        nz, ny, nx = self.shape[:3]
        step = max(1, int(4e6 // (ny * nx * self.n ** 3)))
        out = torch.empty(self.shape, dtype=torch.float64, device="cuda")
        per = ny * nx * self.n ** 3
        for z0 in range(0, nz, step):
            z1 = min(nz, z0 + step)
            u = xu[self.dofs[z0 * per:z1 * per].long()].reshape((z1 - z0,) + self.shape[1:])
            G, m, _ = self.slab(z0, z1)
            sx, dx = self._along(self.S, u, 0), self._along(self.D, u, 0)
            sxy, dxy = self._along(self.S, sx, 1), self._along(self.S, dx, 1)
            g = [self._along(self.S, dxy, 2), self._along(self.S, self._along(self.D, sx, 1), 2),
                 self._along(self.D, sxy, 2)]
            f = [G[0] * g[0] + G[1] * g[1] + G[2] * g[2], G[1] * g[0] + G[3] * g[1] + G[4] * g[2],
                 G[2] * g[0] + G[4] * g[1] + G[5] * g[2]]
            St, Dt = self.S.T, self.D.T
            zx, zy, zz = self._along(St, f[0], 2), self._along(St, f[1], 2), self._along(Dt, f[2], 2)
            if self.mass:
                zz = zz + self._along(St, m * self._along(self.S, sxy, 2), 2)
            yx = self._along(St, zx, 1)
            yy = self._along(Dt, zy, 1) + self._along(St, zz, 1)
            out[z0:z1] = self._along(Dt, yx, 0) + self._along(St, yy, 0)
        return out

    def assemble(self, yc):
        y = torch.zeros(self.nodes, dtype=torch.float64, device="cuda")
        flat, part = yc.reshape(-1), 1 << 24
        for i in range(0, flat.numel(), part):
            y.index_add_(0, self.dofs[i:i + part].long(), flat[i:i + part])
        return y if self.mask is None else y * self.mask

    def apply(self, xu):
        return self.assemble(self.cells(xu if self.mask is None else xu * self.mask))

    def cg(self, b, its, rtol=0.0):
        b = b if self.mask is None else b * self.mask
        x, r, p = torch.zeros_like(b), b.clone(), b.clone()
        rr = torch.dot(r, r)
        stop = rtol * rtol * float(rr)
        for i in range(its):
            q = self.apply(p)
            al = rr / torch.dot(p, q)
            x += al * p
            r -= al * q
            new = torch.dot(r, r)
            if rtol and i % 10 == 9 and float(new) <= stop:
                break
            p = r + (new / rr) * p
            rr = new
        return x

    def rhs(self, weights):
        """The load of the weighted sum of -Lap u for u = prod sin(f pi x_d), f = 1, 2, 3."""
        out = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        x, y, z = self.t
        s = 0.0
        if self.c["geometry"] == "curved":
            s = AMP * torch.sin(math.pi * x) * torch.sin(math.pi * y) * torch.sin(math.pi * z)
        _, _, wd = self.slab(0, self.shape[0])
        for f, wt in enumerate(weights):
            a = math.pi * (f + 1)
            out += wt * 3 * a * a * torch.sin(a * (x + s)) * torch.sin(a * (y + s)) * torch.sin(a * (z + s)) * wd
        for d in range(3):
            out = self._along(self.S.T, out, d)
        return self.assemble(out)

    def native(self, yu):
        """Global node values copied to the cells, in the library's tiled layout (4 x 4 x 2 cells)."""
        nz, ny, nx, n = self.shape[:4]
        tz, ty, tx = -(-nz // 2), -(-ny // 4), -(-nx // 4)
        full = torch.zeros((tz * 2, ty * 4, tx * 4, n ** 3), dtype=torch.float64, device="cuda")
        full[:nz, :ny, :nx] = yu[self.dofs.long()].reshape(nz, ny, nx, n ** 3)
        return full.reshape(tz, 2, ty, 4, tx, 4, n ** 3).permute(0, 2, 4, 6, 1, 3, 5).reshape(-1)


def _splitmix_uniform(seed, count):
    """The served random right-hand side: a splitmix64 counter stream, uniform on [-1, 1)."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, count + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return 2.0 * ((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1.0


def exact(case, seed):
    c = case
    if c["what"] == "serve":
        out = []
        for q in _requests(c, seed):
            e = _Exact(q)
            b = torch.as_tensor(_splitmix_uniform(q["seed"], e.nodes), device="cuda")
            out.append(e.cg(b, 20000, 1e-14).cpu().numpy())
        return out
    e = _Exact(c)
    if c["what"] == "mixed":
        return e.native(e.cg(e.rhs(_rhs_weights(seed)), 20000, 1e-14))
    u = _random_unique(c, seed).double()
    return e.native(e.apply(u) if c["what"] == "apply" else e.cg(u, c["iterations"]))
