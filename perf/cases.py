"""Workloads of the solver as its users run them, for timing and for checking.

A case is one call (or one short sequence of calls) through the public Python
binding, over the sizes and options of the configurations, tests and benchmark
of this repository: operator applies from a 150-vertex hull to a 20000-vertex
high-frequency body, one and several right-hand sides, one and several
objects; the OSRC preconditioner; GMRES solves; the tensor-core GEMM and the
batched dense solve; field evaluation on a grid.

``prepare`` makes what a program holds before the call: the mesh, the problem
handle and the input vectors, seeded.  ``run`` is one call.  What the
matrix-free FP32 and the mixed BF16 / FP32 paths compute (operator applies,
the iteratively evaluated preconditioner, solves to 1e-5 and 1e-6) carries
single precision or its solver's tolerance in FP64 containers; a program that
stores such vectors keeps them in complex64, and so does ``run``.  The FP64
field stays complex128, the GEMM's product float32.

``exact`` evaluates the same discrete operators in FP64 with plain torch: the
6-point triangle rule for triangle pairs that share no vertex, Sauter-Schwab
quadrature (4 Gauss points per dimension) for those that touch, dense or
direct solves instead of Krylov iterations.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2104_04609_gb300 import binding as B
from paper_2104_04609_gb300 import inputs

SPHERES_RHO = (0.95, 1.9)  # fat-like and bone-like objects of the four-sphere configuration


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _case(op, mesh, nv, k_ext, k_int, rho, nrhs, size):
    return dict(op=op, mesh=mesh, nv=nv, k_ext=k_ext, k_int=k_int, rho=rho, nrhs=nrhs, size=size)


def listed():
    c = []

    def add(name, *a):
        c.append(dict(name=name, **_case(*a)))

    # the smallest operator apply: the 150-vertex hull of the parity tests (launches and latency)
    add("apply_hull150", "apply", "hull", 150, 3.0, 4.5, 1.5, 1, 0)
    # one GMRES iteration's far + near field on the headline sphere (plain FP32 phases)
    add("apply_sphere10242", "apply", "ico", 10242, 20.0, 26.0, 1.5, 1, 0)
    # the high-frequency body (centred phases), the largest apply: k 60 / 144 on 20000 vertices
    add("apply_bumpy20000", "apply", "bumpy", 20000, 60.0, 144.0, 1.9, 1, 0)
    # multiple scatterers: four spheres of two materials, 642 vertices each, 0.5 MHz
    add("apply_spheres4x642", "apply", "spheres4", 2568, 10.5, 10.5, 1.0, 1, 0)
    # eight right-hand sides at once on the headline sphere (lockstep iterations)
    add("apply8_sphere10242", "apply", "ico", 10242, 20.0, 26.0, 1.5, 8, 0)
    # a serving request's ragged block: 5 right-hand sides, an odd ellipsoid
    add("apply5_ellipsoid3001", "apply", "ellipsoid", 3001, 15.0, 36.0, 1.9, 5, 0)
    # the OSRC preconditioner of one GMRES iteration on the headline sphere
    add("precond_sphere10242", "precond", "ico", 10242, 20.0, 26.0, 1.5, 1, 0)
    # a whole small solve, matrix-free, one plane wave
    add("solve_sphere642", "solve", "ico", 642, 2.0, 3.0, 1.5, 1, 0)
    # a whole lockstep solve of 8 plane waves
    add("solve8_sphere2562", "solve", "ico", 2562, 10.0, 13.0, 1.5, 8, 0)
    # the batched solve's tensor-core product: 8000 vertices, 128 right-hand sides
    add("gemm_16000x256x32000", "gemm", "", 0, 0.0, 0.0, 0.0, 256, 16000)
    # a dense-route serving request: 64 right-hand sides on a 3000-vertex ellipsoid
    add("batched64_ellipsoid3000", "batched", "ellipsoid", 3000, 8.0, 19.2, 1.9, 64, 0)
    # the paper's accuracy measure: total field on a 101 x 101 grid around the headline sphere
    add("field101_sphere10242", "field", "ico", 10242, 20.0, 26.0, 1.5, 1, 101)
    return c


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _draw(rng):
    op = rng.choice(["apply", "apply", "apply", "applym", "applym", "precond", "solve", "gemm", "batched", "field"])
    rho = round(rng.uniform(1.0, 2.0), 3)
    ratio = 1.0 / rng.uniform(0.4, 1.5)  # k_int / k_ext = 1 / (wave-speed ratio)
    mesh = rng.choice(["hull", "ellipsoid", "bumpy"])
    if op == "gemm":
        n2 = int(_log(rng, 500, 16000))
        return _case("gemm", "", 0, 0.0, 0.0, 0.0, 16 * rng.randint(1, 16), n2)
    if op == "precond":
        nv, k = int(_log(rng, 150, 16000)), _log(rng, 2.0, 20.0)
        return _case("precond", mesh, nv, k, k * ratio, rho, 1, 0)
    if op in ("solve", "batched"):
        nv = int(_log(rng, 150, 3000))
        k = rng.uniform(0.06, 0.14) * math.sqrt(nv)  # six or more elements per wavelength
        n = rng.choice([1, 2, 3, 5, 8]) if op == "solve" else rng.randint(2, 96)
        return _case(op, mesh if mesh != "bumpy" else "hull", nv, k, k * min(max(ratio, 0.7), 1.5), rho, n, 0)
    if op == "field":
        return _case("field", mesh, int(_log(rng, 150, 10000)), _log(rng, 2.0, 20.0), _log(rng, 2.0, 26.0), rho, 1,
                     int(_log(rng, 10, 101)))
    nv, k = int(_log(rng, 150, 12000)), _log(rng, 2.0, 60.0)
    if op == "apply" and rng.random() < 0.2:
        n = int(_log(rng, 40, 2500))
        return _case("apply", "spheres4", 4 * n, k, k, 1.0, 1, 0)
    return _case("apply", mesh, nv, k, k * ratio, rho, 1 if op == "apply" else rng.randint(2, 16), 0)


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        if _cost(c) <= most:
            return c


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def work(case):
    nv, r, op = case["nv"], case["nrhs"], case["op"]
    nt = 2 * nv - 4
    pairs = 36.0 * nt * max(0, nt - 13)
    # vectors in and out, touching-pair blocks (19 a vertex), rule points and normals
    vec = 2.0 * 32 * nv * r
    ap = dict(bytes=vec + 19.0 * 68 * nv + nt * (6 * 16 + 32), flops=pairs * (51 + 32.0 * r))
    sp = dict(bytes=2.0 * 32 * nv + 7.0 * 20 * nv, flops=10.0 * 7 * nv * 8 * 20)  # 10 systems, 20 products each
    if op == "apply":
        return ap
    if op == "precond":
        return sp
    if op == "solve":  # some 20 iterations
        return dict(bytes=20 * ap["bytes"], flops=20 * (ap["flops"] + r * sp["flops"]))
    if op == "gemm":
        m, k = _gemm_shape(case["size"])
        return dict(bytes=2.0 * m * k + 2.0 * r * k + 4.0 * m * r, flops=2.0 * m * r * k)
    if op == "batched":  # some 100 inner iterations of two products
        n2 = 2.0 * nv
        return dict(bytes=100 * 2 * 4 * n2 * n2, flops=100 * 2 * 8 * n2 * n2 * r)
    n = case["size"] ** 2
    return dict(bytes=n * 40.0 + 6.0 * nt * 96, flops=60.0 * n * 6 * nt)


def _gemm_shape(n2):
    return (n2 + 127) // 128 * 128, (2 * n2 + 63) // 64 * 64


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=8)
def _mesh(kind, nv):
    if kind == "ico":
        return inputs.icosphere({162: 2, 642: 3, 2562: 4, 10242: 5}[nv])
    if kind == "hull":
        return inputs.fibonacci_hull(nv)
    if kind == "ellipsoid":
        return inputs.ellipsoid(nv)
    if kind == "bumpy":
        return inputs.bumpy_ellipsoid(nv)
    n = nv // 4
    v, t = inputs.icosphere(3) if n == 642 else inputs.fibonacci_hull(n)
    at = [(-3.0, -1.5, 0.0), (-3.0, 1.5, 0.0), (3.0, -1.5, 0.0), (3.0, 1.5, 0.0)]
    return np.concatenate([v + np.array(a) for a in at]), np.concatenate([t + i * n for i in range(4)]).astype(np.int32)


def _objects(case):
    """Wavenumber and density ratio of each object (two fat-like, two bone-like spheres)."""
    if case["mesh"] != "spheres4":
        return None
    k = case["k_ext"]
    k_int = [k * 1500.0 / 1450.0] * 2 + [k * 1500.0 / 3600.0] * 2
    return k_int, [SPHERES_RHO[0]] * 2 + [SPHERES_RHO[1]] * 2


def _traces(case, seed, n):
    """n vectors [psi; phi] as an iteration meets them: plane-wave traces of random directions
    plus a tenth of noise, scaled to unit norm."""
    v, t = _mesh(case["mesh"], case["nv"])
    rng = np.random.default_rng(seed)
    d = rng.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    nrm = np.zeros_like(v)
    fn = np.cross(v[t[:, 1]] - v[t[:, 0]], v[t[:, 2]] - v[t[:, 0]])
    for a in range(3):
        np.add.at(nrm, t[:, a], fn)
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    k = case["k_ext"]
    phi = np.exp(1j * k * (d @ v.T))
    x = np.concatenate([1j * k * (d @ nrm.T) * phi, phi], axis=1)
    z = rng.standard_normal((2, *x.shape))
    s = np.abs(x).max(axis=1, keepdims=True)
    x = x + 0.1 * s * (z[0] + 1j * z[1])
    return x / np.linalg.norm(x, axis=1, keepdims=True)


def _dirs(seed, n):
    d = np.random.default_rng(seed).standard_normal((n, 3))
    return d / np.linalg.norm(d, axis=1, keepdims=True)


def _grid(size, seed):
    """A size x size grid over [-3, 3]^2 through the origin, tilted by the seed."""
    rng = np.random.default_rng(seed)
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    g = np.linspace(-3.0, 3.0, size)
    u, w = np.meshgrid(g, g, indexing="ij")
    return u.reshape(-1, 1) * q[0] + w.reshape(-1, 1) * q[1]


def _gemm_inputs(case, seed, device):
    m, k = _gemm_shape(case["size"])
    g = torch.Generator(device=device).manual_seed(seed)
    a = torch.randn((m, k), generator=g, device=device, dtype=torch.float32).to(torch.bfloat16)
    b = torch.randn((case["nrhs"], k), generator=g, device=device, dtype=torch.float32).to(torch.bfloat16)
    return a, b


def prepare(case, seed):
    op = case["op"]
    dev = torch.device("cuda", 0)
    if op == "gemm":
        a, b = _gemm_inputs(case, seed, dev)
        m, n, k = a.shape[0], b.shape[0], a.shape[1]
        ws = torch.empty(max(16, B.osrc_gemm_bf16_ws_bytes(m, n, k)), dtype=torch.uint8, device=dev)
        return dict(case=case, A=a, B=b, C=torch.empty((m, n), dtype=torch.float32, device=dev),
                    err=torch.zeros(1, dtype=torch.int32, device=dev), ws=ws)
    v, t = _mesh(case["mesh"], case["nv"])
    kw = {}
    if op == "batched":
        kw = dict(precision=B.OSRC_FP64_DENSE, dense_assembly=B.OSRC_ASSEMBLE_FF)
    S = B.Solver(v, t, case["k_ext"], case["k_int"], case["rho"], objects=_objects(case), **kw)
    st = dict(case=case, S=S)
    if op in ("apply", "precond"):
        st["x"] = torch.from_numpy(_traces(case, seed, case["nrhs"])).to(dev)
    elif op in ("solve", "batched"):
        st["b"] = S.rhs_planewave(_dirs(seed, case["nrhs"]))
        if op == "batched":  # the request's explicit preconditioner, kept with the assembled system
            B.osrc_dense_precond_build(S.pb)
            st["out"] = torch.empty_like(st["b"])
    else:
        st["x"] = torch.from_numpy(_traces(case, seed, 1)[0]).to(dev)
        st["pts"] = torch.from_numpy(_grid(case["size"], seed)).to(dev)
        st["dir"] = _dirs(seed, 1)[0]
    return st


def run(state):
    op = state["case"]["op"]
    if op == "gemm":
        B.osrc_gemm_bf16(state["A"], state["B"], state["C"], state["err"], ws=state["ws"])
        return state["C"]
    S = state["S"]
    if op == "apply":
        return S.apply(state["x"]).to(torch.complex64)
    if op == "precond":
        return S.precond(state["x"]).to(torch.complex64)
    if op == "solve":
        x, _ = S.solve(state["b"], tol=1e-5)
        return x.to(torch.complex64)
    if op == "batched":
        B.osrc_dense_batched_solve(S.pb, state["b"], state["out"], tol=1e-6, inner_maxit=400)
        return state["out"].to(torch.complex64)
    return S.field(state["x"], state["pts"], B.OSRC_INC_PLANEWAVE, state["dir"])


# ---------------------------------------------------------------------------
# the same discrete operators in FP64, plain torch
# ---------------------------------------------------------------------------
_QA = (0.445948490915965, 0.091576213509771)  # 6-point degree-4 rule (Dunavant 1985)
_QW = (0.223381589678011, 0.109951743655322)


def _rule(dev):
    lam = np.empty((6, 3))
    for q in range(6):
        lam[q] = _QA[q // 3]
        lam[q, q % 3] = 1.0 - 2.0 * _QA[q // 3]
    return torch.from_numpy(lam).to(dev), torch.tensor([_QW[q // 3] for q in range(6)], dtype=torch.float64, device=dev)


class _Exact:
    """FP64 geometry, kernels and touching-pair integrals of one case."""

    def __init__(self, case, dev):
        v, t = _mesh(case["mesh"], case["nv"])
        self.case, self.dev, self.nv, self.nt = case, dev, len(v), len(t)
        self.v, self.t = torch.from_numpy(v).to(dev), torch.from_numpy(t.astype(np.int64)).to(dev)
        P = self.v[self.t]
        self.P = P
        c = torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
        ln = c.norm(dim=1)
        self.area, self.n = 0.5 * ln, c / ln[:, None]
        # curl of the hat functions: opposite edges over twice the area
        self.curl = torch.stack([P[:, (a + 1) % 3] - P[:, (a + 2) % 3] for a in range(3)], 1) / ln[:, None, None]
        self.lam, self.w = _rule(dev)
        self.pts = torch.einsum("qa,tad->tqd", self.lam, P)
        # material of each triangle's object
        ob = _objects(case)
        nt = self.nt
        if ob is None:
            comp = np.zeros(nt, dtype=np.int64)
            ob = ([case["k_int"]], [case["rho"]])
        else:
            comp = np.arange(nt) // (nt // 4)
        self.ncomp = len(ob[0])
        self.comp = torch.from_numpy(comp).to(dev)
        self.k1 = torch.tensor(ob[0], dtype=torch.float64, device=dev)[self.comp]
        self.rho = torch.tensor(ob[1], dtype=torch.float64, device=dev)[self.comp]
        self.touch = self._touching(t)

    @staticmethod
    def _touching(t):
        """Ordered touching pairs (t, s), number of shared vertices and the local orders that put
        the shared vertices first (ascending in t)."""
        nt = len(t)
        order = np.argsort(t.reshape(-1), kind="stable")
        vs = t.reshape(-1)[order]
        tri = order // 3
        start = np.searchsorted(vs, np.arange(t.max() + 2))
        cnt = np.diff(start)
        deg = cnt[t].sum(1)
        a = np.repeat(np.arange(nt), deg)
        lists = [tri[start[i]:start[i + 1]] for i in range(t.max() + 1)]
        b = np.concatenate([np.concatenate([lists[i] for i in row]) for row in t])
        ab = np.unique(a * np.int64(nt) + b)
        a, b = ab // nt, ab % nt
        eq = t[a][:, :, None] == t[b][:, None, :]
        sh_t, sh_s = eq.any(2), eq.any(1)
        m = sh_t.sum(1)
        # stable sort puts shared local vertices first, in ascending local order of t
        pt = np.argsort(~sh_t, axis=1, kind="stable")
        match = np.where(sh_t, eq.argmax(2), 9)
        ps = np.take_along_axis(match, pt, 1)
        rest = np.argsort(sh_s, axis=1, kind="stable")  # unshared local vertices of s first, ascending
        for i in range(3):
            fill = ps[:, i] == 9
            ps[fill, i] = rest[fill, i - m[fill]]
        return a, b, m, pt, ps

    def kernels(self, r, k1, rho, same):
        """1/r-free combinations of the two wavenumbers at distances r; same: 1 on one object, else 0."""
        k0 = self.case["k_ext"]
        f = 1.0 / (4.0 * math.pi * r)
        g0 = torch.polar(f, k0 * r)
        g1 = torch.polar(f * same, k1 * r)
        h = (g0 * torch.complex(-torch.ones_like(r), k0 * r) + g1 * torch.complex(-torch.ones_like(r), k1 * r)) / r**2
        return g0, g1, h

    def chunks(self, most):
        step = max(1, most // (36 * self.nt))
        for t0 in range(0, self.nt, step):
            yield t0, min(self.nt, t0 + step)

    def far_blocks(self, t0, t1):
        """Kernel values between the rule points of test triangles t0..t1 and all source points:
        V (G0 + rho G1), K, T, k^2-weighted and curl-weighted G, zero on touching pairs."""
        X = self.pts[t0:t1].reshape(-1, 1, 3)
        Y = self.pts.reshape(1, -1, 3)
        d = X - Y
        keep = torch.ones((t1 - t0, self.nt), dtype=torch.float64, device=self.dev)
        a, b = self.touch[0], self.touch[1]
        i0, i1 = np.searchsorted(a, t0), np.searchsorted(a, t1)
        keep[torch.from_numpy(a[i0:i1] - t0).to(self.dev), torch.from_numpy(b[i0:i1]).to(self.dev)] = 0.0
        keep = keep.repeat_interleave(6, 0).repeat_interleave(6, 1)
        r = d.norm(dim=2)
        r = torch.where(keep > 0, r, torch.ones_like(r))
        k1 = self.k1[t0:t1].repeat_interleave(6)[:, None]
        rho = self.rho[t0:t1].repeat_interleave(6)[:, None]
        if self.ncomp > 1:
            same = (self.comp[t0:t1, None] == self.comp[None]).double().repeat_interleave(6, 0).repeat_interleave(6, 1)
        else:
            same = torch.ones((), dtype=torch.float64, device=self.dev)
        g0, g1, h = self.kernels(r, k1, rho, same)
        g0, g1, h = g0 * keep, g1 * keep, h * keep
        ny = self.n.repeat_interleave(6, 0)
        nx = self.n[t0:t1].repeat_interleave(6, 0)
        K = h * (d * ny[None]).sum(2)  # -(K0 + K1): minus H (y - x).n_y
        T = h * (d * nx[:, None]).sum(2)
        nn = nx @ ny.T
        return g0 + rho * g1, K, T, nn * (self.case["k_ext"] ** 2 * g0 + k1**2 / rho * g1), g0 + g1 / rho

    def near_blocks(self):
        """The four 3 x 3 blocks of every touching pair by Sauter-Schwab quadrature."""
        a, b, m, pt, ps = (torch.from_numpy(np.ascontiguousarray(z)).to(self.dev) for z in self.touch)
        x, w = np.polynomial.legendre.leggauss(4)
        x, w = torch.from_numpy(0.5 * (x + 1)).to(self.dev), torch.from_numpy(0.5 * w).to(self.dev)
        xi, e1, e2, e3 = (z.reshape(-1) for z in torch.meshgrid(x, x, x, x, indexing="ij"))
        ww = torch.einsum("i,j,k,l->ijkl", w, w, w, w).reshape(-1)
        out = torch.zeros((len(a), 4, 3, 3), dtype=torch.complex128, device=self.dev)
        for kase in (1, 2, 3):
            sel = torch.nonzero(m == kase).reshape(-1)
            for part in torch.split(sel, 20000):
                out[part] = self._near_part(part, a, b, pt, ps, _ss_points(kase, xi, e1, e2, e3), ww)
        return a, b, out

    def _near_part(self, part, a, b, pt, ps, rules, ww):
        ta, tb = a[part], b[part]
        pt, ps = pt[part], ps[part]
        Pt = torch.gather(self.P[ta], 1, pt[:, :, None].expand(-1, -1, 3))
        Ps = torch.gather(self.P[tb], 1, ps[:, :, None].expand(-1, -1, 3))
        nt_, ns_ = self.n[ta], self.n[tb]
        scale = 4.0 * self.area[ta] * self.area[tb]
        acc = torch.zeros((len(part), 4, 3, 3), dtype=torch.complex128, device=self.dev)
        dc = torch.zeros(len(part), dtype=torch.complex128, device=self.dev)
        k1, rho = self.k1[ta][:, None], self.rho[ta][:, None]
        one = torch.ones((), dtype=torch.float64, device=self.dev)
        for (x0, x1, y0, y1, jac) in rules:
            la = torch.stack([1.0 - x0, x0 - x1, x1], 1)
            lb = torch.stack([1.0 - y0, y0 - y1, y1], 1)
            d = torch.einsum("qa,pad->pqd", la, Pt) - torch.einsum("qa,pad->pqd", lb, Ps)
            w = (ww * jac)[None] * scale[:, None]
            g0, g1, h = self.kernels(d.norm(dim=2), k1, rho, one)
            vals = torch.stack([g0 + rho * g1, h * (d * ns_[:, None]).sum(2), h * (d * nt_[:, None]).sum(2),
                                self.case["k_ext"] ** 2 * g0 + k1**2 / rho * g1], 1) * w[:, None]
            ll = (la[:, :, None] * lb[:, None, :]).reshape(-1, 9).to(torch.complex128)
            acc += (vals @ ll).reshape(len(part), 4, 3, 3)
            dc += ((g0 + g1 / rho) * w).sum(1)
        ca = torch.gather(self.curl[ta], 1, pt[:, :, None].expand(-1, -1, 3))
        cb = torch.gather(self.curl[tb], 1, ps[:, :, None].expand(-1, -1, 3))
        nn = (nt_ * ns_).sum(1)
        acc[:, 3] = dc[:, None, None] * torch.einsum("pad,pbd->pab", ca, cb) - nn[:, None, None] * acc[:, 3]
        # back to the triangles' own vertex order
        out = torch.empty_like(acc)
        idx = (3 * pt[:, :, None] + ps[:, None, :]).reshape(len(part), 1, 9).expand(-1, 4, -1)
        out.reshape(len(part), 4, 9).scatter_(2, idx, acc.reshape(len(part), 4, 9))
        return out

    def apply(self, x):
        """B x for x (n, 2 nv) complex128."""
        n, nv = x.shape[0], self.nv
        psi, phi = x[:, :nv].T, x[:, nv:].T
        W = (self.w[None] * self.area[:, None]).reshape(-1, 1)
        lamc = self.lam.to(torch.complex128)
        dens = lambda u: torch.einsum("qa,tar->tqr", lamc, u[self.t]).reshape(-1, n) * W  # noqa: E731
        ps, ph = dens(psi), dens(phi)
        c = torch.einsum("tad,tar->tdr", self.curl.to(torch.complex128), phi[self.t])
        cw = (c[:, None] * W.reshape(-1, 6)[:, :, None, None]).reshape(-1, 3 * n)
        y1 = torch.zeros((nv, n), dtype=torch.complex128, device=self.dev)
        y2 = torch.zeros_like(y1)
        for t0, t1 in self.chunks(1 << 25):
            V, K, T, D, C = self.far_blocks(t0, t1)
            wt = (self.w[None] * self.area[t0:t1, None])[:, :, None]
            u1 = (V @ ps + K @ ph).reshape(-1, 6, n) * wt
            u2 = (T @ ps - D @ ph).reshape(-1, 6, n) * wt
            A = ((C @ cw).reshape(-1, 6, 3, n) * wt[:, :, None]).sum(1)
            b1 = torch.einsum("qa,tqr->tar", lamc, u1)
            b2 = torch.einsum("qa,tqr->tar", lamc, u2) + torch.einsum("tad,tdr->tar", self.curl[t0:t1].to(A.dtype), A)
            at = self.t[t0:t1].reshape(-1)
            y1.index_add_(0, at, b1.reshape(-1, n))
            y2.index_add_(0, at, b2.reshape(-1, n))
        a, b, blk = self.near_blocks()
        pb, fb = psi[self.t[b]], phi[self.t[b]]
        at = self.t[a].reshape(-1)
        y1.index_add_(0, at, (blk[:, 0] @ pb + blk[:, 1] @ fb).reshape(-1, n))
        y2.index_add_(0, at, (blk[:, 2] @ pb + blk[:, 3] @ fb).reshape(-1, n))
        return torch.cat([y1, y2]).T.contiguous()

    def matrix(self):
        """The dense 2 nv x 2 nv system."""
        nv, nt = self.nv, self.nt
        A = torch.zeros((2, 2, nv, nv), dtype=torch.complex128, device=self.dev)
        lam = (self.lam * self.w[:, None]).to(torch.complex128)
        flat = [A[0, 0].view(-1), A[0, 1].view(-1), A[1, 0].view(-1), A[1, 1].view(-1)]

        def add(o, ta, tb, blk):
            idx = self.t[ta][:, :, None] * nv + self.t[tb][:, None, :]
            flat[o].index_add_(0, idx.reshape(-1), blk.reshape(-1))

        al = torch.arange(nt, device=self.dev)
        for t0, t1 in self.chunks(1 << 25):
            c = t1 - t0
            aa = (self.area[t0:t1, None] * self.area[None]).to(torch.complex128)[:, :, None, None]
            V, K, T, D, C = self.far_blocks(t0, t1)
            con = lambda Z: torch.einsum("qa,tqspb->tsab", lam, torch.einsum("tqsp,pb->tqsb", Z.reshape(c, 6, nt, 6), lam)[:, :, :, None]) * aa  # noqa: E731
            w = self.w.to(torch.complex128)
            cc = torch.einsum("tad,sbd->tsab", self.curl[t0:t1], self.curl).to(torch.complex128)
            dcur = torch.einsum("tqsp,q,p->ts", C.reshape(c, 6, nt, 6), w, w)[:, :, None, None] * aa * cc
            ta, tb = al[t0:t1].repeat_interleave(nt), al.repeat(c)
            for o, Z in enumerate((con(V), con(K), con(T), dcur - con(D))):
                add(o, ta, tb, Z)
        a, b, blk = self.near_blocks()
        for o in range(4):
            add(o, a, b, blk[:, o])
        return A.permute(0, 2, 1, 3).reshape(2 * nv, 2 * nv)

    def planewave(self, dirs):
        k = self.case["k_ext"]
        out = []
        for d in torch.from_numpy(dirs).to(self.dev):
            ph = k * (self.pts @ d)
            u = torch.polar(torch.ones_like(ph), ph)
            dn = 1j * k * (self.n @ d)[:, None] * u
            wt = (self.w[None] * self.area[:, None])
            b = torch.zeros((2, self.nv), dtype=torch.complex128, device=self.dev)
            for i, z in enumerate((u, dn)):
                c = torch.einsum("qa,tq->ta", self.lam.to(z.dtype), z * wt)
                b[i].index_add_(0, self.t.reshape(-1), c.reshape(-1))
            out.append(b.reshape(-1))
        return torch.stack(out)

    def precond(self, x, n_pade=4, theta=math.pi / 3):
        """diag(L_DtN, L_NtD) of one object by dense direct solves (rotated-branch Pade of the
        square root)."""
        nv, dev = self.nv, self.dev
        M = torch.zeros((nv, nv), dtype=torch.complex128, device=dev)
        S = torch.zeros_like(M)
        idx = (self.t[:, :, None] * nv + self.t[:, None, :]).reshape(-1)
        me = (torch.eye(3, device=dev, dtype=torch.float64) + 1.0) / 12.0
        se = torch.einsum("tad,tbd->tab", self.curl, self.curl) * self.area[:, None, None]
        M.view(-1).index_add_(0, idx, (self.area[:, None, None] * me).reshape(-1).to(M.dtype))
        S.view(-1).index_add_(0, idx, se.reshape(-1).to(M.dtype))
        e = torch.cat([(self.P[:, a] - self.P[:, (a + 1) % 3]).norm(dim=1) for a in range(3)])
        R, k = float(e.mean()), self.case["k_int"]
        ke2 = (k * (1.0 + 0.4j * (k * R) ** (-2.0 / 3.0))) ** 2
        z0 = np.exp(-1j * theta) - 1.0
        j = np.arange(1, n_pade + 1)
        aj = 2.0 / (2 * n_pade + 1) * np.sin(j * math.pi / (2 * n_pade + 1)) ** 2
        bj = np.cos(j * math.pi / (2 * n_pade + 1)) ** 2
        C0 = np.exp(0.5j * theta) * (1.0 + np.sum(aj * z0 / (1.0 + bj * z0)))
        Aj = np.exp(-0.5j * theta) * aj / (1.0 + bj * z0) ** 2
        Bj = np.exp(-1j * theta) * bj / (1.0 + bj * z0)
        gj = Aj / (1.0 - Bj)
        g0 = C0 - gj.sum()
        u, f = x[0, :nv], x[0, nv:]
        su, mf = S @ u, M @ f
        z1 = C0 * u
        z2 = g0 * torch.linalg.solve(M - S / ke2, mf)
        for A_, B_, g_ in zip(Aj, Bj, gj):
            K = M - complex(B_ / ke2) * S
            z = torch.linalg.solve(K, torch.stack([su, mf], 1))
            z1 = z1 - complex(A_ / ke2) * z[:, 0]
            z2 = z2 + complex(g_) * z[:, 1]
        return torch.cat([1j * k * z1, z2 / (1j * k)])[None]

    def field(self, x, pts, direction):
        nv, k0 = self.nv, self.case["k_ext"]
        lamc = self.lam.to(torch.complex128)
        W = (self.w[None] * self.area[:, None]).reshape(-1)
        ps = torch.einsum("qa,ta->tq", lamc, x[:nv][self.t]).reshape(-1) * W
        ph = torch.einsum("qa,ta->tq", lamc, x[nv:][self.t]).reshape(-1) * W
        Y, n = self.pts.reshape(-1, 3), self.n.repeat_interleave(6, 0)
        d = torch.from_numpy(direction).to(self.dev)
        us, regs = [], []
        for X in torch.split(pts, max(1, (1 << 25) // len(Y))):
            e = Y[None] - X[:, None]
            r = e.norm(dim=2)
            dn = (e * n[None]).sum(2)
            inside = ((W * dn / r**3).sum(1) / (4.0 * math.pi)) > 0.5
            k = torch.where(inside, torch.full_like(r[:, 0], self.case["k_int"]), torch.full_like(r[:, 0], k0))[:, None]
            g = torch.polar(1.0 / (4.0 * math.pi * r), k * r)
            sl = g @ ps
            dl = (g * torch.complex(-torch.ones_like(r), k * r) * dn / r**2) @ ph
            p = k0 * (X @ d)
            u = torch.where(inside, self.case["rho"] * sl - dl, torch.polar(torch.ones_like(p), p) + dl - sl)
            us.append(u)
            regs.append(inside.int())
        return torch.cat(us), torch.cat(regs)


def _ss_points(kase, xi, e1, e2, e3):
    """Points and Jacobians of the Sauter-Schwab maps (Sauter & Schwab, Boundary Element Methods,
    Sec. 5.2) for a common vertex (1), a common edge (2) and identical triangles (3); reference
    triangle 0 <= x2 <= x1 <= 1."""
    if kase == 1:
        j = xi**3 * e2
        a, b = (xi, xi * e1), (xi * e2, xi * e2 * e3)
        return [(*a, *b, j), (*b, *a, j)]
    if kase == 2:
        j = xi**3 * e1**2
        return [
            (xi, xi * e1 * e3, xi * (1 - e1 * e2), xi * e1 * (1 - e2), j),
            (xi, xi * e1, xi * (1 - e1 * e2 * e3), xi * e1 * e2 * (1 - e3), j * e2),
            (xi * (1 - e1 * e2), xi * e1 * (1 - e2), xi, xi * e1 * e2 * e3, j * e2),
            (xi * (1 - e1 * e2 * e3), xi * e1 * e2 * (1 - e3), xi, xi * e1, j * e2),
            (xi * (1 - e1 * e2 * e3), xi * e1 * (1 - e2 * e3), xi, xi * e1 * e2, j * e2),
        ]
    j = xi**3 * e1**2 * e2
    pairs = [
        ((xi, xi * (1 - e1 + e1 * e2)), (xi * (1 - e1 * e2 * e3), xi * (1 - e1))),
        ((xi, xi * e1 * (1 - e2 + e2 * e3)), (xi * (1 - e1 * e2), xi * e1 * (1 - e2))),
        ((xi * (1 - e1 * e2 * e3), xi * e1 * (1 - e2 * e3)), (xi, xi * e1 * (1 - e2))),
    ]
    return [(*p, *q, j) for a, b in pairs for p, q in ((a, b), (b, a))]


def exact(case, seed):
    dev = torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")
    op, nv = case["op"], case["nv"]
    if op == "gemm":
        a, b = _gemm_inputs(case, seed, dev)
        return a.double() @ b.double().T
    if op == "apply" and (nv > 11000 or nv * nv * (40 + 32 * case["nrhs"]) > 5e10):
        return None  # longer than some 20 s
    if op == "precond" and nv > 11000:
        return None
    E = _Exact(case, dev)
    if op == "apply":
        return E.apply(torch.from_numpy(_traces(case, seed, case["nrhs"])).to(dev))
    if op == "precond":
        return E.precond(torch.from_numpy(_traces(case, seed, 1)).to(dev))
    if op in ("solve", "batched"):
        return torch.linalg.solve(E.matrix(), E.planewave(_dirs(seed, case["nrhs"])).T).T.contiguous()
    x = torch.from_numpy(_traces(case, seed, 1)[0]).to(dev)
    return E.field(x, torch.from_numpy(_grid(case["size"], seed)).to(dev), _dirs(seed, 1)[0])
