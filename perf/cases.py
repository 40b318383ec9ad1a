"""The work that a user of this library has it do, as cases to time.

Three kinds of call, all through ``paper_1812_10722_gb300.lspr.Context``:

* ``product``   y = A(s) x of one geometry for B wavelengths (``matvec``), the unit every solver
  step consists of: the direct modes on small meshes, the treecode on larger ones, one wavelength
  and batches, FP64, FP32 and float-float arithmetic, one surface or a sensor with analytes;
* ``geometry``  a new mesh: ``mesh_upload`` and ``tree_build``, then the first product on it;
* ``solve``     the cross-section spectrum of B wavelengths (``solve``, FP32 treecode with
  iterative refinement).

Products in an FP32 mode and solves to a relative residual of 1e-6 carry single-precision digits
and are kept as complex64 / float32, as a program that stores them would; the FP64 and
float-float modes return complex128.
"""
from __future__ import annotations

import math

import numpy as np
import torch

R_NM = 10.0            # sphere radius of every workload
EPS_WATER = 1.7689
THRESHOLD = 0.5        # near-singular iff L_j / |c_i - c_j| >= THRESHOLD (mesh_upload's default)
E0 = (0.0, 0.0, 1.0)

# ``f``: the icosahedron's edges are cut into f parts (20 f^2 panels); ``fa``: the same for each of
# the analytes on +-z at a 1-nm gap (0: a bare sphere).  theta / P / ncrit: the treecode.
_BASE = dict(kind="product", mode="tree_fp32", f=32, fa=0, B=1, theta=0.4, P=5, ncrit=256)


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest configuration's product: 1280 panels, plain FP64, one wavelength
        _case("direct_fp64_1280", mode="direct_fp64", f=8),
        # a mid grid of the convergence sequence in FP32, all pairs
        _case("direct_fp32_5120", mode="direct_fp32", f=16),
        # the plain baseline: FP64 treecode, one wavelength
        _case("tree_fp64_20480", mode="tree_fp64"),
        # one wavelength of the 20480-panel sphere at its tuned tree
        _case("tree_fp32_20480"),
        # an odd size (56180 panels) at the configuration's literal tree
        _case("tree_fp32_56180", f=53, theta=0.5, P=6, ncrit=300),
        # 16-wavelength batch
        _case("tree_fp32_20480_b16", B=16),
        # the 64-wavelength sweep's product at its tuned tree
        _case("tree_fp32_81920_b64", f=64, B=64, P=7, ncrit=512),
        # the refinement residual of some running wavelengths (float-float), odd sizes
        _case("tree_ff_40500_b12", mode="tree_ff", f=45, B=12, P=7, ncrit=512),
        # sensor and two analytes, 32 wavelengths
        _case("sensor_145920_b32", f=64, fa=40, B=32, P=7, ncrit=512),
        # a new geometry of the size of the sweep's
        _case("geometry_81920", kind="geometry", f=64, P=7, ncrit=512),
        # 16-wavelength spectrum of the 20480-panel sphere
        _case("solve_20480_b16", kind="solve", B=16),
        # the benchmark's sweep: 64 wavelengths, 81920 panels
        _case("solve_81920_b64", kind="solve", f=64, B=64, P=7, ncrit=512),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["product"] * 7 + ["geometry", "solve", "solve"])
    tree = dict(theta=rng.choice([0.35, 0.4, 0.45, 0.5]), P=rng.choice([4, 5, 6, 7, 8]),
                ncrit=_log_int(rng, 128, 512))
    if kind == "geometry":
        return _case(kind=kind, f=_log_int(rng, 12, 64), **tree)
    if kind == "solve":
        tree["P"] = max(5, tree["P"])
        return _case(kind=kind, f=_log_int(rng, 12, 40), B=_log_int(rng, 1, 40), **tree)
    mode = rng.choice(["direct_fp64", "direct_fp32", "tree_fp64", "tree_fp32", "tree_fp32", "tree_fp32", "tree_fp32",
                       "tree_ff"])
    if mode.startswith("direct"):
        return _case(mode=mode, f=_log_int(rng, 8, 24), B=_log_int(rng, 1, 12), **tree)
    if mode == "tree_fp64":
        return _case(mode=mode, f=_log_int(rng, 16, 40), B=_log_int(rng, 1, 6), **tree)
    if mode == "tree_ff":
        return _case(mode=mode, f=_log_int(rng, 16, 50), B=_log_int(rng, 1, 16), **tree)
    fa = _log_int(rng, 8, 28) if rng.random() < 0.25 else 0
    return _case(mode=mode, f=_log_int(rng, 12, 64), fa=fa, B=_log_int(rng, 1, 64 if not fa else 32), **tree)


# ------------------------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _geodesic(f):
    """Unit sphere of 20 f^2 triangles, counter-clockwise seen from outside: (verts, tris)."""
    g = (1.0 + 5.0 ** 0.5) / 2.0
    ico = np.array([p for a in (-1.0, 1.0) for b in (-g, g) for p in ((0.0, a, b), (a, b, 0.0), (b, 0.0, a))])
    d = np.linalg.norm(ico[:, None] - ico[None], axis=2)
    adj = np.abs(d - 2.0) < 1e-9
    faces = [(i, j, k) for i in range(12) for j in range(i + 1, 12) for k in range(j + 1, 12)
             if adj[i, j] and adj[j, k] and adj[i, k]]
    faces = [(i, j, k) if np.dot(np.cross(ico[j] - ico[i], ico[k] - ico[i]), ico[i]) > 0 else (i, k, j)
             for i, j, k in faces]
    # barycentric lattice of one face: rows i = 0..f, i + 1 points each
    rows = np.repeat(np.arange(f + 1), np.arange(1, f + 2))
    start = np.arange(f + 1) * (np.arange(f + 1) + 1) // 2
    cols = np.arange(len(rows)) - start[rows]
    w = np.stack([f - rows, rows - cols, cols], 1) / f
    r, c = rows[rows < f], cols[rows < f]
    up = np.stack([start[r] + c, start[r + 1] + c, start[r + 1] + c + 1], 1)
    r, c = rows[cols < rows], cols[cols < rows]
    r, c = r[r < f], c[r < f]
    down = np.stack([start[r] + c, start[r + 1] + c + 1, start[r] + c + 1], 1)
    one = np.concatenate([up, down])
    verts = np.concatenate([w @ ico[list(q)] for q in faces])
    verts /= np.linalg.norm(verts, axis=1, keepdims=True)
    tris = np.concatenate([one + len(w) * q for q in range(20)])
    return verts, tris


def _rotation(rng):
    q, r = np.linalg.qr(rng.normal(size=(3, 3)))
    q = q * np.sign(np.diag(r))
    if np.linalg.det(q) < 0:
        q[:, 0] = -q[:, 0]
    return q


def _bumpy_ellipsoid(fa, rng):
    """Closed star-shaped analyte: semi-axes 4 x 4 x 7 nm (long axis z), smooth bumps up to 10 %."""
    v, t = _geodesic(fa)
    k, ph, c = rng.normal(size=(24, 3)) * 3.0, rng.uniform(0, 2 * np.pi, 24), rng.normal(size=24)
    bump = np.cos(v @ k.T + ph) @ c
    bump /= np.abs(bump).max()
    return v * np.array([4.0, 4.0, 7.0]) * (1.0 + 0.1 * bump)[:, None], t


def _mesh(case, seed):
    """(verts, tris, surf) as numpy; the seed turns the sphere and shapes the analytes."""
    rng = np.random.Generator(np.random.PCG64(seed))
    v, t = _geodesic(case["f"])
    vs, ts, ss = [R_NM * (v @ _rotation(rng).T)], [t], [np.zeros(len(t), np.int32)]
    if case["fa"]:
        for side in (1.0, -1.0):
            a, ta = _bumpy_ellipsoid(case["fa"], rng)
            # moved along the axis until its closest vertex is 1 nm from the sphere
            reach = (R_NM + 1.0) ** 2 - a[:, 0] ** 2 - a[:, 1] ** 2
            shift = np.max(np.sqrt(np.maximum(reach, 0.0)) - a[:, 2])
            a = a + np.array([0.0, 0.0, shift])
            if side < 0:
                a = a * np.array([-1.0, 1.0, -1.0])
            ts.append(ta + sum(len(q) for q in vs))
            vs.append(a)
            ss.append(np.full(len(ta), len(ss), np.int32))
    return np.concatenate(vs), np.concatenate(ts).astype(np.int32), np.concatenate(ss)


def _panels(case):
    return 20 * case["f"] ** 2 + 40 * case["fa"] ** 2


def _surfaces(case):
    return 3 if case["fa"] else 1


def _eps(case, seed):
    """Wavelengths of the case over 350-420 nm and the Drude / analyte permittivities [B, S]."""
    rng = np.random.Generator(np.random.PCG64(seed + 77))
    B, S = case["B"], _surfaces(case)
    lam = np.linspace(350.0, 420.0, B) if B > 1 else np.array([380.0])
    lam = lam + rng.uniform(-0.5, 0.5)
    w = 1239.84198 / lam
    eps = 3.7 - 81.0 / (w * w + 0.018j * w)
    if S > 1:
        eps = np.stack([eps] + [np.full(B, 2.25 + 0j)] * (S - 1), 1)
    return lam, eps


def _vectors(case, seed, n):
    gen = torch.Generator(device=_device()).manual_seed(seed)
    x = torch.rand((case["B"], 2 * n, 2), generator=gen, device=_device(), dtype=torch.float64)
    x = torch.view_as_complex(2.0 * x - 1.0)
    return x[0] if case["B"] == 1 else x


class _State:
    pass


def prepare(case, seed):
    from paper_1812_10722_gb300 import lspr
    st = _State()
    st.case = dict(case)
    v, t, s = _mesh(case, seed)
    st.verts = torch.from_numpy(v).to(_device())
    st.tris = torch.from_numpy(t).to(_device())
    st.surf = torch.from_numpy(s).to(_device()) if _surfaces(case) > 1 else None
    st.lam, st.eps = _eps(case, seed)
    st.ratio = st.eps / EPS_WATER
    if case["kind"] != "solve":
        st.x = _vectors(case, seed, len(t))
    st.ctx = lspr.Context(torch.cuda.current_device())
    if case["B"] >= 24:
        st.ctx.set_tensor_cores(3)   # what the solver tuner sets for batches of this size
    if case["kind"] != "geometry":
        st.ctx.mesh_upload(st.verts, st.tris, surf_id=st.surf)
        if case["mode"].startswith("tree"):
            st.ctx.tree_build(case["theta"], case["P"], case["ncrit"])
    return st


def run(st):
    c = st.case
    if c["kind"] == "solve":
        r = st.ctx.solve(st.eps, EPS_WATER, st.lam, E0=E0, tol=1e-6, restart=50, maxiter=2000, mode=c["mode"],
                         refine=True)
        return {"dipole": r.dipole.astype(np.complex64), "sigma_ext": r.sigma_ext.astype(np.float32)}
    if c["kind"] == "geometry":
        st.ctx.mesh_upload(st.verts, st.tris, surf_id=st.surf)
        st.ctx.tree_build(c["theta"], c["P"], c["ncrit"])
    y = st.ctx.matvec(st.x, st.ratio, c["mode"])
    if c["mode"].endswith("fp32"):
        y = y.to(torch.complex64)
    if c["kind"] == "geometry":
        return {"y": y, "sizes": st.ctx.info()}
    return {"y": y}


def work(case):
    """Bytes: vectors (complex128) in and out, for a geometry the mesh and the panels made of it.
    Operations: the direct sums over 4 nodes per panel (18 to form both kernels, 8 per wavelength
    and surface), or the treecode's direct sums and expansions: about 5 Ncrit / theta^2 direct
    sources and 3 log4(4 N / Ncrit) / theta^2 boxes per target on a closed surface."""
    n, B, S = _panels(case), case["B"], _surfaces(case)
    sets = B * S
    vec = 2 * n * 16 * B
    if case["mode"].startswith("direct"):
        flops = 4.0 * n * n * (18 + 8 * sets)
    else:
        nt = (case["P"] + 1) * (case["P"] + 2) * (case["P"] + 3) // 6
        q = 1.0 / case["theta"] ** 2
        near = min(4.0 * n, 5.0 * case["ncrit"] * q)
        boxes = 3.0 * q * max(1.0, math.log(4.0 * n / case["ncrit"], 4))
        flops = n * (near * (18 + 8 * sets) + boxes * nt * (8 + 8 * sets)) + 4.0 * n * nt * (6 + 8 * sets)
    nbytes = 2.0 * vec + 48.0 * n
    if case["kind"] == "geometry":
        nbytes += 4 * 64.0 * n + 25 * 20.0 * n
        flops += 25.0 * n * 23 * 20
    if case["kind"] == "solve":
        steps = 60      # products of a wavelength to 1e-6 (the sphere near its resonance)
        nbytes = 48.0 * n + steps * 2.0 * vec
        flops *= steps
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------- 64-bit reference
# Dunavant's symmetric rules: (a, b, weight), b = None: permutations of (a, (1-a)/2, (1-a)/2)
_RULE4 = [(1 / 3, None, -0.5625), (0.6, None, 0.520833333333333)]
_RULE19 = [(1 / 3, None, 0.097135796282799), (0.020634961602525, None, 0.031334700227139),
           (0.125820817014127, None, 0.077827541004774), (0.623592928761935, None, 0.079647738927210),
           (0.910540973211095, None, 0.025577675658698), (0.036838412054736, 0.221962989160766, 0.043283539377289)]


def _nodes(rule):
    out = []
    for a, b, w in rule:
        if b is None:
            h = 0.5 * (1.0 - a)
            pts = [(a, h, h)] if abs(a - h) < 1e-9 else [(a, h, h), (h, a, h), (h, h, a)]
        else:
            c = 1.0 - a - b
            pts = [(a, b, c), (a, c, b), (b, a, c), (b, c, a), (c, a, b), (c, b, a)]
        out += [(p, w) for p in pts]
    return out


class _Dense:
    """Rows of the discretised layer potentials in 64 bits (single layer V, double layer K): the
    4-point rule on far panels, the 19-point rule on near-singular ones, and on a panel itself 9
    Gauss-Legendre nodes per edge in the angle (its double layer vanishes)."""

    def __init__(self, verts, tris):
        dev = _device()
        self.v = torch.from_numpy(verts).to(dev)[torch.from_numpy(tris).to(dev).long()]   # [N, 3, 3]
        e1, e2 = self.v[:, 1] - self.v[:, 0], self.v[:, 2] - self.v[:, 0]
        c = torch.linalg.cross(e1, e2)
        nc = torch.sqrt(c[:, 0] * c[:, 0] + c[:, 1] * c[:, 1] + c[:, 2] * c[:, 2])
        self.n, self.area = c / nc[:, None], 0.5 * nc
        self.L = torch.sqrt(2.0 * self.area)
        self.c = (self.v[:, 0] + self.v[:, 1] + self.v[:, 2]) / 3.0
        self.N = len(tris)
        self.far = [(torch.einsum("k,nkd->nd", torch.tensor(p, device=dev, dtype=torch.float64), self.v), w)
                    for p, w in _nodes(_RULE4)]
        self.self_v = self._self_v()

    def _self_v(self):
        x, w = np.polynomial.legendre.leggauss(9)
        s = torch.zeros_like(self.area)
        for e in range(3):
            a, b = self.v[:, e] - self.c, self.v[:, (e + 1) % 3] - self.c
            t = (b - a) / (b - a).norm(dim=1, keepdim=True)
            sa, sb = (a * t).sum(1), (b * t).sum(1)
            h = (a - sa[:, None] * t).norm(dim=1)
            pa, pb = torch.atan2(sa, h), torch.atan2(sb, h)
            mid, half = 0.5 * (pa + pb), 0.5 * (pb - pa)
            s += h * half * sum(float(wk) / torch.cos(mid + float(xk) * half) for xk, wk in zip(x, w))
        return s / (4.0 * math.pi)

    def rows(self, i0, i1):
        ci = self.c[i0:i1]
        V = torch.zeros((i1 - i0, self.N), device=ci.device, dtype=torch.float64)
        K = torch.zeros_like(V)
        for y, w in self.far:
            d = [ci[:, None, q] - y[None, :, q] for q in range(3)]
            r = torch.rsqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
            dn = d[0] * self.n[None, :, 0] + d[1] * self.n[None, :, 1] + d[2] * self.n[None, :, 2]
            V += w * r
            K += w * dn * r * r * r
        d = [ci[:, None, q] - self.c[None, :, q] for q in range(3)]
        dist = torch.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
        own = torch.arange(i0, i1, device=ci.device)
        near = self.L[None, :] / dist >= THRESHOLD
        near[own - i0, own] = False
        i, j = near.nonzero(as_tuple=True)
        fv, fk = torch.zeros(len(i), device=ci.device, dtype=torch.float64), 0.0
        for p, w in _nodes(_RULE19):
            y = torch.einsum("k,nkd->nd", torch.tensor(p, device=ci.device, dtype=torch.float64), self.v[j])
            d = ci[i] - y
            r = 1.0 / d.norm(dim=1)
            fv = fv + w * r
            fk = fk + w * (d * self.n[j]).sum(1) * r ** 3
        V[i, j], K[i, j] = fv, fk
        V *= self.area / (4.0 * math.pi)
        K *= self.area / (4.0 * math.pi)
        V[own - i0, own] = self.self_v[own]
        K[own - i0, own] = 0.0
        return V, K

    def blocks(self):
        step = max(16, int(1.5e8) // self.N)
        return [(i, min(self.N, i + step)) for i in range(0, self.N, step)]


def _product(dense, surf, x, ratio):
    """A(s) x for x [B, 2N] complex128 and s [B, S]."""
    N, B, S = dense.N, x.shape[0], ratio.shape[1]
    phi, dphi = (torch.view_as_real(x[:, k * N:(k + 1) * N]).permute(1, 0, 2).reshape(N, 2 * B) for k in (0, 1))
    y = torch.empty_like(x)
    cut = [0] + [int((surf <= s).sum()) for s in range(S)]
    cplx = lambda a: torch.view_as_complex(a.reshape(-1, B, 2).contiguous()).T   # noqa: E731
    own = torch.from_numpy(surf).to(x.device)
    for i0, i1 in dense.blocks():
        V, K = dense.rows(i0, i1)
        Vd = [cplx(V[:, cut[s]:cut[s + 1]] @ dphi[cut[s]:cut[s + 1]]) for s in range(S)]
        Kp = [cplx(K[:, cut[s]:cut[s + 1]] @ phi[cut[s]:cut[s + 1]]) for s in range(S)]
        half = 0.5 * x[:, i0:i1]
        top, bot = half.clone(), half.clone()
        for s in range(S):
            mine = (own[i0:i1] == s)[None, :]
            top += torch.where(mine, Kp[s] - Vd[s], torch.zeros_like(half))
            bot += ratio[:, s:s + 1] * Vd[s] - Kp[s]
        y[:, i0:i1], y[:, N + i0:N + i1] = top, bot
    return y


def _solve(dense, lam, eps):
    """Dipoles and cross-sections of one surface by batched GMRES on the dense matrices."""
    N, B, dev = dense.N, len(lam), _device()
    V, K = (torch.empty((N, N), device=dev, dtype=torch.float64) for _ in range(2))
    for i0, i1 in dense.blocks():
        V[i0:i1], K[i0:i1] = dense.rows(i0, i1)
    e = torch.from_numpy(eps.reshape(B)).to(dev)
    s = (e / EPS_WATER)[:, None]
    f = ((EPS_WATER - e) / EPS_WATER)[:, None]

    def real_mm(M, u):   # [B, N] complex
        return torch.view_as_complex((M @ torch.view_as_real(u).permute(1, 0, 2).reshape(N, 2 * B))
                                     .reshape(N, B, 2).contiguous()).T

    def op(u):
        kp, vd = real_mm(K, u[:, :N]), real_mm(V, u[:, N:])
        return torch.cat([0.5 * u[:, :N] + kp - vd, 0.5 * u[:, :N] - kp + s * vd], 1)

    vii = dense.self_v[None, :]

    def precond(u):
        a, b = u[:, :N], u[:, N:]
        return torch.cat([2.0 * (s * a + b) / (1.0 + s), (b - a) / (vii * (1.0 + s))], 1)

    dinc = -(dense.n @ torch.tensor(E0, device=dev, dtype=torch.float64))
    vinc = (V @ dinc)[None, :]
    b = torch.cat([torch.zeros((B, N), device=dev, dtype=torch.complex128), f * vinc], 1)
    beta = b.norm(dim=1)
    most = 200
    Q = torch.empty((most + 1, B, 2 * N), device=dev, dtype=torch.complex128)
    H = torch.zeros((B, most + 1, most), device=dev, dtype=torch.complex128)
    Q[0] = b / beta[:, None]
    for j in range(most):
        w = op(precond(Q[j]))
        for _ in range(2):
            h = torch.einsum("jbn,bn->bj", Q[:j + 1].conj(), w)
            H[:, :j + 1, j] += h
            w = w - torch.einsum("jbn,bj->bn", Q[:j + 1], h)
        H[:, j + 1, j] = w.norm(dim=1)
        Q[j + 1] = w / H[:, j + 1, j][:, None]
        if j % 10 == 9 or j == most - 1:
            g = torch.zeros((B, j + 2, 1), device=dev, dtype=torch.complex128)
            g[:, 0, 0] = beta
            Hj = H[:, :j + 2, :j + 1]
            y = torch.linalg.lstsq(Hj, g).solution
            if ((Hj @ y - g).norm(dim=(1, 2)) / beta).max() < 1e-11:
                break
    x = precond(torch.einsum("jbn,bj->bn", Q[:j + 1], y[:, :, 0]))
    phi, d1 = x[:, :N], x[:, N:]
    d2 = s * d1 - f * dinc[None, :]
    p = -EPS_WATER * ((dense.area * d2) @ dense.c.to(d2.dtype) - (dense.area * phi) @ dense.n.to(d2.dtype))
    k = torch.from_numpy(2.0 * np.pi * math.sqrt(EPS_WATER) / lam).to(dev)
    sigma = (k * k * p[:, 2] / EPS_WATER).imag / k
    return p, sigma


def exact(case, seed):
    n, B = _panels(case), case["B"]
    if case["kind"] == "solve":
        if n > 21000 or n * B > 400000:
            return None
    elif float(n) * n * (200 + 4 * B * _surfaces(case)) > 3.2e12:
        return None
    verts, tris, surf = _mesh(case, seed)
    dense = _Dense(verts, tris)
    lam, eps = _eps(case, seed)
    if case["kind"] == "solve":
        p, sigma = _solve(dense, lam, eps)
        return {"dipole": p, "sigma_ext": sigma}
    x = _vectors(case, seed, n)
    y = _product(dense, surf, x.reshape(B, 2 * n), torch.from_numpy((eps / EPS_WATER).reshape(B, -1)).to(x.device))
    y = y[0] if B == 1 else y
    return {"y": y, "sizes": None} if case["kind"] == "geometry" else {"y": y}
