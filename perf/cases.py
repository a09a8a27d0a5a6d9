"""What this library is used for, as calls that can be timed.

Every case goes through the public binding (``paper_2503_16994_gb300.lqcd``, or
the C ABI behind it where the binding has no device form) with inputs on the
GPU.  Lattices, couplings and masses are those of this repository's benchmark
and tests: SU(3) links exp(i eps H), kappa 0.120 to 0.132, c_sw 1.0 to 1.7,
antiperiodic time.  Solves stop at a true residual of 1e-12, between the
library's default (1e-10) and the paper's example (1e-13): tight enough that
two correct solvers agree to 1e-9 in the solution.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2503_16994_gb300 import lqcd

DEV = "cuda"
TOL = 1e-12
THETA = (1.0, 1.0, 1.0, -1.0)


def _case(name, kind, dims, **more):
    c = {"name": name, "kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3]}
    c.update(more)
    return c


def listed():
    return [
        # one FP64 Dirac application on the smallest test lattice: launches and latency
        _case("dirac_4c4", "dirac", (4, 4, 4, 4), kappa=0.120, csw=1.0, eps=0.2, mu=0.0, bc="periodic", dagger=False),
        # the same on the benchmark's lattice, adjoint: residual checks and sequential sources of a production run
        _case("dirac_32c64_dag", "dirac", (32, 32, 32, 64), kappa=0.132, csw=1.7, eps=0.4, mu=0.0, bc="periodic",
              dagger=True),
        # the plain FP64 solve of one point source (the benchmark's first configuration)
        _case("point_4c4_fp64", "solve", (4, 4, 4, 4), kappa=0.120, csw=1.0, eps=0.2, mu=0.0, bc="periodic",
              nrhs=1, prec="fp64", source="point"),
        # one noise source on the benchmark's lattice: stochastic estimators, one right-hand side at a time
        _case("noise_32c64_fp16", "solve", (32, 32, 32, 64), kappa=0.132, csw=1.7, eps=0.4, mu=0.0, bc="periodic",
              nrhs=1, prec="fp16", source="noise"),
        # twisted mass on a ragged lattice, a few sources at once
        _case("twisted_12c10x24_fp16", "solve", (12, 12, 10, 24), kappa=0.130, csw=1.5, eps=0.4, mu=0.05,
              bc="periodic", nrhs=5, prec="fp16", source="noise"),
        # the 12-column propagator and its pion correlator, FP32 inner vectors (the benchmark's second configuration)
        _case("pion_16c32_fp32", "pion", (16, 16, 16, 32), kappa=0.130, csw=1.5, eps=0.4, mu=0.0, bc="periodic",
              nrhs=12, prec="fp32"),
        # the flagship: 12 columns in FP16 storage on the largest of the batched sizes
        _case("pion_24c48_fp16", "pion", (24, 24, 24, 48), kappa=0.132, csw=1.7, eps=0.4, mu=0.0, bc="periodic",
              nrhs=12, prec="fp16"),
        # propagators on uneven small lattices in one call (served requests, parameter scans)
        _case("batch_uneven_fp16", "batch", (8, 8, 8, 16), sizes="8x8x8x16,12x12x12x24,8x8x8x16,6x8x10x12",
              kappa=0.126, csw=1.5, eps=0.3, prec="fp16"),
        # the Wilson flow with its observables on 32^4
        _case("flow_32c32", "flow", (32, 32, 32, 32), eps=0.4, steps=2, step=0.01),
        # twelve quark fields flowed with the links
        _case("fermion_flow_16c32", "fermion_flow", (16, 16, 16, 32), eps=0.4, steps=2, step=0.01, nrhs=12),
        # the adjoint flow of a few fields from checkpoints
        _case("backflow_12c24", "backflow", (12, 12, 12, 24), eps=0.4, steps=4, step=0.02, nrhs=6, nsave=2),
        # all sixteen meson channels of a propagator on the benchmark's lattice
        _case("meson_32c64", "meson", (32, 32, 32, 64), ng=16),
    ]


def _dims(rng, vmax, vmin=16):
    """Even extents, spread over the logarithm of the volume, ragged more often than not."""
    while True:
        v = math.exp(rng.uniform(math.log(vmin * 16), math.log(vmax)))
        side = (v / 2) ** 0.25
        d = [max(2, 2 * round(side * math.exp(rng.uniform(-0.35, 0.35)) / 2)) for _ in range(3)]
        d.append(max(2, 2 * round(v / (d[0] * d[1] * d[2]) / 2)))
        if vmin <= d[0] * d[1] * d[2] * d[3] <= vmax and d[3] <= 96:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["dirac", "solve", "solve", "pion", "pion", "batch", "flow", "fermion_flow", "backflow", "meson"])
    c = {"kappa": round(rng.uniform(0.120, 0.132), 5), "csw": round(rng.uniform(1.0, 1.7), 3),
         "eps": round(rng.uniform(0.2, 0.4), 3)}
    prec = rng.choice(["fp16", "fp16", "fp32", "fp64"])
    step = round(rng.uniform(0.005, 0.02), 5)
    if kind == "dirac":
        return _drop(_case("", kind, _dims(rng, 2 ** 21, 256), **c, mu=rng.choice([0.0, 0.0, 0.05]),
                           bc=rng.choice(["periodic", "periodic", "open"]), dagger=rng.random() < 0.5))
    if kind == "solve":
        nrhs, mu = rng.choice([1, 1, 2, 3, 5, 6, 8, 12]), rng.choice([0.0, 0.0, 0.03, 0.08])
        most = 2 ** 21 // {"fp16": 1, "fp32": 8, "fp64": 64}[prec] // (4 if mu else 1)
        return _drop(_case("", kind, _dims(rng, max(512, most // nrhs), 256), **c, mu=mu,
                           bc=rng.choice(["periodic", "periodic", "open"]), nrhs=nrhs, prec=prec,
                           source=rng.choice(["noise", "point"])))
    if kind == "pion":
        return _drop(_case("", kind, _dims(rng, {"fp16": 400000, "fp32": 150000, "fp64": 8000}[prec], 256), **c,
                           mu=0.0, bc="periodic", nrhs=12, prec=prec))
    if kind == "batch":
        sizes = ["x".join(map(str, _dims(rng, 30000, 256))) for _ in range(rng.randint(2, 4))]
        first = tuple(int(v) for v in sizes[0].split("x"))
        return _drop(_case("", kind, first, sizes=",".join(sizes), prec=rng.choice(["fp16", "fp32"]), **c))
    if kind == "flow":
        return _drop(_case("", kind, _dims(rng, 2 ** 20, 256), eps=c["eps"], steps=rng.randint(1, 2), step=step))
    if kind == "fermion_flow":
        n = rng.choice([1, 2, 3, 4, 6, 12])
        return _drop(_case("", kind, _dims(rng, 131072, 256), eps=c["eps"], steps=rng.randint(1, 2), step=step,
                           nrhs=n))
    if kind == "backflow":
        return _drop(_case("", kind, _dims(rng, 41472, 256), eps=c["eps"], steps=rng.randint(2, 4), step=step,
                           nrhs=rng.choice([1, 2, 3, 6]), nsave=rng.randint(1, 3)))
    return _drop(_case("", kind, _dims(rng, 2 ** 21, 256), ng=rng.choice([1, 3, 16])))


def _drop(c):
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _links(dims, eps, g):
    """Near-unit SU(3) links: 1 + i eps H - (eps H)^2 / 2 for a Gaussian traceless Hermitian H, made special
    unitary by Gram-Schmidt and the cross product; complex128 [T, Z, Y, X, 4, 3, 3] on the GPU."""
    lx, ly, lz, lt = dims
    h = torch.randn(lt * lz * ly * lx * 4, 8, dtype=torch.float64, device=DEV, generator=g) * (0.5 * eps)
    r3 = 1.0 / math.sqrt(3.0)
    z = torch.zeros_like(h[:, 0])
    re = torch.stack([h[:, 2] + r3 * h[:, 7], h[:, 0], h[:, 3], h[:, 0], -h[:, 2] + r3 * h[:, 7], h[:, 5],
                      h[:, 3], h[:, 5], -2 * r3 * h[:, 7]], 1)
    im = torch.stack([z, -h[:, 1], -h[:, 4], h[:, 1], z, -h[:, 6], h[:, 4], h[:, 6], z], 1)
    H = torch.complex(re, im).reshape(-1, 3, 3)
    a, b = [], []
    for k, out in ((0, a), (1, b)):  # the first two rows of 1 + iH - H^2 / 2
        for c in range(3):
            hh = H[:, k, 0] * H[:, 0, c] + H[:, k, 1] * H[:, 1, c] + H[:, k, 2] * H[:, 2, c]
            out.append((1.0 if k == c else 0.0) + 1j * H[:, k, c] - 0.5 * hh)
    a = torch.stack(a, 1)
    b = torch.stack(b, 1)
    a = a / torch.linalg.vector_norm(a, dim=1, keepdim=True)
    b = b - (a.conj() * b).sum(1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=1, keepdim=True)
    c = torch.stack([a[:, 1] * b[:, 2] - a[:, 2] * b[:, 1], a[:, 2] * b[:, 0] - a[:, 0] * b[:, 2],
                     a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]], 1).conj()
    return torch.stack([a, b, c], 1).reshape(lt, lz, ly, lx, 4, 3, 3)


def _spinors(dims, n, g):
    lx, ly, lz, lt = dims
    return torch.randn(n, lt, lz, ly, lx, 4, 3, dtype=torch.complex128, device=DEV, generator=g)


def _sources(case, dims, g):
    """Right-hand sides: full-lattice Gaussian noise, or point sources at one random site, spin-colours in turn."""
    n = case["nrhs"]
    if case["source"] == "noise":
        return _spinors(dims, n, g)
    lx, ly, lz, lt = dims
    b = torch.zeros(n, lt, lz, ly, lx, 4, 3, dtype=torch.complex128, device=DEV)
    x, y, z, t = _site(dims, g)
    for j in range(n):
        b[j, t, z, y, x, (j % 12) // 3, j % 3] = 1.0
    return b


def _site(dims, g):
    r = torch.randint(0, 1 << 30, (4,), device=DEV, generator=g).tolist()
    return tuple(v % d for v, d in zip(r, dims))


class _Lattice:
    """A lattice handle with one resident gauge field, freed with its state."""

    def __init__(self, dims, links):
        self.dims = dims
        self.lat = lqcd.lattice_create(dims)
        self.gid = lqcd.gauge_upload(self.lat, links.cpu().numpy())

    def links(self, out):
        """The resident links into a CUDA tensor (the binding's form returns host arrays)."""
        rc = lqcd.load().lqcd_gauge_download(self.lat, self.gid, ctypes.c_void_p(out.data_ptr()), lqcd.DEVICE_PTRS,
                                             None)
        if rc != lqcd.OK:
            raise lqcd.LqcdError(rc, lqcd.last_error())
        return out

    def __del__(self):
        if getattr(self, "lat", None) is not None:
            lqcd.lattice_destroy(self.lat)
            self.lat = None


def _shape(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def _sizes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["sizes"].split(",")]


def _params(case):
    return lqcd.dirac_params(case["kappa"], case["csw"], THETA, mu=case.get("mu", 0.0), bc=case.get("bc", "periodic"))


def _gammas(n):
    """The first n of the sixteen Clifford elements (chiral basis), g5 first."""
    s = [np.array(m, dtype=complex) for m in ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]
    o, e = np.zeros((2, 2)), np.eye(2)
    gk = [np.block([[o, -1j * m], [1j * m, o]]) for m in s]
    gt = np.block([[o, -e], [-e, o]]).astype(complex)
    g5 = np.diag([1, 1, -1, -1]).astype(complex)
    g4 = gk + [gt]
    out = [g5, np.eye(4, dtype=complex)] + g4 + [g5 @ m for m in g4]
    out += [g4[a] @ g4[b] for a in range(4) for b in range(a + 1, 4)]
    return np.stack(out[:n])


def prepare(case, seed):
    g = _gen(seed)
    kind, dims = case["kind"], _shape(case)
    st = {"case": dict(case)}
    if kind == "meson":
        lx, ly, lz, lt = dims
        st["lat"] = _Lattice.__new__(_Lattice)  # the contraction needs the geometry only
        st["lat"].dims, st["lat"].lat = dims, lqcd.lattice_create(dims)
        st["prop"] = _spinors(dims, 12, g)
        st["src_t"] = _site(dims, g)[3]
        st["gammas"] = _gammas(case["ng"])
        st["corr"] = torch.empty(case["ng"], lt, dtype=torch.complex128, device=DEV)
        return st
    if kind == "batch":
        st["lats"] = [_Lattice(d, _links(d, case["eps"], g)) for d in _sizes(case)]
        st["jobs"] = [(L.lat, L.gid, lqcd.dirac_params(case["kappa"] - 0.0007 * k, case["csw"], THETA),
                       _site(L.dims, g), L.dims[3]) for k, L in enumerate(st["lats"])]
        st["sp"] = lqcd.solver_params(tol=TOL, maxiter=20000, precision=case["prec"])
        return st
    st["lat"] = _Lattice(dims, _links(dims, case["eps"], g))
    if kind in ("flow", "fermion_flow"):
        st["links"] = torch.empty(dims[3], dims[2], dims[1], dims[0], 4, 3, 3, dtype=torch.complex128, device=DEV)
    if kind in ("fermion_flow", "backflow"):
        st["dp"] = lqcd.dirac_params(0.13, 0.0, THETA)
        st["psi"] = _spinors(dims, case["nrhs"], g)
        st["out"] = torch.empty_like(st["psi"])
    if kind == "dirac":
        st["dp"] = _params(case)
        st["psi"] = _spinors(dims, 1, g)[0]
        st["out"] = torch.empty_like(st["psi"])
    if kind == "solve":
        st["dp"] = _params(case)
        st["sp"] = lqcd.solver_params(tol=TOL, maxiter=20000, precision=case["prec"])
        st["b"] = _sources(case, dims, g)
        st["x"] = torch.empty_like(st["b"])
    if kind == "pion":
        st["dp"] = _params(case)
        st["sp"] = lqcd.solver_params(tol=TOL, maxiter=20000, precision=case["prec"])
        st["src"] = _site(dims, g)
        st["corr"] = torch.empty(dims[3], dtype=torch.float64, device=DEV)
        st["prop"] = torch.empty(12, dims[3], dims[2], dims[1], dims[0], 4, 3, dtype=torch.complex128, device=DEV)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        return lqcd.pion_corr_batch(st["jobs"], st["sp"])[0]
    L = st["lat"]
    if kind == "meson":
        return lqcd.meson_contract(L.lat, st["prop"], st["src_t"], st["gammas"], corr=st["corr"])
    if kind == "dirac":
        return lqcd.dirac_apply(L.lat, L.gid, st["dp"], st["psi"], out=st["out"], dagger=case["dagger"])
    if kind == "solve":
        return lqcd.cg_solve(L.lat, L.gid, st["dp"], st["sp"], st["b"], nrhs=case["nrhs"], x=st["x"])[0]
    if kind == "pion":
        corr, prop, _, _ = lqcd.pion_corr(L.lat, L.gid, st["dp"], st["sp"], st["src"],
                                          device_out=(st["corr"], st["prop"]))
        return corr, prop
    if kind == "flow":  # the links keep flowing from call to call, as along a flow trajectory
        lqcd.gauge_flow(L.lat, L.gid, case["step"], case["steps"])
        plaq, ep, ec, q = lqcd.gauge_observables(L.lat, L.gid, L.dims[3])
        return plaq, ep, ec, q, L.links(st["links"])
    st["out"].copy_(st["psi"])
    if kind == "fermion_flow":
        psi = lqcd.fermion_flow(L.lat, L.gid, st["dp"], st["out"], case["step"], case["steps"], nrhs=case["nrhs"])
        return psi, L.links(st["links"])
    return lqcd.fermion_backflow(L.lat, L.gid, st["dp"], st["out"], case["step"], case["steps"], nrhs=case["nrhs"],
                                 nsave=case["nsave"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
HOP = 1320.0         # eight projected SU(3) products and their sums, per site
CLOVER = 504.0       # two 6x6 Hermitian blocks on a spinor
PRODUCT = 198.0      # 3x3 complex matrix product
LINKS = 4 * 144.0    # FP64 links of a site
SPINOR = 192.0       # FP64 spinor of a site
DECADE = 35.0        # CG iterations on D^dag D per decade of the residual at these masses (about 430 for 1e-12)


def _solve_work(v, n, tol, read, written):
    iters = DECADE * -math.log10(tol)
    return {"bytes": v * (LINKS + (read + written) * SPINOR), "flops": iters * n * v * 2.0 * (HOP + CLOVER)}


def work(case):
    kind, dims = case["kind"], _shape(case)
    v = float(dims[0] * dims[1] * dims[2] * dims[3])
    if kind == "dirac":
        return {"bytes": v * (LINKS + 2 * SPINOR), "flops": v * (HOP + CLOVER + 24)}
    if kind == "solve":
        return _solve_work(v, case["nrhs"], TOL, case["nrhs"], case["nrhs"])
    if kind == "pion":
        return _solve_work(v, 12, TOL, 0, 12)
    if kind == "batch":
        w = [_solve_work(float(np.prod(d)), 12, TOL, 0, 0) for d in _sizes(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    # per link and stage: 13 products of the staples, 1 of the update, the exponential as a quadratic in X
    stage = 4 * (13 + 1 + 2) * PRODUCT
    laplace = 8 * 4 * 72.0 + 4 * 48.0
    if kind == "flow":
        return {"bytes": v * 2 * LINKS, "flops": v * (3 * case["steps"] * stage + 6 * 20 * PRODUCT)}
    if kind == "fermion_flow":
        n = case["nrhs"]
        return {"bytes": v * (2 * LINKS + 2 * n * SPINOR), "flops": v * 3 * case["steps"] * (stage + n * laplace)}
    if kind == "backflow":
        n = case["nrhs"]
        return {"bytes": v * (LINKS + 2 * n * SPINOR), "flops": v * case["steps"] * (5 * stage + 3 * n * laplace)}
    # one colour inner product of 9 complex terms for each pair of the 16 blocks that a channel needs, at most 136
    pairs = min(136, 16 * case["ng"])
    return {"bytes": v * 12 * SPINOR, "flops": v * pairs * 72.0}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------
AXIS = (3, 2, 1, 0)  # x, y, z, t in [T, Z, Y, X, ...]


def _sigma():
    g = torch.tensor(_gammas(6)[2:], device=DEV)  # x, y, z, t
    return g


def _leaf_field(U, mu, nu):
    """F_{mu nu} = (Q - Q^dag) / 8 without its trace, Q the four leaves, each walked mu first."""
    def at(m, *shifts):
        w = U[..., m, :, :]
        for d, s in shifts:
            w = torch.roll(w, -s, AXIS[d])
        return w

    def dg(a):
        return a.conj().transpose(-1, -2)

    q = at(mu) @ at(nu, (mu, 1)) @ dg(at(mu, (nu, 1))) @ dg(at(nu))
    q = q + at(nu) @ dg(at(mu, (mu, -1), (nu, 1))) @ dg(at(nu, (mu, -1))) @ at(mu, (mu, -1))
    q = q + dg(at(mu, (mu, -1))) @ dg(at(nu, (mu, -1), (nu, -1))) @ at(mu, (mu, -1), (nu, -1)) @ at(nu, (nu, -1))
    q = q + dg(at(nu, (nu, -1))) @ at(mu, (nu, -1)) @ at(nu, (mu, 1), (nu, -1)) @ dg(at(mu))
    f = (q - dg(q)) / 8
    tr = (f[..., 0, 0] + f[..., 1, 1] + f[..., 2, 2]) / 3
    return f - tr[..., None, None] * torch.eye(3, dtype=f.dtype, device=f.device), q


class _Plain:
    """D psi for fields [T, Z, Y, X, 3, 4 n] (colour rows; spin, field columns)."""

    def __init__(self, U, case):
        self.k, self.g = case["kappa"], _sigma()
        U = U.clone()
        if case.get("bc") == "open":
            U[-1, ..., 3, :, :] = 0
        V = U.shape[:4]
        term = torch.zeros(*V, 4, 3, 4, 3, dtype=U.dtype, device=U.device)
        eye4 = torch.eye(4, dtype=U.dtype, device=U.device)
        for mu in range(4):
            for nu in range(mu + 1, 4):
                s = 0.5j * (self.g[mu] @ self.g[nu] - self.g[nu] @ self.g[mu])
                f = _leaf_field(U, mu, nu)[0]
                term += 1j * self.k * case["csw"] * torch.einsum("st,...ab->...satb", s, f)
        for a in range(3):
            term[..., :, a, :, a] += eye4
            if case.get("mu"):
                term[..., :, a, :, a] += 2j * self.k * case["mu"] * torch.diag(
                    torch.tensor([1, 1, -1, -1], dtype=U.dtype, device=U.device))
        self.site = term.reshape(*V, 12, 12)
        if case.get("bc") != "open":
            for d in range(4):
                idx = [slice(None)] * 4
                idx[AXIS[d]] = -1
                U[tuple(idx)][..., d, :, :] *= THETA[d]
        self.U = U

    def __call__(self, psi, dagger=False):
        V, n = psi.shape[:4], psi.shape[-1] // 4
        p = psi.reshape(*V, 3, 4, n)
        site = self.site.conj().transpose(-1, -2) if dagger else self.site
        out = (site @ p.transpose(-3, -2).reshape(*V, 12, n)).reshape(*V, 4, 3, n).transpose(-3, -2)
        eye = torch.eye(4, dtype=psi.dtype, device=psi.device)
        for mu in range(4):
            for d in (1, -1):
                P = eye - d * (-1 if dagger else 1) * self.g[mu]
                h = torch.einsum("st,...ctn->...csn", P, torch.roll(p, -d, AXIS[mu])).reshape(*V, 3, 4 * n)
                W = self.U[..., mu, :, :]
                if d < 0:
                    W = torch.roll(W, 1, AXIS[mu]).conj().transpose(-1, -2)
                out = out - self.k * (W @ h).reshape(*V, 3, 4, n)
        return out.reshape(*V, 3, 4 * n)


def _to_plain(psi):  # [n, T, Z, Y, X, 4, 3] -> [T, Z, Y, X, 3, 4 n]
    n = psi.shape[0]
    return psi.permute(1, 2, 3, 4, 6, 5, 0).reshape(*psi.shape[1:5], 3, 4 * n).contiguous()


def _from_plain(p):
    n = p.shape[-1] // 4
    return p.reshape(*p.shape[:5], 4, n).permute(6, 0, 1, 2, 3, 5, 4).contiguous()


def _solve_plain(D, b, tol=2e-15):
    """CG on the normal equations, restarted from the true residual until it stops falling."""
    n = b.shape[-1] // 4

    def dot(a, c):
        return (a.conj() * c).reshape(-1, 4, n).real.sum((0, 1))

    def by(s, v):
        return (v.reshape(*v.shape[:-1], 4, n) * s).reshape(v.shape)

    x, bb = torch.zeros_like(b), dot(b, b)
    r, last = b.clone(), None
    for _ in range(4):
        z = D(r, True)
        p, gam = z.clone(), dot(z, z)
        e, rr0 = torch.zeros_like(b), dot(r, r)
        for it in range(4000):
            w = D(p)
            al = gam / dot(w, w).clamp_min(1e-300)
            e = e + by(al, p)
            r = r - by(al, w)
            z = D(r, True)
            new = dot(z, z)
            p = z + by(new / gam.clamp_min(1e-300), p)
            gam = new
            if it % 10 == 9:
                rr = dot(r, r)
                if bool((rr <= torch.maximum(1e-16 * rr0, tol * tol * bb)).all()):
                    break
        x = x + e
        r = b - D(x)
        now = float((dot(r, r) / bb).max())
        if now <= tol * tol or (last is not None and now > 0.25 * last):
            break
        last = now
    return x


def _force(U):
    out = torch.zeros_like(U)

    def at(m, *shifts):
        w = U[..., m, :, :]
        for d, s in shifts:
            w = torch.roll(w, -s, AXIS[d])
        return w

    def dg(a):
        return a.conj().transpose(-1, -2)

    for mu in range(4):
        S = torch.zeros_like(U[..., 0, :, :])
        for nu in range(4):
            if nu != mu:
                S = S + at(nu, (mu, 1)) @ dg(at(mu, (nu, 1))) @ dg(at(nu))
                S = S + dg(at(nu, (mu, 1), (nu, -1))) @ dg(at(mu, (nu, -1))) @ at(nu, (nu, -1))
        om = U[..., mu, :, :] @ S
        Z = -0.5 * (om - dg(om))
        tr = (Z[..., 0, 0] + Z[..., 1, 1] + Z[..., 2, 2]) / 3
        out[..., mu, :, :] = Z - tr[..., None, None] * torch.eye(3, dtype=U.dtype, device=U.device)
    return out


def _expm(X):
    eye = torch.eye(3, dtype=X.dtype, device=X.device)
    Y = X / 64
    E = eye
    for k in range(14, 0, -1):
        E = eye + (Y @ E) / k
    for _ in range(6):
        E = E @ E
    return E


def _stages(U, eps):
    """The fields W0, W1, W2, W3 of one RK3 step."""
    X = 0.25 * eps * _force(U)
    W1 = _expm(X) @ U
    X = 8.0 / 9.0 * eps * _force(W1) - 17.0 / 9.0 * X
    W2 = _expm(X) @ W1
    X = 0.75 * eps * _force(W2) - X
    return U, W1, W2, _expm(X) @ W2


def _laplace(U, p):
    """Covariant Laplacian of [T, Z, Y, X, 3, m] with antiperiodic time."""
    out = -8.0 * p
    for mu in range(4):
        W = U[..., mu, :, :].clone()
        idx = [slice(None)] * 4
        idx[AXIS[mu]] = -1
        W[tuple(idx)] *= THETA[mu]
        out = out + W @ torch.roll(p, -1, AXIS[mu])
        out = out + torch.roll(W, 1, AXIS[mu]).conj().transpose(-1, -2) @ torch.roll(p, 1, AXIS[mu])
    return out


def _observables(U):
    eye = torch.eye(3, dtype=U.dtype, device=U.device)
    F, plaq, ep = {}, 0.0, 0.0

    def tr(a, b):
        return (a * b.transpose(-1, -2)).sum((-1, -2)).real

    for mu in range(4):
        for nu in range(mu + 1, 4):
            a, b = U[..., mu, :, :], U[..., nu, :, :]
            P = a @ torch.roll(b, -1, AXIS[mu]) @ torch.roll(a, -1, AXIS[nu]).conj().transpose(-1, -2) \
                @ b.conj().transpose(-1, -2)
            re = (P * eye).sum((-1, -2)).real
            plaq = plaq + re.sum() / 18.0 / re.numel()
            ep = ep + (2.0 * (3.0 - re)).sum((1, 2, 3))
            F[mu, nu] = _leaf_field(U, mu, nu)[0]
    ec = -sum(tr(f, f).sum((1, 2, 3)) for f in F.values())
    q = (tr(F[0, 1], F[2, 3]) - tr(F[0, 2], F[1, 3]) + tr(F[0, 3], F[1, 2])).sum((1, 2, 3))
    return float(plaq), ep.cpu().numpy(), ec.cpu().numpy(), (-8.0 / (32.0 * math.pi ** 2) * q).cpu().numpy()


def _contract_pion(prop, src_t):
    return torch.roll((prop.abs() ** 2).sum((0, 2, 3, 4, 5, 6)), -src_t)


def exact(case, seed):
    g = _gen(seed)
    kind, dims = case["kind"], _shape(case)
    v = dims[0] * dims[1] * dims[2] * dims[3]
    if kind == "meson":
        prop = _spinors(dims, 12, g)
        src_t = _site(dims, g)[3]
        gam = torch.tensor(_gammas(case["ng"]), device=DEV)
        g5, gt = torch.tensor(_gammas(1)[0], device=DEV), torch.tensor(_gammas(6)[5], device=DEV)
        out = torch.empty(case["ng"], dims[3], dtype=torch.complex128, device=DEV)
        for t in range(dims[3]):
            S = prop[:, t].reshape(4, 3, -1, 4, 3).permute(2, 3, 4, 0, 1)  # [x, sink spin, colour, source spin, colour]
            for k in range(case["ng"]):
                G = gam[k]
                right = (gt @ G.conj().T @ gt) @ g5
                A = torch.einsum("ab,xbcde,df->xacfe", G, S, right)
                B = torch.einsum("ab,xbcde->xacde", g5, S)
                out[k, (t - src_t) % dims[3]] = -(A * B.conj()).sum()
        return out
    if kind == "batch":
        if case["prec"] == "fp64" or max(np.prod(d) for d in _sizes(case)) > 8200:
            return None
        outs, Ls = [], []
        for d in _sizes(case):
            Ls.append(_links(d, case["eps"], g))
        for k, (d, U) in enumerate(zip(_sizes(case), Ls)):
            src = _site(d, g)
            D = _Plain(U, {"kappa": case["kappa"] - 0.0007 * k, "csw": case["csw"]})
            b = _point(d, src)
            outs.append(_contract_pion(_from_plain(_solve_plain(D, _to_plain(b))), src[3]).cpu().numpy())
        return outs
    U = _links(dims, case["eps"], g)
    if kind == "dirac":
        return _from_plain(_Plain(U, case)(_to_plain(_spinors(dims, 1, g)), case["dagger"]))[0]
    if kind == "solve":
        if v * case["nrhs"] > 40000:
            return None
        return _from_plain(_solve_plain(_Plain(U, case), _to_plain(_sources(case, dims, g))))
    if kind == "pion":
        if v > 4000:
            return None
        src = _site(dims, g)
        x = _from_plain(_solve_plain(_Plain(U, case), _to_plain(_point(dims, src))))
        return _contract_pion(x, src[3]), x
    if kind == "flow":
        for _ in range(case["steps"]):
            U = _stages(U, case["step"])[3]
        return (*_observables(U), U)
    eps = case["step"]
    p = _to_plain(_spinors(dims, case["nrhs"], g))
    if kind == "fermion_flow":
        for _ in range(case["steps"]):
            W = _stages(U, eps)
            d0 = _laplace(W[0], p)
            l1 = p + 0.25 * eps * d0
            l2 = p + 8.0 / 9.0 * eps * _laplace(W[1], l1) - 2.0 / 9.0 * eps * d0
            p = l1 + 0.75 * eps * _laplace(W[2], l2)
            U = W[3]
        return _from_plain(p), U
    steps = []
    for _ in range(case["steps"]):
        steps.append(_stages(U, eps))
        U = steps[-1][3]
    for W in reversed(steps):
        z2 = 0.75 * eps * _laplace(W[2], p)
        u = p + 8.0 / 9.0 * eps * _laplace(W[1], z2)
        p = u + z2 + _laplace(W[0], 0.25 * eps * u - 2.0 / 9.0 * eps * z2)
    return _from_plain(p)


def _point(dims, src):
    lx, ly, lz, lt = dims
    b = torch.zeros(12, lt, lz, ly, lx, 4, 3, dtype=torch.complex128, device=DEV)
    x, y, z, t = src
    for j in range(12):
        b[j, t, z, y, x, j // 3, j % 3] = 1.0
    return b
