"""The work that users of this library have it do, as cases that can be timed and compared.

Every case is one call of the public binding (``paper_1302_4018_gb300.hprobe.Context``) on synthetic
inputs of the shapes that the configurations, the tests and bench.py use: operator applications,
probing vectors, and trace estimates of Tr(A^-1) for the shifted Laplacian, the Wilson and the
clover-Wilson matrix and a general sparse matrix.  ``exact`` gives the same results from plain torch /
numpy in 64 bits: the Laplacian by its Fourier diagonalisation, the others by Krylov solves to
1e-13 with an operator written out here from its definition.

A case is a dict of plain values.  ``kind`` selects the call; ``L1`` .. ``L4`` are the extents (x_1
varies fastest); ``s`` is the number of probing vectors.
"""
import math

import numpy as np
import torch

from paper_1302_4018_gb300 import hprobe as hp

DEV = "cuda:0"


# ------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # one FP64 Wilson application on a small lattice: the building block of a user's own solver or
        # of a residual check, where the latency of the call is what counts
        _wilson("apply_8x8x8x8", "apply", (8, 8, 8, 8), nrhs=1),
        # the same for the twelve spin-colour sources of one point on a mid-sized lattice
        _wilson("apply_16x16x16x32", "apply", (16, 16, 16, 32), nrhs=12),
        # the vectors of a probing study written out: 512 vectors of the 64^3 grid with a random z_0
        {"name": "probes_64x64x64", "kind": "probes", "L1": 64, "L2": 64, "L3": 64, "L4": 1, "s": 512, "probe": "hp"},
        # the plain method at its smallest: 8^4 Laplacian, 256 vectors, CG to 1e-12 in FP64
        {"name": "laplace_8x8x8x8", "kind": "laplace", "L1": 8, "L2": 8, "L3": 8, "L4": 8, "s": 256,
         "mass": 0.05, "tol": 1e-12, "probe": "hp"},
        # the Laplacian of the variance studies: 64^3 at condition number 100
        {"name": "laplace_64x64x64", "kind": "laplace", "L1": 64, "L2": 64, "L3": 64, "L4": 1, "s": 32,
         "mass": 12.0 / 99.0, "tol": 1e-10, "probe": "hp"},
        # the default precision: a plain FP64 solve of the twelve sources of one probe
        _wilson("wilson_fp64_12x12x12x12", "trace", (12, 12, 12, 12), s=1, precision="fp64", even_odd=1),
        # many probes on a small lattice, binary16 iteration on the even-odd Schur complement
        _wilson("wilson_fp16_16x16x16x16", "trace", (16, 16, 16, 16), s=8, kappa=0.115, eps=0.3),
        # the headline workload: two probes (24 right-hand sides) on 32^3x64
        _wilson("wilson_fp16_32x32x32x64", "trace", (32, 32, 32, 64), s=2, kappa=0.12, eps=0.4),
        # extents with odd factors: no even-odd split, the full lattice is iterated, bfloat16 storage,
        # a per-site mass field
        _wilson("wilson_bf16_15x10x12x18", "trace", (15, 10, 12, 18), s=2, precision="bf16", even_odd=0, field=1),
        # the gradient with respect to a per-site mass field of the clover-Wilson matrix, FP32 iteration
        _wilson("grad_clover_fp32_16x16x16x32", "grad", (16, 16, 16, 32), s=2, precision="fp32", csw=1.0, field=1,
                tol=1e-11),
        # an uneven batch of lattices in one schedule
        {"name": "batch_fp16_8_12_16x32", "kind": "batch", "nlat": 3, "L1": 8, "L2": 8, "L3": 8, "L4": 8, "M1": 12,
         "M2": 12, "M3": 12, "M4": 12, "N1": 16, "N2": 16, "N3": 16, "N4": 32, "s": 8, "t": 4, "u": 2,
         "precision": "fp16", "even_odd": 1, "tol": 1e-10},
        # a general sparse matrix: the weighted graph Laplacian of a renumbered 64^3 grid with a
        # hierarchical colouring the user brings, FP32 iteration with FP64 reliable updates
        {"name": "sparse_fp32_64x64x64", "kind": "sparse", "L1": 64, "L2": 64, "L3": 64, "s": 32, "shift": 0.1,
         "precision": "fp32", "tol": 1e-10},
    ]


def _wilson(name, kind, dims, nrhs=0, s=0, precision="fp16", even_odd=1, kappa=0.12, eps=0.3, csw=0.0, field=0,
            tol=1e-10):
    c = {"kind": kind, "L1": dims[0], "L2": dims[1], "L3": dims[2], "L4": dims[3], "kappa": kappa, "eps": eps,
         "csw": csw, "field": field}
    if name:
        c["name"] = name
    if kind == "apply":
        c["nrhs"] = nrhs
    else:
        c.update(s=s, precision=precision, even_odd=even_odd, tol=tol)
    return c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "probes", "laplace", "trace", "trace", "trace", "grad", "batch", "sparse"])
    if kind == "apply":   # 4^4 .. 24^3x48, ragged extents among them
        nrhs = rng.randint(1, 12)
        dims = _extents(rng, 200, min(600000, 1600000 // nrhs), False)
        return _wilson(None, "apply", dims, nrhs=nrhs, csw=rng.choice([0.0, 0.0, 1.0]), field=rng.randint(0, 1))
    if kind == "probes":
        V = _log(rng, 4000, 500000)
        dims = _extents(rng, V // 2, V, False)
        n = 1 << sum(_twos(d) for d in dims)
        s = min(n, _log(rng, 16, 1024))
        return {"kind": "probes", "L1": dims[0], "L2": dims[1], "L3": dims[2], "L4": dims[3], "s": s,
                "probe": rng.choice(["hp", "hp", "z2"])}
    if kind == "laplace":
        V = _log(rng, 3000, 262144)
        dims = _extents(rng, V // 2, V, False)
        n = 1 << sum(_twos(d) for d in dims)
        tol = rng.choice([1e-10, 1e-12])
        s = min(n, _log(rng, 8, 256), max(1, 8000000 // V))
        return {"kind": "laplace", "L1": dims[0], "L2": dims[1], "L3": dims[2], "L4": dims[3], "s": s,
                "mass": rng.choice([0.05, 0.15, 0.5]), "tol": tol, "probe": rng.choice(["hp", "hp", "z2"])}
    if kind in ("trace", "grad"):
        precision = rng.choice(["fp16", "fp16", "fp32", "bf16", "fp64"])
        even_odd = rng.randint(0, 3) > 0
        V = _log(rng, 2000, 10000 if precision == "fp64" else 300000)
        dims = _extents(rng, V // 2, V, even_odd)
        n = 1 << sum(_twos(d) for d in dims)
        s = max(1, min(n, rng.randint(1, 8), 600000 // V))
        if precision == "fp64":
            s = 1
        return _wilson(None, kind, dims, s=s, precision=precision, even_odd=int(even_odd),
                       kappa=round(rng.uniform(0.10, 0.12), 4), eps=round(rng.uniform(0.2, 0.4), 3),
                       csw=rng.choice([0.0, 0.0, 1.0]), field=rng.randint(0, 1),
                       tol=1e-11 if kind == "grad" else 1e-10)
    if kind == "batch":
        c = {"kind": "batch", "nlat": 3, "precision": rng.choice(["fp16", "fp32", "bf16"]), "even_odd": 1, "tol": 1e-10}
        for p, q, hi in (("L", "s", 6000), ("M", "t", 40000), ("N", "u", 120000)):
            d = _extents(rng, hi // 4, hi, True)
            c.update({p + "1": d[0], p + "2": d[1], p + "3": d[2], p + "4": d[3], q: rng.randint(1, 8 if p == "L" else 3)})
        return c
    side = [2 * rng.randint(4, 32) for _ in range(3)]
    return {"kind": "sparse", "L1": side[0], "L2": side[1], "L3": side[2], "s": rng.choice([4, 8, 12, 16, 31, 32]),
            "shift": rng.choice([0.1, 0.3]), "precision": rng.choice(["fp32", "fp32", "fp64"]), "tol": 1e-10}


def _extents(rng, lo, hi, even):
    """Four extents (even ones where asked, any otherwise) of a volume in [lo, hi]."""
    while True:
        side = (lo * hi) ** 0.125
        d = []
        for _ in range(4):
            x = max(2, int(round(side * math.exp(rng.uniform(-0.6, 0.6)))))
            d.append(max(4, x + x % 2) if even else x)
        if lo <= d[0] * d[1] * d[2] * d[3] <= hi and min(d) >= 3:
            return d


def _twos(n):
    k = 0
    while n % 2 == 0:
        n //= 2
        k += 1
    return k


# ------------------------------------------------------------------------------------ inputs
def _dims(c, p="L"):
    return tuple(c[p + str(j)] for j in (1, 2, 3, 4))


def _seeded(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _links(V, eps, g):
    """U = exp(i eps H) with H traceless Hermitian from Gaussian numbers: complex128 [V, 4, 3, 3]."""
    out = torch.empty(V, 4, 3, 3, dtype=torch.complex128, device=DEV)
    eye = torch.eye(3, dtype=torch.complex128, device=DEV)
    for v0 in range(0, V, 1 << 18):
        n = min(1 << 18, V - v0)
        ab = torch.randn(2, n, 4, 3, 3, dtype=torch.float64, device=DEV, generator=g)
        H = torch.complex(ab[0], ab[1]) / math.sqrt(2.0)
        H = 0.5 * (H + H.mH)
        H = H - (torch.diagonal(H, dim1=-2, dim2=-1).sum(-1).real / 3.0)[..., None, None] * eye
        U = torch.linalg.matrix_exp(1j * eps * H)
        # re-unitarised to rounding: Gram-Schmidt on two rows, the third their conjugate cross product
        a = U[..., 0, :] / torch.linalg.vector_norm(U[..., 0, :], dim=-1, keepdim=True)
        b = U[..., 1, :] - (a.conj() * U[..., 1, :]).sum(-1, keepdim=True) * a
        b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
        out[v0:v0 + n] = torch.stack([a, b, torch.linalg.cross(a, b, dim=-1).conj()], dim=-2)
    return out


def _wilson_inputs(c, seed, p="L"):
    dims = _dims(c, p)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    g = _seeded(seed)
    U = _links(V, c.get("eps", 0.3), g)
    mu = 0.01 * torch.randn(V, dtype=torch.float64, device=DEV, generator=g) if c.get("field") else None
    return dims, V, U, mu, g


def _z0_seed(seed):
    return 2003 + 17 * int(seed)


def _grid_matrix(c, seed):
    """The weighted graph Laplacian + shift of a periodic grid with randomly renumbered rows (CSR with
    int32 indices, seven entries a row), and a two-level-per-scale colouring of the grid in the new
    numbering: parity, then the low coordinate bits that parity leaves open."""
    L = (c["L1"], c["L2"], c["L3"])
    n = L[0] * L[1] * L[2]
    g = _seeded(seed)
    new = torch.randperm(n, device=DEV, generator=g)
    site = torch.arange(n, device=DEV)
    x = [site % L[0], (site // L[0]) % L[1], site // (L[0] * L[1])]
    st = [1, L[0], L[0] * L[1]]
    cols, vals = [], []
    diag = torch.full((n,), float(c["shift"]), dtype=torch.float64, device=DEV)
    for j in range(3):
        w = 0.5 + torch.rand(n, dtype=torch.float64, device=DEV, generator=g)   # the edge site -> site + e_j
        up = site + torch.where(x[j] + 1 == L[j], st[j] * (1 - L[j]), st[j])
        dn = site + torch.where(x[j] == 0, st[j] * (L[j] - 1), -st[j])
        cols += [new[up], new[dn]]
        vals += [-w, -w[dn]]
        diag += w + w[dn]
    col = torch.stack([new] + cols, dim=1)
    val = torch.stack([diag] + vals, dim=1)
    col, order = torch.sort(col, dim=1)
    val = torch.gather(val, 1, order)
    ci = torch.empty_like(col)
    va = torch.empty_like(val)
    ci[new] = col
    va[new] = val
    rp = torch.arange(0, 7 * n + 1, 7, dtype=torch.int32, device=DEV)
    levels, radices = [], []
    for b in range(min(_twos(v) for v in L)):
        y = [(v >> b) & 1 for v in x]
        for lev, r in (((y[0] + y[1] + y[2]) & 1, 2), (y[0] + 2 * y[1], 4)):
            row = torch.empty(n, dtype=torch.int32, device=DEV)
            row[new] = lev.to(torch.int32)
            levels.append(row)
            radices.append(r)
    return n, rp, ci.to(torch.int32).reshape(-1).contiguous(), va.reshape(-1).contiguous(), torch.stack(levels), radices


def _sparse_vectors(c):
    """The vectors a case asks for, as far as its grid's colouring resolves them."""
    return min(c["s"], 8 ** min(_twos(c["L1"]), _twos(c["L2"]), _twos(c["L3"])))


def prepare(case, seed):
    c = dict(case, z0=_z0_seed(seed))
    ctx = hp.Context(0)
    st = {"case": c, "ctx": ctx}
    k = c["kind"]
    if k == "probes":
        V = c["L1"] * c["L2"] * c["L3"] * c["L4"]
        st["out"] = torch.empty(c["s"] * V, dtype=torch.int16, device=DEV)
    elif k == "laplace":
        st["op"] = ctx.make_operator(hp.OP_LAPLACIAN, c["mass"])
        st["opts"] = ctx.make_opts("fp64", z0_seed=c["z0"], probe_kind=c["probe"])
    elif k == "sparse":
        st["n"], st["rp"], st["ci"], st["val"], st["paths"], st["radices"] = _grid_matrix(c, seed)
        st["opts"] = ctx.make_opts(c["precision"], z0_seed=c["z0"])
    elif k == "batch":
        ops = []
        for i, p in enumerate("LMN"):
            _, _, U, _, _ = _wilson_inputs(dict(c, eps=0.2 + 0.1 * i), seed * 3 + i, p)
            ops.append(ctx.make_operator(hp.OP_WILSON, 0.0, 0.10 + 0.01 * i, U))
        st["ops"] = ops
        st["opts"] = ctx.make_opts(c["precision"], z0_seed=c["z0"], even_odd=c["even_odd"])
    else:
        dims, V, U, mu, g = _wilson_inputs(c, seed)
        st["op"] = ctx.make_operator(hp.OP_WILSON, 0.0, c["kappa"], U, mu, c["csw"])
        if k == "apply":
            v = torch.randn(2, c["nrhs"] * V * 12, dtype=torch.float64, device=DEV, generator=g)
            st["in"] = torch.complex(v[0], v[1]).reshape(c["nrhs"], V, 4, 3).contiguous()
            st["out"] = torch.empty_like(st["in"])
        else:
            st["opts"] = ctx.make_opts(c["precision"], z0_seed=c["z0"], even_odd=c["even_odd"])
            st["grad"] = torch.empty(V, dtype=torch.float64, device=DEV)
    return st


def run(st):
    c, ctx = st["case"], st["ctx"]
    k = c["kind"]
    if k == "apply":
        return ctx.operator_apply(st["op"], _dims(c), c["nrhs"], "fp64", st["in"], st["out"])
    if k == "probes":
        ctx.probe_vectors(_dims(c), 0, c["s"], c["z0"], st["out"], c["probe"])
        return st["out"]
    if k == "laplace":
        T, q, _ = ctx.trace_inv(st["op"], _dims(c), c["s"], c["tol"], st["opts"], np.zeros(c["s"], dtype=complex))
        return {"T": T, "q": q}
    if k == "sparse":
        s = _sparse_vectors(c)
        T, q, _ = ctx.trace_inv_sparse(st["rp"], st["ci"], st["val"], st["paths"], st["radices"], s, c["tol"],
                                       st["opts"], np.zeros(s, dtype=complex))
        return {"T": T, "q": q}
    if k == "batch":
        T, _ = ctx.trace_inv_batch(st["ops"], [_dims(c, p) for p in "LMN"], [c["s"], c["t"], c["u"]], c["tol"], st["opts"])
        return T
    if k == "grad":
        T, dm, _ = ctx.trace_inv_grad(st["op"], _dims(c), c["s"], c["tol"], st["opts"], st["grad"])
        return {"T": T, "dm": dm, "grad": st["grad"]}
    T, q, _ = ctx.trace_inv(st["op"], _dims(c), c["s"], c["tol"], st["opts"], np.zeros(c["s"], dtype=complex))
    return {"T": T, "q": q}


# ------------------------------------------------------------------------------------ the least work
def work(case):
    """Inputs read once and outputs written once; for the solves, the arithmetic of the least number of
    operator applications and vector updates that reach the tolerance, at the iteration counts that
    BiCGStab / CG take on these operators (22 on the Schur complement, twice that on the full lattice)."""
    c = case
    k = c["kind"]

    def wilson(V, s, eo, csw, tol):   # twelve solves a probe; 1368 flop a site and application, 504 more with clover
        n = 22.0 * math.log(tol) / math.log(1e-10) * (1.0 if eo else 2.0)
        return 12.0 * s * V * n * (2 * (1368.0 + (504.0 if csw else 0.0)) + 0.5 * (6 * 96) * (1 if eo else 2))

    if k == "sparse":
        n = c["L1"] * c["L2"] * c["L3"]
        s = _sparse_vectors(c)
        return {"bytes": n * (7 * 12.0 + 4.0) + 16.0 * 2 * s, "flops": 2.0 * s * n * 100 * (14 + 10)}
    V = c["L1"] * c["L2"] * c["L3"] * c["L4"]
    if k == "apply":
        return {"bytes": V * (576.0 + 384.0 * c["nrhs"] + 8.0 * c["field"]),
                "flops": c["nrhs"] * V * (1368.0 + (504.0 if c["csw"] else 0.0))}
    if k == "probes":
        return {"bytes": 2.0 * c["s"] * V, "flops": 0.0}
    if k == "laplace":
        cond = 1 + 16.0 / c["mass"]
        its = 0.35 * math.sqrt(cond) * math.log(2 / c["tol"])
        return {"bytes": 32.0 * c["s"], "flops": c["s"] * V * its * (10 + 10.0)}
    if k == "batch":
        b = f = 0.0
        for p, q in (("L", "s"), ("M", "t"), ("N", "u")):
            v = float(np.prod(_dims(c, p)))
            b += 576.0 * v
            f += wilson(v, c[q], True, False, c["tol"])
        return {"bytes": b, "flops": f}
    eo = c["even_odd"] and all(d % 2 == 0 for d in _dims(c))
    return {"bytes": V * (576.0 + 8.0 * c["field"] + (8.0 if k == "grad" else 0.0)),
            "flops": wilson(V, c["s"], eo, c["csw"], c["tol"])}


# ------------------------------------------------------------------------------------ 64-bit results
def _splitmix_sign(seed, index):
    """-1 where the top bit of output `index` of SplitMix64(seed) is set, else +1."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (index.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return 1.0 - 2.0 * (z >> np.uint64(63)).astype(np.float64)


def _parity(v):
    p = np.zeros_like(v)
    while v.any():
        p ^= v & 1
        v = v >> 1
    return p


def _probes(dims, s, seed, kind="hp"):
    """The first s hierarchical vectors (s <= 2^K: real, from the binary digits of the hierarchical
    position alone) times z_0, or Z_2 noise vectors: float64 [s, V] on the GPU."""
    V = int(np.prod(dims))
    if kind == "z2":
        return torch.from_numpy(_splitmix_sign(seed, np.arange(s * V)).reshape(s, V)).to(DEV)
    site = np.arange(V)
    x, r = [], site
    for d in dims:
        x.append(r % d)
        r = r // d
    ks = [_twos(d) for d in dims]
    K, pos = sum(ks), np.zeros(V, dtype=np.int64)
    for b in range(max(ks)):
        bits = [(x[j] >> b) & 1 for j in range(len(dims)) if b < ks[j]]
        i = np.zeros(V, dtype=np.int64)
        for y in bits:
            i = 2 * i + y
        pos = (pos << len(bits)) | (i >> 1) | (_parity(i) << (len(bits) - 1))
    z0 = _splitmix_sign(seed, site)
    out = np.empty((s, V))
    for m in range(s):
        col = int(format(m, "0%db" % K)[::-1], 2) if K else 0
        out[m] = z0 * (1.0 - 2.0 * _parity(pos & col))
    return torch.from_numpy(out).to(DEV)


def _prefix(q):
    q = np.asarray(q, dtype=complex)
    return np.cumsum(q) / np.arange(1, len(q) + 1)


_SIGMA = (((0, 1), (1, 0)), ((0, -1j), (1j, 0)), ((1, 0), (0, -1)))


class _Dirac:
    """D = A - kappa hop on fields [n, x4, x3, x2, x1, 4, 3], chiral gammas, periodic; A = 1 + mu(x) + C(x)."""

    def __init__(self, dims, U, kappa, mu=None, csw=0.0):
        self.shape = tuple(reversed(dims))
        self.U = [U.reshape(self.shape + (4, 3, 3))[..., m, :, :] for m in range(4)]
        self.kappa = kappa
        self.mu = None if mu is None else mu.reshape(self.shape)[..., None, None]
        off = [-1j * torch.tensor(s, dtype=torch.complex128, device=DEV) for s in _SIGMA]
        self.A = off + [torch.eye(2, dtype=torch.complex128, device=DEV)]   # g_mu = [[0, A], [A^H, 0]]
        self.clover = self._clover(csw) if csw else None

    def _sh(self, f, mu, n, lead=0):   # value at x + n e_mu
        return torch.roll(f, -n, dims=lead + 3 - mu)

    def _clover(self, csw):
        U, V = self.U, int(np.prod(self.shape))
        z = torch.zeros(2, 2, dtype=torch.complex128, device=DEV)
        gam = [torch.cat([torch.cat([z, a], 1), torch.cat([a.mH, z], 1)], 0) for a in self.A]
        C = torch.zeros(V, 4, 3, 4, 3, dtype=torch.complex128, device=DEV)
        for m in range(4):
            for n in range(m + 1, 4):
                a, b = U[m], U[n]
                am, bn = self._sh(a, m, -1), self._sh(b, n, -1)
                Q = a @ self._sh(b, m, 1) @ self._sh(a, n, 1).mH @ b.mH
                Q = Q + b @ self._sh(am, n, 1).mH @ self._sh(b, m, -1).mH @ am
                Q = Q + am.mH @ self._sh(self._sh(b, m, -1), n, -1).mH @ self._sh(am, n, -1) @ bn
                Q = Q + bn.mH @ self._sh(a, n, -1) @ self._sh(bn, m, 1) @ a.mH
                F = (Q - Q.mH) / 8j
                F = F - (torch.diagonal(F, dim1=-2, dim2=-1).sum(-1) / 3)[..., None, None] * torch.eye(3, device=DEV)
                sig = 0.5j * (gam[m] @ gam[n] - gam[n] @ gam[m])
                C -= csw * self.kappa * torch.einsum("st,vab->vsatb", sig, F.reshape(V, 3, 3))
        return C.reshape(V, 12, 12)

    def __call__(self, p):
        out = p * (1.0 if self.mu is None else 1.0 + self.mu)
        if self.clover is not None:
            n = p.shape[0]
            out = out + torch.einsum("vij,nvj->nvi", self.clover, p.reshape(n, -1, 12)).reshape(p.shape)
        up, dn = p[..., :2, :], p[..., 2:, :]
        for m in range(4):
            A = self.A[m]
            Ad = torch.einsum("st,...tc->...sc", A, dn)
            # forward: (1 - g) U(x) psi(x + mu); backward: (1 + g) U(x - mu)^H psi(x - mu)
            h = torch.einsum("...ab,n...sb->n...sa", self.U[m], self._sh(up - Ad, m, 1, 1))
            out[..., :2, :] -= self.kappa * h
            out[..., 2:, :] += self.kappa * torch.einsum("st,...tc->...sc", A.mH, h)
            h = self._sh(torch.einsum("...ba,n...sb->n...sa", self.U[m].conj(), up + Ad), m, -1, 1)
            out[..., :2, :] -= self.kappa * h
            out[..., 2:, :] -= self.kappa * torch.einsum("st,...tc->...sc", A.mH, h)
        return out


def _bicgstab(D, b, tol=1e-13, most=400):
    """D x = b for all fields of b at once (the iteration of each goes on until all are done, restarted
    from the true residual)."""
    n = b.shape[0]

    def dot(u, v):
        return (u.reshape(n, -1).conj() * v.reshape(n, -1)).sum(1)

    def bc(a):
        return a.reshape((n,) + (1,) * (b.dim() - 1))

    def ratio(u, v):
        return torch.where(v == 0, torch.zeros_like(u), u / torch.where(v == 0, torch.ones_like(v), v))

    x = torch.zeros_like(b)
    nb = dot(b, b).real
    for _ in range(4):
        r = b - D(x)
        if float((dot(r, r).real / nb).max()) <= tol * tol:
            break
        rh, p, rho = r.clone(), r.clone(), dot(r, r)
        for it in range(most):
            v = D(p)
            al = ratio(rho, dot(rh, v))
            s = r - bc(al) * v
            t = D(s)
            om = ratio(dot(t, s), dot(t, t))
            x += bc(al) * p + bc(om) * s
            r = s - bc(om) * t
            if it % 4 == 3 and float((dot(r, r).real / nb).max()) <= 0.25 * tol * tol:
                break
            new = dot(rh, r)
            be = ratio(new, rho) * ratio(al, om)
            rho = new
            p = r + bc(be) * (p - bc(om) * v)
    return x


def _wilson_exact(dims, U, kappa, mu, csw, s, seed, grad):
    V = int(np.prod(dims))
    D = _Dirac(dims, U, kappa, mu, csw)
    z = _probes(dims, s, seed)
    q = np.zeros(s, dtype=complex)
    g = torch.zeros(V, dtype=torch.float64, device=DEV)
    g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device=DEV)[:, None].expand(4, 3).reshape(12)
    for m in range(s):
        b = torch.zeros(12, V, 12, dtype=torch.complex128, device=DEV)
        for a in range(12):
            b[a, :, a] = z[m].to(torch.complex128)
        x = _bicgstab(D, b.reshape((12,) + D.shape + (4, 3))).reshape(12, V, 12)
        q[m] = complex((b.conj() * x).sum())
        if grad:   # the adjoint solution is g5_a g5 x_a
            g -= torch.einsum("a,c,avc->v", g5, g5, x.real ** 2 + x.imag ** 2) / s
    return q, g


def exact(case, seed):
    c = dict(case, z0=_z0_seed(seed))
    k = c["kind"]
    if k == "probes":
        return None   # whole numbers
    if k == "laplace":
        dims = _dims(c)
        sh = tuple(reversed(dims))
        lam = torch.full(sh, 8.0 + c["mass"], dtype=torch.float64, device=DEV)
        for j, d in enumerate(dims):
            w = 2 * torch.cos(2 * math.pi * torch.arange(d, dtype=torch.float64, device=DEV) / d)
            lam = lam - w.reshape([d if i == 3 - j else 1 for i in range(4)])
        q = []
        for z in _probes(dims, c["s"], c["z0"], c["probe"]):
            f = torch.fft.fftn(z.reshape(sh).to(torch.complex128))
            q.append(float(((f.real ** 2 + f.imag ** 2) / lam).sum()) / z.numel())
        return {"T": _prefix(q), "q": np.asarray(q, dtype=complex)}
    if k == "sparse":
        n, rp, ci, val, paths, radices = _grid_matrix(c, seed)
        s = _sparse_vectors(c)
        ci, val = ci.reshape(n, 7).long(), val.reshape(n, 7)

        def mul(x):
            y = torch.zeros_like(x)
            for j in range(7):
                y += val[:, j, None] * x[ci[:, j]]
            return y

        m = torch.arange(s, device=DEV)
        ph = torch.zeros(n, s, dtype=torch.float64, device=DEV)
        for lev, r in zip(paths, radices):
            ph += ((m % r)[None, :] * lev[:, None].long() % r).double() / r
            m = m // r
        z0 = torch.from_numpy(_splitmix_sign(c["z0"], np.arange(n))).to(DEV)[:, None]
        b = torch.cat([z0 * torch.cos(2 * math.pi * ph), z0 * torch.sin(2 * math.pi * ph)], dim=1)
        b = torch.where(b.abs() < 1e-12, torch.zeros_like(b), b)
        x, r = torch.zeros_like(b), b.clone()
        p, rr, bb = r.clone(), (b * b).sum(0), (b * b).sum(0).clamp_min(1e-300)
        for it in range(3000):
            Ap = mul(p)
            al = rr / (p * Ap).sum(0).clamp_min(1e-300)
            x += al * p
            r -= al * Ap
            new = (r * r).sum(0)
            if it % 8 == 7 and float((new / bb).max()) < 1e-26:
                break
            p = r + (new / rr.clamp_min(1e-300)) * p
            rr = new
        q = (b * x).sum(0).reshape(2, s).sum(0).cpu().numpy()
        return {"T": _prefix(q), "q": q.astype(complex)}
    if k == "batch":
        out = []
        for i, (p, s) in enumerate((("L", "s"), ("M", "t"), ("N", "u"))):
            dims, V, U, _, _ = _wilson_inputs(dict(c, eps=0.2 + 0.1 * i), seed * 3 + i, p)
            out.append(_prefix(_wilson_exact(dims, U, 0.10 + 0.01 * i, None, 0.0, c[s], c["z0"], False)[0]))
        return out
    dims, V, U, mu, g = _wilson_inputs(c, seed)
    if k == "apply":
        v = torch.randn(2, c["nrhs"] * V * 12, dtype=torch.float64, device=DEV, generator=g)
        D = _Dirac(dims, U, c["kappa"], mu, c["csw"])
        y = D(torch.complex(v[0], v[1]).reshape((c["nrhs"],) + D.shape + (4, 3)))
        return y.reshape(c["nrhs"], V, 4, 3)
    if V * c["s"] > 600000:
        return None   # over 20 seconds of 64-bit solves
    q, gr = _wilson_exact(dims, U, c["kappa"], mu, c["csw"], c["s"], c["z0"], k == "grad")
    if k == "grad":
        return {"T": _prefix(q), "dm": float(gr.sum()), "grad": gr}
    return {"T": _prefix(q), "q": q}
