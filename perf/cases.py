"""Timed cases of the library: the calls that a program computing sgn(H_w(mu)) x makes.

Every case goes through the Python binding with device tensors, as a program
that keeps its vectors on the GPU does. A state is one gauge field (a handle)
with its deflation basis installed and its sources in device memory, or, for
the batched form, several of them. Links are seeded near-identity SU(3)
matrices exp(i eps X), sources are unit complex Gaussians, and the deflation
vectors are seeded near-biorthonormal pairs (the formula of the method holds
for any such pair, and its cost does not depend on the pair).

The mixed form computes in 32 bits and its results carry single precision, so
programs that use it keep them as complex64; the FP64 form's results are kept
as complex128.
"""

import math

import numpy as np
import torch

import paper_0704_3486_gb300 as ovs

M_W = -1.5
DEV = "cuda"


def _case(name, kind, dims, nrhs, k, m, prec, eps, mu, **more):
    c = {"name": name, "kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3], "nrhs": nrhs, "k": k,
         "m": m, "prec": prec, "eps": eps, "mu": mu, "harmonic": False, "op": 1, "instances": 1, "cap": 0, "tol": 0.0}
    c.update(more)
    return c


def listed():
    return [
        # one operator application on the smallest lattice of the configurations: all latency
        _case("matvec 4^4 f64", "matvec", (4, 4, 4, 4), 1, 0, 0, "f64", 0.5, 0.3),
        # the operator in FP64 at a middle size (H_w^2 is what eigensolvers apply)
        _case("matvec2 12^4 f64", "matvec", (12, 12, 12, 12), 4, 0, 0, "f64", 0.7, 0.2, op=2),
        # the operator at the benchmark's lattice and batch
        _case("matvec 16^3x32 mixed", "matvec", (16, 16, 16, 32), 16, 0, 0, "mixed", 0.6, 0.1),
        # the plain method on the smallest lattice (configuration 1): one source, no deflation
        _case("sign 4^4 f64", "sign", (4, 4, 4, 4), 1, 100, 0, "f64", 0.5, 0.3),
        # odd extents, an odd Krylov dimension and an odd batch
        _case("sign 3x5x7x9 f64", "sign", (3, 5, 7, 9), 3, 75, 8, "f64", 0.6, 0.2),
        # configuration 2: the deflated method in FP64
        _case("sign 8^4 f64", "sign", (8, 8, 8, 8), 4, 200, 30, "f64", 0.7, 0.2),
        # one source in the mixed form, as a solver's single application
        _case("sign 8^4 mixed one", "sign", (8, 8, 8, 8), 1, 200, 30, "mixed", 0.7, 0.2),
        # configuration 3: the batched mixed form
        _case("sign 12^4 mixed", "sign", (12, 12, 12, 12), 16, 250, 50, "mixed", 0.7, 0.2),
        # the benchmark's lattice; batch, Krylov dimension and basis small enough to be prepared often
        _case("sign 16^3x32 mixed", "sign", (16, 16, 16, 32), 8, 200, 16, "mixed", 0.6, 0.1),
        # D_ov with a long Krylov space (what an accurate sign takes on these fields), harmonic form
        _case("overlap 6^4 long f64", "overlap", (6, 6, 6, 6), 2, 340, 16, "f64", 0.6, 0.2, harmonic=True),
        # Schur deflation, mixed, a full batch
        _case("schur 8^4 mixed", "schur", (8, 8, 8, 8), 16, 80, 30, "mixed", 0.7, 0.2),
        # several gauge fields in one call, each source stopped by its own convergence
        _case("batched mixed", "batched", (4, 4, 4, 4), 4, 0, 20, "mixed", 0.6, 0.2, instances=6, cap=300, tol=1e-4),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["matvec", "sign", "sign", "sign", "overlap", "schur", "batched"])
    prec = rng.choice(["f64", "mixed"])
    eps, mu = round(rng.uniform(0.5, 0.7), 3), round(rng.uniform(0.05, 0.3), 3)
    nrhs = log_int(1, 16)
    if kind == "matvec":
        dims = [rng.randint(3, 16) for _ in range(4)]
        return _pure(_case("", kind, dims, nrhs, 0, 0, prec, eps, mu, op=rng.choice([0, 1, 2])))
    if kind == "batched":
        dims = [rng.randint(3, 5) for _ in range(4)]
        return _pure(_case("", kind, dims, rng.randint(1, 6), 0, rng.randint(4, 20), prec, eps, mu,
                           instances=rng.randint(2, 6), cap=rng.randint(100, 300), tol=10.0 ** rng.uniform(-5, -3)))
    top = 6 if prec == "f64" else 12
    dims = [rng.randint(3, top) for _ in range(4)]
    m = rng.choice([0, rng.randint(4, 40)]) if kind != "schur" else rng.randint(4, 40)
    n = 12 * dims[0] * dims[1] * dims[2] * dims[3]
    k = min(log_int(20, 150 if kind == "schur" else 360), (n - m) // 4)
    if prec == "mixed":  # an odd k has a Ritz value near 0 on these spectra, which single precision does not resolve
        k -= k % 2
    return _pure(_case("", kind, dims, nrhs, k, m, prec, eps, mu, harmonic=kind != "schur" and rng.random() < 0.25))


def _pure(c):
    return {q: v for q, v in c.items() if q != "name"}


# ------------------------------------------------------------------- inputs
def _dims(case):
    return (case["lx"], case["ly"], case["lz"], case["lt"])


def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _gauss(shape, gen):
    return torch.complex(torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64),
                         torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64))


def _links(dims, eps, seed):
    """exp(i eps X), X traceless Hermitian from complex Gaussians: complex128 [V][4][3][3]."""
    v = dims[0] * dims[1] * dims[2] * dims[3]
    a = _gauss((v * 4, 3, 3), _gen(seed, 1))
    x = 0.5 * (a + a.mH)
    x -= torch.eye(3, device=DEV) * (torch.diagonal(x, dim1=-2, dim2=-1).sum(-1) / 3)[:, None, None]
    return torch.linalg.matrix_exp(1j * eps * x).reshape(v, 4, 3, 3)


def _vectors(count, n, gen):
    x = _gauss((count, n), gen)
    return x / torch.linalg.vector_norm(x, dim=1, keepdim=True)


def _deflation(kind, m, n, seed):
    """R, L [m][N] and lambda: near-biorthonormal pairs; for Schur deflation R
    only, projected on chiralities in turn so that S^+ H_w S is well conditioned."""
    gen = _gen(seed, 3)
    r = _vectors(m, n, gen)
    if kind == "schur":
        chi = torch.ones(12, device=DEV, dtype=torch.float64)
        chi[6:] = -1.0
        side = torch.where(torch.arange(m, device=DEV) % 2 == 0, 1.0, -1.0)
        r = r * (0.5 * (1.0 + side[:, None] * chi.repeat(n // 12)[None, :]))
        return r / torch.linalg.vector_norm(r, dim=1, keepdim=True), None, None
    left = r + 0.3 * _vectors(m, n, gen)
    left = left / torch.linalg.vector_norm(left, dim=1, keepdim=True)
    u = torch.rand((3, m), generator=gen, device=DEV, dtype=torch.float64)
    lam = torch.complex((0.05 + 0.45 * u[0]) * torch.where(u[1] < 0.5, -1.0, 1.0).double(), 0.6 * u[2] - 0.3)
    return r, left, lam


def _inputs(case, seed):
    """(dims, links, deflation, x) of every gauge field of the case."""
    out = []
    for i in range(case["instances"]):
        d = tuple(q + 2 * (i % 3) for q in _dims(case)) if case["kind"] == "batched" else _dims(case)
        nrhs = 1 + (case["nrhs"] * (i + 2) * 5) % 16 if case["kind"] == "batched" else case["nrhs"]
        s = int(seed) * 64 + i
        n = 12 * d[0] * d[1] * d[2] * d[3]
        defl = _deflation(case["kind"], case["m"], n, s) if case["m"] else (None, None, None)
        out.append((d, _links(d, case["eps"], s), defl, _vectors(nrhs, n, _gen(s, 2))))
    return out


def prepare(case, seed):
    prec = ovs.F64 if case["prec"] == "f64" else ovs.MIXED
    gauges, xs, ys = [], [], []
    for d, links, (r, left, lam), x in _inputs(case, seed):
        g = ovs.create_gauge_from_links(d, links.cpu().numpy(), prec)
        ovs.set_mu(g, case["mu"], M_W)
        if case["m"] and case["kind"] == "schur":
            ovs.deflate_load_schur(g, r.cpu().numpy())
        elif case["m"]:
            ovs.deflate_load(g, r.cpu().numpy(), left.cpu().numpy(), lam.cpu().numpy())
        gauges.append(g)
        xs.append(x)
        ys.append(torch.empty_like(x))
    return {"case": case, "prec": prec, "g": gauges, "x": xs, "y": ys}


def run(state):
    c, g, x, y, prec = state["case"], state["g"], state["x"], state["y"], state["prec"]
    keep = (lambda t: t) if prec == ovs.F64 else (lambda t: t.to(torch.complex64))
    if c["kind"] == "matvec":
        ovs.matvec(g[0], c["op"], x[0], y[0], prec=prec)
        return keep(y[0])
    if c["kind"] == "batched":
        _, info = ovs.sign_apply_batched(g, x, y, c["cap"], prec=prec, check_every=10, tol=c["tol"], skip_ahead=True)
        return {"y": [keep(t) for t in y], "k_used": np.array([i["k_used"] for i in info]),
                "status": np.array([i["status"] for i in info])}
    call = ovs.overlap_apply if c["kind"] == "overlap" else ovs.sign_apply
    call(g[0], x[0], y[0], c["k"], prec=prec, want_info=False, harmonic=c["harmonic"])
    return keep(y[0])


# ------------------------------------------------------------ work of a pass
def work(case):
    """Inputs read once, outputs written once; k operator applications, one
    orthogonalisation of the basis, one recombination, and the sign of the k x k
    matrix as the first column of a k x k function (one solve's worth of k^3)."""
    size = 16 if case["prec"] == "f64" else 8
    nbytes = flops = 0
    for i in range(case["instances"]):
        d = tuple(q + 2 * (i % 3) for q in _dims(case)) if case["kind"] == "batched" else _dims(case)
        nrhs = 1 + (case["nrhs"] * (i + 2) * 5) % 16 if case["kind"] == "batched" else case["nrhs"]
        v = d[0] * d[1] * d[2] * d[3]
        n, m, k = 12 * v, case["m"], case["cap"] // 2 if case["kind"] == "batched" else case["k"]
        out = 16 if case["prec"] == "f64" else 8
        nbytes += n * nrhs * (16 + out) + 36 * v * size + n * m * size * (1 if case["kind"] == "schur" else 2)
        if case["kind"] == "matvec":
            flops += nrhs * v * 1392 * (2 if case["op"] == 2 else 1)
            continue
        per = k * v * 1392 + 8 * n * k * k + 8 * n * k + 8 * k ** 3 + 24 * n * m
        if case["kind"] == "schur":
            per += 16 * n * m * k + 16 * m * k * k
        flops += nrhs * per
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------- 64-bit values of a pass
_SIGMA = [np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]], complex), np.array([[1, 0], [0, -1]], complex)]


def _gammas():
    """Each gamma matrix has one entry per row: (its columns, its values)."""
    out = []
    for a in _SIGMA + [None]:
        z = np.zeros((2, 2))
        g = np.block([[z, np.eye(2)], [np.eye(2), z]]) if a is None else np.block([[z, -1j * a], [1j * a, z]])
        col = np.abs(g).argmax(axis=1)
        out.append((torch.from_numpy(col).to(DEV), torch.from_numpy(g[np.arange(4), col].astype(complex)).to(DEV)))
    return out


class _Wilson:
    """D_w(mu) and H_w(mu) of canonical complex128 vectors [B][N], written out term by term."""

    def __init__(self, dims, links, mu):
        self.shape = (dims[3], dims[2], dims[1], dims[0])
        self.links = links.reshape(*self.shape, 4, 3, 3)
        self.mu, self.kappa, self.gam = mu, 1.0 / (8.0 + 2.0 * M_W), _gammas()

    def _dw1(self, x):
        psi = x.reshape(*self.shape, 4, 3)
        acc = torch.zeros_like(psi)
        for nu in range(4):
            ax, u, (col, val) = 3 - nu, self.links[..., nu, :, :], self.gam[nu]
            up = torch.roll(psi, -1, ax)
            dn = torch.roll((u.conj().mT[..., None, :, :] * psi[..., None, :]).sum(-1), 1, ax)
            if nu == 3:
                up[-1] *= -1
                dn[0] *= -1
                up, dn = up * math.exp(self.mu), dn * math.exp(-self.mu)
            up = (u[..., None, :, :] * up[..., None, :]).sum(-1)
            acc += up + dn - (up - dn)[..., col, :] * val[:, None]
        return (psi - self.kappa * acc).reshape(-1)

    def dw(self, x):
        return torch.stack([self._dw1(q) for q in x])

    def hw(self, x):
        return _gamma5(self.dw(x))


def _gamma5(x):
    y = x.clone().reshape(x.shape[0], -1, 12)
    y[..., 6:] *= -1
    return y.reshape(x.shape)


def _sgn(a):
    """Sign of a small matrix (on the host: its LU factorisations are quicker there)."""
    s = a.cpu().numpy()
    for _ in range(60):
        t = 0.5 * (s + np.linalg.inv(s))
        d = np.linalg.norm(t - s) / np.linalg.norm(t)
        s = t
        if d < 1e-13:
            break
    return torch.from_numpy(s).to(DEV)


def _arnoldi(op, x, k, against=None):
    """Arnoldi with twice-repeated Gram-Schmidt, all vectors of x together:
    V [B][k][N], Hbar [B][k+1][k], the norms, X = S^+ A V_k for `against` = S."""
    b, n = x.shape
    beta = torch.linalg.vector_norm(x, dim=1)
    v = torch.zeros((b, k + 1, n), dtype=torch.complex128, device=DEV)
    h = torch.zeros((b, k + 1, k), dtype=torch.complex128, device=DEV)
    xs = torch.zeros((b, 0 if against is None else against.shape[0], k), dtype=torch.complex128, device=DEV)
    v[:, 0] = x / beta[:, None]
    for j in range(k):
        w = op(v[:, j])
        for _ in range(2):
            if against is not None:
                c = w @ against.mH
                w = w - c @ against
                xs[:, :, j] += c
        for _ in range(2):
            for i in range(b):  # matrix-vector products: a product with one row is slow in 64 bits
                q = v[i, : j + 1]
                c = torch.mv(q, w[i].conj()).conj()
                w[i] -= torch.mv(q.T, c)
                h[i, : j + 1, j] += c
        nrm = torch.linalg.vector_norm(w, dim=1)
        h[:, j + 1, j] = nrm
        v[:, j + 1] = w / nrm[:, None]
    return v[:, :k], h, beta, xs


def _combine(c, v):
    return torch.stack([torch.mv(v[i].T, c[i]) for i in range(v.shape[0])])


def _lr(x, defl):
    """(x - R c, R sgn(Re lambda) c) with c = (L^+ R)^-1 L^+ x."""
    r, left, lam = defl
    if r is None:
        return x, torch.zeros_like(x)
    c = torch.linalg.solve(left.conj() @ r.T, left.conj() @ x.T).T
    return x - c @ r, (c * torch.sign(lam.real)) @ r


def _sign(op, x, k, defl, harmonic):
    rest, y = _lr(x, defl)
    v, h, beta, _ = _arnoldi(op, rest, k)
    hk = h[:, :k].clone()
    if harmonic:
        e = torch.zeros((x.shape[0], k, 1), dtype=torch.complex128, device=DEV)
        e[:, -1] = 1.0
        hk[:, :, -1:] += (h[:, k, k - 1].abs() ** 2)[:, None, None] * torch.linalg.solve(hk.mH, e)
    c = torch.stack([beta[i] * _sgn(hk[i])[:, 0] for i in range(x.shape[0])])
    return y + _combine(c, v)


def _sign_schur(op, x, k, r):
    s = torch.linalg.qr(r.T)[0].T.contiguous()  # rows: Schur vectors
    m = s.shape[0]
    t = torch.triu(s.conj() @ op(s).T)
    c = x @ s.mH
    rest = x - c @ s
    c2 = rest @ s.mH
    rest, c = rest - c2 @ s, c + c2
    v, h, beta, xs = _arnoldi(op, rest, k, s)
    big = torch.zeros((x.shape[0], m + k, m + k), dtype=torch.complex128, device=DEV)
    big[:, :m, :m], big[:, :m, m:], big[:, m:, m:] = t, xs, h[:, :k]
    vec = torch.zeros((x.shape[0], m + k, 1), dtype=torch.complex128, device=DEV)
    vec[:, :m, 0], vec[:, m, 0] = c, beta
    f = torch.stack([(_sgn(big[i]) @ vec[i])[:, 0] for i in range(x.shape[0])])
    return f[:, :m] @ s + _combine(f[:, m:], v)


def _stop(cs, every, cap, tol):
    """The Krylov dimension at which a source stops: convergence checks on the
    skip-ahead schedule. cs(j): the coefficients at j."""
    old, jl, hist, j = None, 0, [], every
    last = every * ((cap - 1) // every)
    while 0 < j < cap:
        c = cs(j)
        diff = c.clone()
        if old is not None:
            diff[: old.shape[0]] -= old
        e = float(torch.linalg.vector_norm(diff) / torch.linalg.vector_norm(c))
        if e < tol:
            return j
        nxt = j + every
        if jl > 0 and j - jl == every:
            hist.append((j, e))
            if len(hist) > 1 and hist[-1][1] < hist[-2][1]:
                (j0, e0), (j1, e1) = hist[-2:]
                t = j1 + math.log(tol / e1) / (math.log(e1 / e0) / (j1 - j0))
                nxt = max(nxt, last - every if t >= last else every * math.floor(t / every) - every)
        old, jl, j = c, j, nxt
    return cap


def _sign_stopped(op, x, defl, cap, tol):
    rest, y = _lr(x, defl)
    v, h, beta, _ = _arnoldi(op, rest, cap)
    out = []
    for b in range(x.shape[0]):
        kept = {}

        def coeff(j):
            if j not in kept:
                kept[j] = beta[b] * _sgn(h[b, :j, :j])[:, 0]
            return kept[j]

        k = _stop(coeff, 10, cap, tol)
        out.append(y[b] + torch.mv(v[b, :k].T, coeff(k)))
    return torch.stack(out)


def exact(case, seed):
    kind, got = case["kind"], []
    for d, links, defl, x in _inputs(case, seed):
        w = _Wilson(d, links, case["mu"])
        if kind == "matvec":
            got.append(w.dw(x) if case["op"] == 0 else w.hw(x) if case["op"] == 1 else w.hw(w.hw(x)))
        elif kind == "batched":
            got.append(_sign_stopped(w.hw, x, defl, case["cap"], case["tol"]))
        elif kind == "schur":
            got.append(_sign_schur(w.hw, x, case["k"], defl[0]))
        else:  # one source at a time: its basis is large in 64 bits
            y = torch.cat([_sign(w.hw, q[None], case["k"], defl, case["harmonic"]) for q in x])
            got.append(x + _gamma5(y) if kind == "overlap" else y)
    return {"y": got, "k_used": None, "status": None} if kind == "batched" else got[0]
