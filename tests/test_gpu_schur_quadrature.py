"""Schur coefficients by quadrature on [T X; 0 H_k] (csrc/signquad.cu) at the
edges of its compiled sizes, against Roberts' iteration on that matrix formed
from the oracle's Schur form and twice-repeated Gram-Schmidt: 1e-11 (FP64) and
1e-6 (mixed), the bounds of the Schur form everywhere in these tests. (The
oracle's own coefficients come from App. A's recurrences, which are 1.3e-11 off
this at m = 33 and 4.5e-10 at m = 65.) The vectors are chirally projected
Gaussians, so that sgn(T) is well conditioned."""

import numpy as np
import pytest
import torch

import synth
from oracle import lattice, newton, schur

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def composite(h, x, s, t, k):
    """S f_1 + V_k f_2 with f = sgn([T X; 0 H_k]) [c; beta e_1]."""
    m = s.shape[1]
    c = s.conj().T @ x
    rest = x - s @ c
    again = s.conj().T @ rest
    rest, c = rest - s @ again, c + again
    beta = np.linalg.norm(rest)
    v = np.zeros((x.shape[0], k + 1), complex)
    big = np.zeros((m + k + 1, m + k), complex)
    big[:m, :m] = t
    v[:, 0] = rest / beta
    for j in range(k):
        w = h @ v[:, j]
        for _ in range(2):
            for basis, rows in ((s, slice(0, m)), (v[:, :j + 1], slice(m, m + j + 1))):
                a = basis.conj().T @ w
                w = w - basis @ a
                big[rows, m + j] += a
        big[m + j + 1, m + j] = np.linalg.norm(w)
        v[:, j + 1] = w / big[m + j + 1, m + j]
    vec = np.zeros(m + k, complex)
    vec[:m], vec[m] = c, beta
    f = newton.roberts_sign(big[:-1])[0] @ vec
    return s @ f[:m] + v[:, :k] @ f[m:]


@pytest.mark.parametrize("m", [1, 31, 32, 33, 64, 65, 128, 129, 256])
def test_matches_oracle(gpu, m):
    dims, mu, k, nrhs = (4, 4, 4, 4), 0.2, 24, 3
    links = synth.gauge_links(dims, 4, 0.6)
    h = lattice.hw_operator(links, dims, mu, -1.5)
    n = h.shape[0]
    g = gpu.create_gauge_from_links(dims, links, gpu.MIXED)
    gpu.set_mu(g, mu, -1.5)
    r = synth.gaussian_vectors(n, m, 31).T.copy()
    chi = lattice.gamma5_diag(n // 12)[:, None] * np.where(np.arange(m) % 2 == 0, 1.0, -1.0)[None, :]
    r = 0.5 * (r + chi * r)
    gpu.deflate_load_schur(g, r.T.copy())
    s, t = schur.schur_from_eigvecs(lambda q: h @ q, r)
    x = synth.gaussian_vectors(n, nrhs, 32)
    x[2] = s[:, 0]  # in the span of S: an empty Krylov space up to rounding
    refs = [composite(h, x[q], s, t, k) for q in range(2)]
    xd = torch.from_numpy(x).cuda()
    yd = torch.empty_like(xd)
    for prec, tol in ((gpu.F64, 1e-11), (gpu.MIXED, 1e-6)):
        gpu.sign_apply(g, xd, yd, k, prec=prec)
        y = yd.cpu().numpy()
        for q in range(2):
            assert rel(y[q], refs[q]) < tol, (m, prec, q)
    g.destroy()
