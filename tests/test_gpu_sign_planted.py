"""sgn(H_k) e_1 where H_k has an eigenvalue close to 0 or to the imaginary axis, with
any weight in the source, through ovs_sign_apply in FP64.

Free field on 2x2x2x3 with constant temporal links diag(e^(i theta), e^(-i theta), 1):
a plane wave x of momentum p and one colour has H_w^2 x = lambda^2 x with
  lambda^2 = (2 kappa)^2 (a^2 + sum_j sin^2 p_j + sin^2 q),
  a = m_w + sum_j (1 - cos p_j) + 1 - cos q,  q = p_t + theta - i mu,
so sgn(H_w) x = H_w x / sqrt(lambda^2) exactly. p = (0, 0, 0, pi) has lambda =
kappa (2 m_w + 4) at mu = 0 and lambda^2 = (2 kappa)^2 (2 - 2 cos theta cosh mu - 2i
sin theta sinh mu) at m_w = -2.

Tolerance: 1e-12 (the FP64 form's everywhere in these tests) plus rounding of H_w in
any of the N terms of a sum, amplified by the sign's condition: N 2^-52 ||H_w|| / min
|Re lambda|, with the triangle inequality's bound of ||H_w||.
"""

import numpy as np
import pytest
import torch

from oracle import lattice

pytestmark = pytest.mark.gpu

DIMS, K = (2, 2, 2, 3), 12
N = 12 * 24
NEAR, HALF, TOP = (0, 0, 0, 1), (1, 0, 0, 0), (1, 1, 0, 1)


def links_of(theta):
    links = np.zeros((N // 12, 4, 3, 3), dtype=complex)
    links[:] = np.eye(3)
    links[:, 3] = np.diag([np.exp(1j * theta), np.exp(-1j * theta), 1.0])
    return links


def plane_wave(mode):
    p = [np.pi * mode[0], np.pi * mode[1], np.pi * mode[2], np.pi * (2 * mode[3] + 1) / DIMS[3]]
    phase = np.exp(1j * sum(a * c for a, c in zip(p, lattice.site_coords(DIMS))))
    x = np.zeros((N // 12, 4, 3), dtype=complex)
    x[:, :, 0] = phase[:, None] * np.array([1.0, 0.3, -0.7j, 0.5 + 0.2j])
    return x.reshape(-1) / np.linalg.norm(x), p


def problem(mu, m_w, theta, weights):
    """(links, x, sgn(H_w) x, tolerance, H_w, the waves and their lambda) for x = sum of
    weight times wave."""
    h = lattice.hw_operator(links_of(theta), DIMS, mu, m_w)
    kappa = lattice.kappa_of(m_w)
    x, y, lams, waves = 0.0, 0.0, [], []
    for mode, w in weights:
        v, p = plane_wave(mode)
        q = p[3] + theta - 1j * mu
        a = m_w + sum(1.0 - np.cos(t) for t in p[:3]) + 1.0 - np.cos(q)
        lam = 2.0 * kappa * np.sqrt(a * a + sum(np.sin(t) ** 2 for t in p[:3]) + np.sin(q) ** 2 + 0j)
        assert np.linalg.norm(h @ (h @ v) - lam**2 * v) < 1e-13
        x, y = x + w * v, y + w * (h @ v) / lam
        lams.append(lam)
        waves.append(v)
    hnorm = 2.0 * kappa * (abs(m_w + 4.0) + 3.0 + np.exp(abs(mu)))
    tol = 1e-12 + N * 2.0**-52 * hnorm / min(abs(v.real) for v in lams)
    return links_of(theta), x, y, tol, h, list(zip(waves, lams))


def apply(gpu, links, mu, m_w, x, schur=None):
    g = gpu.create_gauge_from_links(DIMS, links, gpu.F64)
    gpu.set_mu(g, mu, m_w)
    if schur is not None:
        gpu.deflate_load_schur(g, schur)
    xd = torch.from_numpy(x[None]).cuda()
    yd = torch.empty_like(xd)
    st, _ = gpu.sign_apply(g, xd, yd, K, prec=gpu.F64)
    g.destroy()
    return st, yd.cpu().numpy()[0]


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("schur", [False, True])
@pytest.mark.parametrize("p,w", [(1, 1.0), (3, 1.0), (5, 1.0), (7, 1.0), (9, 1.0), (10, 1.0), (3, 1e-6), (5, 1e-4),
                                 (7, 1e-2)])
def test_next_to_zero(gpu, p, w, schur):
    """|lambda| = 10^-p / 2 at weight w; with Schur deflation of another wave's two
    eigenvectors lambda x +- H_w x."""
    m_w = -2.0 + 10.0**-p
    links, x, y, tol, h, waves = problem(0.0, m_w, 0.0, [(NEAR, w), (HALF, 1.0), (TOP, 1.0)])
    v, lam = waves[1]
    s = np.stack([lam * v + h @ v, lam * v - h @ v]) if schur else None
    st, got = apply(gpu, links, 0.0, m_w, x, s)
    assert st == 0 and rel(got, y) < tol


@pytest.mark.parametrize("theta,w", [(0.3, 1.0), (0.1, 1.0), (1e-2, 1.0), (1e-3, 1.0), (0.1, 1e-6), (1e-2, 1e-4),
                                     (1e-2, 1e-6), (1e-3, 1e-6)])
def test_next_to_the_imaginary_axis(gpu, theta, w):
    """lambda about theta radians off the imaginary axis, at weight w."""
    links, x, y, tol, _, _ = problem(1.0, -2.0, theta, [(NEAR, w), (HALF, 1.0), (TOP, 1.0)])
    st, got = apply(gpu, links, 1.0, -2.0, x)
    assert st == 0 and rel(got, y) < tol


@pytest.mark.parametrize("w", [1.0, 1e-3])
def test_singular_is_not_ok(gpu, w):
    """H_k singular to rounding: sgn(H_k) does not exist, and no call says OK."""
    v = [plane_wave(m)[0] for m in (NEAR, HALF, TOP)]
    try:
        st, _ = apply(gpu, links_of(0.0), 0.0, -2.0, w * v[0] + v[1] + v[2])
    except gpu.OvsError as e:
        st = e.status
    assert st in (1, -6)  # OVS_NOT_CONVERGED, OVS_ESIGN
