"""Two Arnoldi steps per pass over the complex64 basis (csrc/pair_sweeps.cu):
taken for bases of 272 MB and more (8^4, 16 right-hand sides, k >= 44).

Against the FP64 oracle at equal k, 1e-6 relative (the mixed form's bound
everywhere in these tests), for even and odd k; the basis orthonormal and the
Arnoldi relation to 1e-5 (the bounds of the single-step basis); convergence
checks at the oracle's steps; and right-hand sides that leave the blocks early
(an invariant Krylov space of a few vectors) beside ordinary ones.
"""

import numpy as np
import pytest
import torch

import synth
from oracle import arnoldi, freefield, lattice

pytestmark = pytest.mark.gpu

MW = -1.5


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.fixture(scope="module")
def problem(gpu):
    dims, mu = (8, 8, 8, 8), 0.2
    links = synth.gauge_links(dims, 3, 0.7)
    h = lattice.hw_operator(links, dims, mu, MW)
    g = gpu.create_gauge_from_links(dims, links, gpu.MIXED)
    gpu.set_mu(g, mu, MW)
    x = synth.gaussian_vectors(h.shape[0], 17, 21)
    yield g, h, x
    g.destroy()


@pytest.mark.parametrize("nrhs,k", [(16, 44), (16, 45), (17, 60), (11, 77)])
def test_matches_oracle(gpu, problem, nrhs, k):
    g, h, x = problem
    xd = torch.from_numpy(x[:nrhs]).cuda()
    yd = torch.empty_like(xd)
    st, info = gpu.sign_apply(g, xd, yd, k, prec=gpu.MIXED)
    assert st == 0 and all(i["k_used"] == k for i in info)
    y = yd.cpu().numpy()
    for r in (0, nrhs - 1):
        ref, _ = arnoldi.arnoldi_sign(lambda q: h @ q, x[r], k)
        assert rel(y[r], ref) < 1e-6, r
    V, Hb = gpu.get_krylov(g, nrhs - 1)
    Vk = V.T
    assert np.abs(Vk.conj().T @ Vk - np.eye(k)).max() < 1e-5
    res = h @ Vk - Vk @ Hb[:k, :k]
    hn = np.abs(Hb).max()
    assert np.abs(res[:, :k - 1]).max() < 1e-5 * hn
    assert abs(np.linalg.norm(res[:, k - 1]) - abs(Hb[k, k - 1])) < 1e-5 * hn


@pytest.mark.parametrize("skip", [False, True])
def test_checks_stop_at_the_oracles_step(gpu, problem, skip):
    g, h, x = problem
    xd = torch.from_numpy(x[:16]).cuda()
    yd = torch.empty_like(xd)
    st, info = gpu.sign_apply(g, xd, yd, 120, prec=gpu.MIXED, check_every=10, tol=2e-2, skip_ahead=skip)
    y = yd.cpu().numpy()
    for r in (0, 9):
        ref, oinfo = arnoldi.arnoldi_sign_adaptive(lambda q: h @ q, x[r], 120, 10, 2e-2, skip_ahead=skip)
        assert info[r]["k_used"] == oinfo["k_used"] < 120
        assert abs(info[r]["est_err"] - oinfo["est"]) <= 1e-4 * oinfo["est"]
        assert rel(y[r], ref) < 1e-6


def test_invariant_spaces_leave_the_blocks(gpu):
    """Plane waves on the free field (Krylov spaces of a few vectors, exact
    there) beside Gaussian sources, against the closed form; the Gaussian
    sources at k = 60 against the oracle."""
    dims, mu, k = (8, 8, 8, 8), 0.3, 60
    links = synth.unit_links(dims)
    h = lattice.hw_operator(links, dims, mu, MW)
    g = gpu.create_gauge_from_links(dims, links, gpu.MIXED)
    gpu.set_mu(g, mu, MW)
    n = h.shape[0]
    x = synth.gaussian_vectors(n, 16, 5)
    modes = {1: [(1, 0, 0, 0)], 6: [(1, 0, 0, 0), (0, 2, 1, 3)], 15: [(1, 2, 3, 0)]}
    for r, m in modes.items():
        x[r] = synth.plane_wave_vectors(dims, m, 7 + r)[0]
    x[9] = 0.0
    yd = torch.empty((16, n), dtype=torch.complex128, device="cuda")
    gpu.sign_apply(g, torch.from_numpy(x).cuda(), yd, k, prec=gpu.MIXED)
    y = yd.cpu().numpy()
    assert not y[9].any()
    for r in modes:
        assert rel(y[r], freefield.apply_free(x[r], dims, mu, MW, "sgnH")) < 1e-6, r
    for r in (0, 7):
        assert rel(y[r], arnoldi.arnoldi_sign(lambda q: h @ q, x[r], k)[0]) < 1e-6, r
    g.destroy()
