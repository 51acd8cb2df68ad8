"""The complex128 form's sweeps on the integer multipliers
(csrc/fix_sweeps.cu): fields that end inside a tile (128 units) and a scale
group (1024), both splits of each kernel, sums over more vectors than the
accumulators take before a carry (8) and a flush (32), sources of very different
magnitude (the scales) and with a single non-zero element.

Against the oracle at equal k, 1e-12 relative (the FP64 form's bound everywhere
in these tests); the basis orthonormal and the Arnoldi relation to 1e-13: an
element is rounded by 2^-59 of the largest, the recurrences by FP64.
"""

import numpy as np
import pytest
import torch

import synth
from oracle import arnoldi, lattice

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("dims,nrhs,k", [((2, 2, 2, 2), 1, 33), ((2, 3, 5, 3), 3, 7), ((4, 4, 4, 4), 1, 260),
                                         ((4, 4, 4, 4), 40, 40), ((6, 6, 6, 6), 3, 100), ((6, 6, 6, 6), 6, 130),
                                         ((5, 7, 6, 9), 9, 65)])
@pytest.mark.parametrize("kind", ["gauss", "point", "scaled"])
def test_sign_and_basis(gpu, dims, nrhs, k, kind):
    links = synth.gauge_links(dims, 13, 0.6)
    h = lattice.hw_operator(links, dims, 0.2, -1.5)
    n = h.shape[0]
    x = synth.gaussian_vectors(n, nrhs, 17)
    if kind == "point":
        x[:] = 0.0
        x[np.arange(nrhs), (np.arange(nrhs) * 97 + 5) % n] = 1.0 - 0.5j
    if kind == "scaled":
        x *= 10.0 ** np.linspace(-60, 60, nrhs)[:, None] if nrhs > 1 else 1e60
    g = gpu.create_gauge_from_links(dims, links, gpu.F64)
    gpu.set_mu(g, 0.2, -1.5)
    xd = torch.from_numpy(x).cuda()
    yd = torch.empty_like(xd)
    st, info = gpu.sign_apply(g, xd, yd, k, prec=gpu.F64)
    assert st == 0 and all(i["k_used"] == k for i in info)
    y = yd.cpu().numpy()
    for r in sorted({0, nrhs - 1}):
        ref = arnoldi.arnoldi_sign(lambda q: h @ q, x[r], k)[0]
        assert rel(y[r], ref) < 1e-12, r
        V, Hb = gpu.get_krylov(g, r)
        Vk = V.T
        assert np.abs(Vk.conj().T @ Vk - np.eye(k)).max() < 1e-13
        res = h @ Vk[:, :k - 1] - Vk @ Hb[:k, :k - 1]
        assert np.abs(res).max() < 1e-13 * np.abs(Hb).max()
    g.destroy()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_sources_stay_apart(gpu, bad):
    """One non-finite right-hand side among ordinary ones."""
    dims = (4, 4, 4, 4)
    links = synth.gauge_links(dims, 13, 0.6)
    g = gpu.create_gauge_from_links(dims, links, gpu.F64)
    gpu.set_mu(g, 0.2, -1.5)
    x = torch.from_numpy(synth.gaussian_vectors(12 * 256, 3, 2)).cuda()
    good, y = torch.empty_like(x), torch.empty_like(x)
    gpu.sign_apply(g, x, good, 40, prec=gpu.F64)
    x[1, 77] = bad
    try:
        gpu.sign_apply(g, x, y, 40, prec=gpu.F64)
    except gpu.OvsError:
        pass
    assert torch.equal(y[0], good[0]) and torch.equal(y[2], good[2])
    g.destroy()
