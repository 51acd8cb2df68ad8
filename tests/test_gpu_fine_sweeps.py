"""The sweeps and the stencil of small problems (csrc/fine_sweeps.cu,
k_wilson_split) at the edges of their splits: fields that end inside a tile of
128 units or a group of 32 sites, fewer vectors than a set of four, one and many
right-hand sides on either side of each rule. Against the oracle at equal k,
1e-12 (FP64) and 1e-6 (mixed) relative, the bounds of the two forms everywhere
in these tests; the spread stencil gives the bits of the plain one.
"""

import numpy as np
import pytest
import torch

import synth
from oracle import arnoldi, lattice

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("dims,nrhs,k", [((2, 2, 2, 2), 1, 40), ((3, 3, 3, 3), 4, 30), ((2, 3, 5, 7), 2, 64),
                                         ((4, 4, 4, 4), 1, 2), ((4, 4, 4, 4), 7, 66), ((5, 3, 7, 3), 9, 50),
                                         ((6, 6, 6, 6), 16, 50), ((8, 8, 8, 8), 16, 36)])
def test_sign_matches_oracle(gpu, dims, nrhs, k):
    links = synth.gauge_links(dims, 9, 0.6)
    h = lattice.hw_operator(links, dims, 0.2, -1.5)
    g = gpu.create_gauge_from_links(dims, links, gpu.MIXED)
    gpu.set_mu(g, 0.2, -1.5)
    x = synth.gaussian_vectors(h.shape[0], nrhs, 11)
    xd = torch.from_numpy(x).cuda()
    yd = torch.empty_like(xd)
    refs = {r: arnoldi.arnoldi_sign(lambda q: h @ q, x[r], k)[0] for r in {0, nrhs // 2, nrhs - 1}}
    for prec, tol in ((gpu.F64, 1e-12), (gpu.MIXED, 1e-6)):
        st, info = gpu.sign_apply(g, xd, yd, k, prec=prec)
        assert st == 0 and all(i["k_used"] == k for i in info)
        y = yd.cpu().numpy()
        for r, ref in refs.items():
            assert rel(y[r], ref) < tol, (prec, r)
    g.destroy()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 3, 5, 3), (4, 4, 4, 4), (2, 6, 3, 5), (8, 8, 8, 8), (9, 8, 8, 8)])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("op", [0, 1, 2])
def test_spread_stencil_is_bit_identical(gpu, dims, prec, op):
    """One right-hand side (spread over the hops) and the same among 300
    (one thread per site)."""
    links = synth.gauge_links(dims, 3, 0.6)
    g = gpu.create_gauge_from_links(dims, links, gpu.MIXED)
    gpu.set_mu(g, 0.2, -1.5)
    x = torch.from_numpy(synth.gaussian_vectors(12 * int(np.prod(dims)), 300, 5)).cuda()
    many, one = torch.empty_like(x), torch.empty_like(x[:1])
    gpu.matvec(g, op, x, many, prec=prec)
    for r in (0, 299):
        gpu.matvec(g, op, x[r:r + 1].contiguous(), one, prec=prec)
        assert torch.equal(one[0], many[r])
    g.destroy()


@pytest.mark.parametrize("dims,nrhs", [((8, 8, 8, 9), 2), ((9, 9, 9, 9), 2), ((5, 7, 9, 11), 6), ((8, 8, 8, 8), 5)])
@pytest.mark.parametrize("op", [0, 1, 2])
def test_two_threads_per_site_is_bit_identical(gpu, dims, nrhs, op):
    """complex128 by two threads per site (288, 412, 654, 640 groups of 32 sites)
    against two right-hand sides per thread (k_wilson)."""
    links = synth.gauge_links(dims, 3, 0.6)
    g = gpu.create_gauge_from_links(dims, links, gpu.F64)
    gpu.set_mu(g, 0.2, -1.5)
    x = torch.from_numpy(synth.gaussian_vectors(12 * int(np.prod(dims)), nrhs, 5)).cuda()
    ref, y = torch.empty_like(x), torch.empty_like(x)
    gpu.set_stencil_shape(g, gpu.F64, nrhs, (2, 32, 1))
    gpu.matvec(g, op, x, ref, prec=gpu.F64)
    for sites, rb in ((32, 1), (32, 8), (64, 4), (128, 2)):
        gpu.set_stencil_shape(g, gpu.F64, nrhs, (1, sites, rb))
        y.zero_()
        gpu.matvec(g, op, x, y, prec=gpu.F64)
        assert torch.equal(y, ref), (sites, rb)
    g.destroy()
