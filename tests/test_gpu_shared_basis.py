"""The shared-basis sweeps of the mixed form (k_shared_dots, k_shared_combine in
csrc/blas.cu) where their splits change: one to many groups of threads per staged
tile, sums that do not fill the threads, one and two units per thread. Against
the same application in FP64, 1e-6 relative (the mixed form's bound everywhere in
these tests)."""

import numpy as np
import pytest
import torch

import synth
from oracle import lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,m,nrhs", [((4, 4, 4, 4), 5, 1), ((3, 4, 5, 4), 30, 16), ((4, 4, 4, 4), 33, 17),
                                         ((4, 4, 4, 4), 100, 16), ((4, 4, 4, 4), 64, 32), ((8, 8, 8, 8), 6, 64),
                                         ((8, 8, 8, 8), 30, 16)])
def test_mixed_projection_matches_fp64(gpu, dims, m, nrhs):
    links = synth.gauge_links(dims, 4, 0.6)
    n = 12 * int(np.prod(dims))
    g = gpu.create_gauge_from_links(dims, links, gpu.MIXED)
    gpu.set_mu(g, 0.2, -1.5)
    r = synth.gaussian_vectors(n, m, 31).T.copy()
    chi = lattice.gamma5_diag(n // 12)[:, None] * np.where(np.arange(m) % 2 == 0, 1.0, -1.0)[None, :]
    gpu.deflate_load_schur(g, (0.5 * (r + chi * r)).T.copy())
    xd = torch.from_numpy(synth.gaussian_vectors(n, nrhs, 32)).cuda()
    y = {}
    for prec in (gpu.F64, gpu.MIXED):
        y[prec] = torch.empty_like(xd)
        gpu.sign_apply(g, xd, y[prec], 20, prec=prec)
    err = torch.linalg.norm(y[gpu.MIXED] - y[gpu.F64], dim=1) / torch.linalg.norm(y[gpu.F64], dim=1)
    assert err.max().item() < 1e-6
    g.destroy()
