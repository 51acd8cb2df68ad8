"""Long Krylov spaces on small complex64 fields (csrc/fine_sweeps.cu), whose update
needs more than 48 KB of shared memory from 677 steps on, up to the largest k.

Against the FP64 form at equal k, 1e-6 relative (the mixed form's bound everywhere in
these tests)."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nrhs,k", [((8, 8, 8, 8), 1, 790), ((8, 8, 8, 8), 3, 682), ((4, 4, 4, 4), 16, 678),
                                         ((4, 4, 4, 4), 50, 700)])
def test_long_spaces(gpu, dims, nrhs, k):
    g = gpu.create_gauge(dims, 1, 0.6, gpu.MIXED)
    gpu.set_mu(g, 0.2, -1.5)
    x = torch.from_numpy(synth.gaussian_vectors(12 * int(np.prod(dims)), nrhs, 9)).cuda()
    ys = []
    for prec in (gpu.F64, gpu.MIXED):
        y = torch.empty_like(x)
        st, info = gpu.sign_apply(g, x, y, k, prec=prec)
        assert st == 0 and all(i["k_used"] == k for i in info)
        ys.append(y)
    g.destroy()
    err = torch.linalg.vector_norm(ys[1] - ys[0], dim=1) / torch.linalg.vector_norm(ys[0], dim=1)
    assert float(err.max()) < 1e-6
