"""sgn(H_k) e_1 at orders above 320 with spectra up to the imaginary axis (mu = 1.5 to
2.5 on 4^4, 87 to 89 degrees off the real axis): the third and the fourth rule of
csrc/signquad.cu, through ovs_sign_apply in FP64, against the oracle at equal k.

Tolerance: 1e-12 (the FP64 form's everywhere in these tests) times the amplification of
rounding by the sign, ||H|| / min |Re lambda| of H_k from the oracle's Hessenberg
matrix over the 10 that it is below mu = 1."""

import numpy as np
import pytest
import torch

import synth
from oracle import arnoldi, lattice, newton

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mu,k", [(1.5, 321), (1.5, 400), (2.0, 400), (2.5, 400)])
def test_wide_and_long(gpu, mu, k):
    dims = (4, 4, 4, 4)
    links = synth.gauge_links(dims, 1, 0.6)
    h = lattice.hw_operator(links, dims, mu, -1.5)
    x = synth.gaussian_vectors(h.shape[0], 2, 3)
    g = gpu.create_gauge_from_links(dims, links, gpu.F64)
    gpu.set_mu(g, mu, -1.5)
    yd = torch.empty((2, h.shape[0]), dtype=torch.complex128, device="cuda")
    st, info = gpu.sign_apply(g, torch.from_numpy(x).cuda(), yd, k, prec=gpu.F64)
    g.destroy()
    assert st == 0
    for r in range(2):
        V, Hb, beta, _ = arnoldi.arnoldi(lambda q: h @ q, x[r], k)
        Hk = Hb[:k, :k]
        ref = V[:, :k] @ (beta * newton.roberts_sign(Hk)[0][:, 0])
        tol = 1e-12 * max(1.0, np.linalg.norm(Hk, 2) / np.abs(np.linalg.eigvals(Hk).real).min() / 10.0)
        err = np.linalg.norm(yd[r].cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err < tol, (r, err, tol, info[r]["newton_iters"])
