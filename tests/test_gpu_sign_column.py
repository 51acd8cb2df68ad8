"""The first column of sgn(H_k) by quadrature (csrc/signquad.cu) against the
oracle's Roberts iteration, through ovs_sign_apply in FP64.

Krylov dimensions at the edges of the kernel's 32-row slots and of its compiled
sizes, the largest one the interface takes, and the four ways a right-hand side
is served: the first rule, the second rule (spectrum up to 36 degrees off the
real axis, mu = 1), the third (73 to 78 degrees, mu = 2) and Roberts' iteration
itself (89.8 degrees at k = 41, mu = 3 on 2x2x2x4).

Tolerance: 1e-12 relative (the FP64 form against the oracle at equal k
everywhere in these tests); 1e-11 at mu >= 1, where the sign amplifies
rounding of H_k by up to ||H|| / min |Re lambda| ~ 10.
"""

import numpy as np
import pytest
import torch

import synth
from oracle import arnoldi, lattice

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _run(gpu, dims, mu, eps, nrhs, k, harmonic=False):
    links = synth.gauge_links(dims, 1, eps)
    h = lattice.hw_operator(links, dims, mu, -1.5)
    g = gpu.create_gauge_from_links(dims, links, gpu.F64)
    gpu.set_mu(g, mu, -1.5)
    x = synth.gaussian_vectors(h.shape[0], nrhs, 3)
    yd = torch.empty((nrhs, h.shape[0]), dtype=torch.complex128, device="cuda")
    st, info = gpu.sign_apply(g, torch.from_numpy(x).cuda(), yd, k, prec=gpu.F64, harmonic=harmonic)
    g.destroy()
    refs = [arnoldi.arnoldi_sign(lambda q: h @ q, x[r], k, harmonic=harmonic) for r in range(nrhs)]
    return st, info, yd.cpu().numpy(), refs


@pytest.mark.parametrize("k", [1, 2, 31, 32, 33, 64, 65, 127, 128, 129, 192, 193, 256, 257])
def test_slot_edges(gpu, k):
    st, info, y, refs = _run(gpu, (2, 4, 4, 4), 0.3, 0.5, 2, k)
    assert st == 0
    for r in range(2):
        assert info[r]["k_used"] == k and 0 < info[r]["newton_iters"] <= 9
        assert rel(y[r], refs[r][0]) < 1e-12, (k, r)


@pytest.mark.parametrize("k", [384, 385, 512, 513, 640, 641, 790])
def test_long_spaces(gpu, k):
    st, info, y, refs = _run(gpu, (4, 4, 4, 4), 0.2, 0.6, 1, k)
    assert st == 0 and info[0]["k_used"] == k
    assert rel(y[0], refs[0][0]) < 1e-12


@pytest.mark.parametrize("mu,iters", [(1.0, 9), (2.0, 13)])
@pytest.mark.parametrize("k,harmonic", [(40, False), (60, False), (60, True)])
def test_wide_spectra(gpu, mu, iters, k, harmonic):
    st, info, y, refs = _run(gpu, (3, 3, 3, 3), mu, 0.6, 2, k, harmonic)
    assert st == 0
    for r in range(2):
        assert info[r]["newton_iters"] <= iters
        assert rel(y[r], refs[r][0]) < 1e-11, (mu, k, r)


def test_next_to_the_imaginary_axis(gpu):
    """Right-hand side 0 has an eigenvalue 0.2 degrees off the imaginary axis
    (|Re lambda| = 2e-3 of the largest |lambda|): Roberts' iteration, with its
    iteration count; 1e-9, the 1e-12 of the tests above times that ratio and
    the norm of the non-normal part (cosh 3 = 10)."""
    st, info, y, refs = _run(gpu, (2, 2, 2, 4), 3.0, 0.6, 1, 41)
    assert st == 0
    assert info[0]["newton_iters"] == refs[0][1]["newton_iters"]
    assert rel(y[0], refs[0][0]) < 1e-9
