"""Rounding of the complex128 form's Krylov basis (csrc/fix_sweeps.cu): the first
basis vector against x / ||x||, for sources whose elements differ by many orders of
magnitude or are zero.

An element is a whole number of units of 2^-58 of a scale that is a power of two at
most four times the vector's largest element, within 3/4 of a unit: 3 * 2^-58 of that
element. x / ||x|| itself adds 2^-51 of the element (a norm, a square root and a product
in FP64). Zeros stay zeros.
"""

import math

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def source(kind, n):
    x = synth.gaussian_vectors(n, 1, 23)[0]
    if kind == "point":
        x[:] = 0.0
        x[5] = 1.0 - 0.5j
    if kind == "chiral":
        x.reshape(-1, 12)[:, 6:] = 0.0
    if kind == "real":
        x = x.real + 0j
    if kind == "steep":
        x *= 10.0 ** -np.linspace(0.0, 25.0, n)
    return x


@pytest.mark.parametrize("dims", [(2, 3, 5, 3), (4, 4, 4, 4), (6, 6, 6, 6)])
@pytest.mark.parametrize("kind", ["point", "chiral", "real", "steep", "gauss"])
def test_first_vector(gpu, dims, kind):
    n = 12 * int(np.prod(dims))
    x = source(kind, n)
    g = gpu.create_gauge(dims, 1, 0.6, gpu.F64)
    gpu.set_mu(g, 0.2, -1.5)
    xd = torch.from_numpy(x[None]).cuda()
    gpu.sign_apply(g, xd, torch.empty_like(xd), 3, prec=gpu.F64)
    got = gpu.get_krylov(g, 0)[0][0]
    g.destroy()
    want = x / math.sqrt(math.fsum((x.real**2).tolist() + (x.imag**2).tolist()))
    top = max(np.abs(want.real).max(), np.abs(want.imag).max())
    for a, b in ((got.real, want.real), (got.imag, want.imag)):
        assert np.all(a[b == 0.0] == 0.0)
        assert np.all(np.abs(a - b) <= 3.0 * 2.0**-58 * top + 2.0**-51 * np.abs(b))
