"""An application does the same work on a handle that has served other sizes before as
on a fresh one: the work space carries over, the split of the sums does not depend on
it (the profile's bytes count the partial sums)."""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

DIMS = (6, 6, 6, 6)
N = 12 * 6**4


def pairs(m, seed):
    r = synth.gaussian_vectors(N, max(m, 1), seed)[:m]
    left = r + 0.3 * synth.gaussian_vectors(N, max(m, 1), seed + 1)[:m]
    return r, left, [0.3 - 0.1j] * m


@pytest.mark.parametrize("prec", ["F64", "MIXED"])
@pytest.mark.parametrize("before,m", [(0, 1), (20, 10), (10, 20)])
def test_deflation_of_another_size_before(gpu, prec, before, m):
    prec = getattr(gpu, prec)
    x = torch.from_numpy(synth.gaussian_vectors(N, 16, 5)).cuda()
    ys, profiles = [], []
    for used in (False, True):
        g = gpu.create_gauge(DIMS, 1, 0.6, gpu.MIXED)
        gpu.set_mu(g, 0.2, -1.5)
        y = torch.empty_like(x)
        if used:
            gpu.deflate_load(g, *pairs(before, 7))
            gpu.sign_apply(g, x[:1].contiguous(), y[:1], 10, prec=prec)
            gpu.set_mu(g, 0.2, -1.5)  # forgets the deflation basis
            gpu.sign_apply(g, x, y, 10, prec=prec)
        gpu.deflate_load(g, *pairs(m, 9))
        gpu.profile_enable(g, False)
        gpu.sign_apply(g, x, y, 10, prec=prec)
        profiles.append({c: (p["launches"], p["bytes"]) for c, p in gpu.profile_read(g).items()})
        g.destroy()
        ys.append(y)
    assert profiles[0] == profiles[1]
    assert torch.equal(ys[0], ys[1])
