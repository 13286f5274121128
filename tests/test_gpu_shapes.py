"""Sizes at which the splits of the kernels change, against the FP64 oracle.

Neighbour counts are exact.  Sums: an FP32 term is off by a few 2^-24 of itself, a sum
of up to a few hundred terms of one sign by no more than 1e-6; 1e-5 leaves room for the
terms near the support's edge, whose kernel is a difference.  Accelerations cancel, so
they are compared on the scale of their root mean square (1e-4, as elsewhere here).
"""
import numpy as np
import pytest

from oracle import sph as orc
from paper_1309_3783_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1309_3783_gb300 import build, sph
    build.build()
    return sph


# a warp per particle and four per block, a thread of an 8 x 1024 cluster per particle
# or two, cell lists of 1 (open) or 3 (periodic) to 20 cells per dimension
@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("n,scale", [(1, 1.0), (2, 3.0), (31, 1.0), (33, 2.0), (1025, 1.0), (8191, 0.4), (8193, 1.0),
                                     (16384, 0.3), (16384, 1.0)])
def test_static_density_sizes(api, n, scale, periodic):
    import torch
    rng = np.random.default_rng(n)
    L = 2.5
    x = rng.uniform(0.0, L, (n, 3))
    x[: n // 8] = np.mod(0.3 + 0.02 * rng.standard_normal((n // 8, 3)), L)     # a clump across no particular cell
    h = (scale * 1.2 * L * n ** (-1 / 3) * rng.uniform(0.6, 1.3, n)).astype(np.float32)
    if periodic:
        h = np.minimum(h, np.float32(0.33 * L / 1.8258))
    m = rng.uniform(0.5, 2.0, n).astype(np.float32)
    rho = torch.full((n,), -1.0, device="cuda")
    cnt = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    dev = [torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda() for a in (x, m, h)]
    assert api.sph_density_static(*dev, L, periodic, rho, cnt) == 0
    ref = orc.density(x, m, orc.support_radius(h), L, periodic)
    assert np.array_equal(cnt.cpu().numpy(), ref["count"])
    np.testing.assert_allclose(rho.cpu().numpy(), ref["rho"], rtol=1e-5)
