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


def _check_passes(api, box, leaf, cmax):
    p = api.sph_params_default()
    p.leaf_max = leaf
    c = api.sph_ctx_create(p, device=0)
    try:
        b = api.box_from(c, box)
        try:
            b.set_cluster_max(cmax)
            b.density()
            b.force()
            got = {k: b.get(k) for k in ("count", "rho", "a", "dudt", "vsig")}
        finally:
            b.close()
    finally:
        api.sph_ctx_destroy(c)
    ref = orc.full_step(box, iterate_h=False, method="kdtree")
    assert np.array_equal(got["count"], ref["count"])
    np.testing.assert_allclose(got["rho"], ref["rho"], rtol=1e-5)
    rms = np.sqrt(np.mean(np.sum(ref["a"] ** 2, axis=1)))
    assert np.max(np.abs(got["a"] - ref["a"])) <= 1e-4 * rms
    assert np.max(np.abs(got["dudt"] - ref["dudt"])) <= 1e-4 * np.sqrt(np.mean(ref["dudt"] ** 2))
    np.testing.assert_allclose(got["vsig"], ref["vsig"], rtol=1e-5)


# Clusters: Morton nodes of up to four clusters' size divided by position (leaves below,
# at and above that size), batches of 32 partners with remainders, a dense clump beside
# sparse cells (the candidates tested against every particle; more pairs in a force batch
# than its list holds).  Units: parts of one cluster (few clusters), one or two per warp,
# and from 4256 clusters on the list of units.
@pytest.mark.parametrize("n,leaf,cmax,clump", [(33, 400, 32, 0.0), (131, 400, 32, 0.0), (1025, 31, 24, 0.1),
                                               (1500, 130, 16, 0.3), (4097, 4800, 32, 0.4), (30000, 400, 32, 0.2),
                                               (60001, 48, 24, 0.1), (130003, 400, 32, 0.2),
                                               (20000, 4800, 32, 0.6), (20000, 1100, 16, 0.6), (9000, 4800, 32, -1.0)])
def test_clusters_and_units(api, n, leaf, cmax, clump):
    side = int(np.ceil(n ** (1 / 3)))
    box = inputs.lattice_box(side, jitter=0.3, seed=n, v_sigma=0.3, periodic=n != 1500)
    box = box.subset(np.arange(box.n - n, box.n))
    rng = np.random.default_rng(n)
    k = int(max(clump, 0.0) * n)
    if k:      # a clump ten times as dense as its surroundings, h to match
        r = 0.5 * (k / n / 10) ** (1 / 3)
        box.x[:k] = np.mod(np.array([0.4, 0.55, 0.6]) + rng.uniform(-r, r, (k, 3)), box.L)
        box.h[:k] *= np.float32(10 ** (-1 / 3))
    if clump < 0:      # points shared by more particles than a node takes: their keys are equal
        box.x[: n // 3] = box.x[rng.integers(0, 12, n // 3) + n // 2]
    box.h = np.minimum(box.h * rng.uniform(0.8, 1.2, n), 0.24 * box.L / 1.8258).astype(np.float32)
    _check_passes(api, box, leaf, cmax)


# Keys from the bits of x / L: coordinates on the borders of cells and one rounding to
# either side, in boxes whose L is a power of two and others (where x / L rounds).
@pytest.mark.parametrize("L", [1.0, 2.5, 0.7, 3.0])
def test_cells_of_coordinates_on_borders(api, L):
    from oracle import decomposition as dc
    box = inputs.lattice_box(18, jitter=0.4, seed=3, L=L)
    rng = np.random.default_rng(11)
    grid = np.round(box.x / L * 64) * (L / 64)
    for pick, x in ((0, grid), (1, np.nextafter(grid, 0.0)), (2, np.nextafter(grid, 2 * L))):
        sel = rng.integers(0, 4, box.x.shape) == pick
        box.x[sel] = np.clip(x, 0.0, np.nextafter(L, 0.0))[sel]
    box.h[rng.integers(0, 3, box.n) > 0] *= np.float32(0.3)
    p = api.sph_params_default()
    p.leaf_max = 8
    c = api.sph_ctx_create(p, device=0)
    try:
        b = api.box_from(c, box)
        try:
            b.build()
            cells = b.cells()
        finally:
            b.close()
    finally:
        api.sph_ctx_destroy(c)
    D = dc.decompose(box.x, orc.support_radius(box.h), L, True, leaf_max=8, headroom=float(p.split_headroom))
    keys = [(int(l), tuple(int(v) for v in ijk)) for l, ijk in zip(cells["level"], cells["ijk"])]
    assert set(keys) == set(D.cells)
    for k, cnt in zip(keys, cells["count"]):
        assert cnt == len(D.cells[k])
