"""Density sums are made of fixed parts, each added up in the order of the sorted particles.

N~ decides which particles iterate h once more, so the rounding of its sum must not
depend on how the work was grouped.  Here every pair has w = 1 to the last bit: piles of
coincident particles sit at the corners where eight cells meet, a few 2^-18 of a cell
apart.  The sums are then sums of masses, which numpy's FP32 additions reproduce.  A
particle of the first cluster of a corner's lowest cell is nobody's partner: its sum is
one part per interaction, first its own cell's, then those of the seven neighbours by
axis, and is compared bit by bit.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIDE = 16                  # cells per dimension: 512 corners, more clusters than the device has warps
H = 0.72 / SIDE
# the lowest cell's neighbours by axis (x first, then y, then z)
NEIGHBOURS = [(1, 0, 0), (0, 1, 0), (1, 1, 0), (0, 0, 1), (1, 0, 1), (0, 1, 1), (1, 1, 1)]


@pytest.fixture(scope="module")
def api():
    from paper_1309_3783_gb300 import build, sph
    build.build()
    return sph


@pytest.mark.parametrize("cmax", [32, 8])
def test_density_parts_are_ordered_sums(api, cmax):
    rng = np.random.default_rng(cmax)
    corners = np.stack(np.meshgrid(*[np.arange(1, SIDE, 2)] * 3, indexing="ij"), -1).reshape(-1, 3)
    cells = [(0, 0, 0)] + NEIGHBOURS
    x, pile = [], {}
    n = 0
    for c, corner in enumerate(corners):
        for d in cells:
            k = int(rng.integers(1, 60))
            at = (corner + np.where(np.array(d) == 1, 1.0, -1.0) * 2.0 ** -18) / SIDE
            x.append(np.repeat(at[None], k, 0))
            pile[c, d] = np.arange(n, n + k)
            n += k
    x = np.concatenate(x)
    order = rng.permutation(n)                   # caller order: piles are sorted by index
    inv = np.empty(n, np.int64)
    inv[order] = np.arange(n)
    x = x[order]
    pile = {k: np.sort(inv[v]) for k, v in pile.items()}
    m = rng.uniform(0.5, 2.0, n).astype(np.float32)
    p = api.sph_params_default()
    p.compensated = 0
    p.cluster_max = cmax
    h = np.full(n, H / p.gamma_kernel, np.float32)
    ctx = api.sph_ctx_create(p, 0)
    try:
        b = api.Box(ctx, n, 1.0, False)
        b.set(x, np.zeros((n, 3), np.float32), m, np.ones(n, np.float32), h)
        b.density()
        rho, count, stats = b.get("rho"), b.get("count"), b.stats()
        b.close()
    finally:
        api.sph_ctx_destroy(ctx)
    assert stats["top_level"] == 4 and stats["n_leaves"] == SIDE ** 3
    f = np.float32
    ih = f(1) / (f(p.gamma_kernel) * h[0])
    k3 = f(2.5464790894703255) * ih * ih * ih
    for c in range(0, len(corners), 8):
        own = pile[c, (0, 0, 0)]
        total = sum(len(pile[c, d]) for d in cells)
        for i in own[:cmax]:
            assert count[i] == total - 1
            s = f(0)
            for d in cells:
                part = f(0)
                for j in pile[c, d]:
                    if j != i:
                        part = part + m[j]
                s = s + part
            assert rho[i] == k3 * (s + m[i]), (c, i)
