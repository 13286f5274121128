"""Device memory of a box."""
import pytest

from paper_1309_3783_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_bytes_per_particle():
    """A box of 100^3 particles held 606 bytes per particle after its first passes before
    the passes took their pairs by cell, and holds no more with them."""
    import torch

    from paper_1309_3783_gb300 import build, sph
    build.build()
    ctx = sph.sph_ctx_create(device=0)
    try:
        small = sph.box_from(ctx, inputs.lattice_box(16))      # what the context itself holds
        small.step(0.0)
        small.close()
        box = inputs.lattice_box(100, jitter=0.2, seed=1)
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        b = sph.box_from(ctx, box)
        b.step(0.0)
        torch.cuda.synchronize()
        used = (free0 - torch.cuda.mem_get_info()[0]) / box.n
        b.close()
    finally:
        sph.sph_ctx_destroy(ctx)
    assert used <= 606 + 4 * 2 ** 20 / box.n, used          # (memory comes in 2 MB blocks)
