"""An autotuner that cannot save the state: it launches nothing and reports what failed."""
import numpy as np
import pytest

from synthetic import random_disks_droplet

pytestmark = pytest.mark.gpu


# a lattice that runs tiles and one whose strip was set
@pytest.mark.parametrize("strip", [0, 16])
@pytest.mark.parametrize("given", [0, 1, 2])
def test_refused_save_area_is_reported(lbm_lib, strip, given):
    import torch
    L = lbm_lib
    geo, theta = random_disks_droplet(n=128, seed=5)
    pool = L.TorchAllocator()
    left = [1 << 30]                         # allocations still granted

    def alloc(nbytes, stream, user):
        left[0] -= 1
        return pool.alloc(nbytes, stream, user) if left[0] >= 0 else None
    refusing = type("Refusing", (), {})()
    refusing.alloc, refusing.free = L.lbm_alloc_fn(alloc), pool.free
    stream = torch.cuda.Stream()
    ctx = L.Context(L.LBM_D2Q9, 128, 128, 1, periodic=(True, True, False), allocator=refusing, stream=stream.cuda_stream,
                    params=L.lbm_default_params(theta_deg=theta, kappa=geo.kappa))
    try:
        if strip:
            ctx.set_launch(strip)
        ctx.set_solid(geo.phi0.astype(np.float32))
        ctx.set_phase(geo.phi1.astype(np.float32))
        left[0] = given
        with pytest.raises(L.LbmError, match="out of memory"):
            ctx.tune(2)
    finally:
        left[0] = 1 << 30
        ctx.close()
