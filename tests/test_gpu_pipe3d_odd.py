"""The pipelined 3D step on rows that are not on 16 bytes (4-byte asynchronous copies) against the generic form
(lbm_set_launch depth 1): bitwise equal states, for every wrap and mirror of the x axis, ragged tiles, lattices
narrower than a tile, batches, with and without the mass flux, free rates, and the inlet / outlet columns."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (nx, ny, nz, periodic, instances)
FORMS = [(33, 9, 7, (True, True, True), 1), (35, 8, 12, (False, True, False), 1), (3, 5, 4, (False, False, False), 2),
         (1, 6, 5, (True, True, True), 1), (66, 17, 40, (True, False, True), 1), (2, 9, 9, (False, True, True), 1),
         (31, 20, 18, (False, False, False), 2)]


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("lattice", ["D3Q19", "D3Q15"])
@pytest.mark.parametrize("kw", [dict(rho=(2.0, 2.0, 1.0)), dict(), dict(s_free_ch=0.8, s_free_ns=1.2)],
                         ids=["flux", "equal", "free"])
def test_odd_rows_pipelined_equals_generic(lbm_lib, form, lattice, kw):
    L = lbm_lib
    nx, ny, nz, per, nb = form
    r = np.random.default_rng(5)
    z, y, x = np.mgrid[:nz, :ny, :nx]
    d = 0.3 * max(form[:3]) - np.sqrt((x - nx / 2) ** 2 + (y - ny / 2) ** 2 + (z - nz / 2) ** 2)
    phi0 = np.broadcast_to(0.5 + 0.5 * np.tanh(1.0 - z / 2.0), (nb, nz, ny, nx)).astype(np.float32)
    phi1 = ((1 - phi0) * (0.5 + 0.5 * np.tanh(d / 2)) * r.uniform(0.95, 1.0, (nb, 1, 1, 1))).astype(np.float32)
    prm = [L.lbm_default_params(theta_deg=70.0 + 30 * k, d0=0.3, eta_hat=0.05, mu=(0.1, 0.1, 0.05),
                                body_force=(1e-6, 0, 2e-6), **kw) for k in range(nb)]
    out = []
    for depth in (0, 1):
        with L.Context({"D3Q19": L.LBM_D3Q19, "D3Q15": L.LBM_D3Q15}[lattice], nx, ny, nz, periodic=per,
                       batch=prm) as ctx:
            ctx.set_launch(5, depth)
            ctx.set_solid(phi0)
            ctx.set_phase(phi1)
            if not per[0] and nx >= 4:
                ctx.set_inout(3, np.stack([np.full((nz, ny), 0.01)] + [np.zeros((nz, ny))] * 2).astype(np.float32), 0.0,
                              0.0)
            ctx.step(12)
            out.append((ctx.get_fields(), ctx.get_state()))
    assert all(np.isfinite(v).all() for v in out[0][0])
    assert all(np.array_equal(u, v) for u, v in zip(out[0][0], out[1][0]))
    assert out[0][1] == out[1][1]
