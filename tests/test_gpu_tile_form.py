"""The one-node-per-thread form of the D2Q9 step (small lattices) against the swept form: bitwise equal states.

Sizes at the edges of the 32 x 4 and 32 x 8 tiles and of the sweep's 128-column tiles, walls on either axis, lattices
narrower than a halo, batches, FP16 populations, free relaxation rates and the inlet / outlet columns."""
import numpy as np
import pytest

from synthetic import random_disks_droplet

pytestmark = pytest.mark.gpu

# (nx, ny, periodic x, periodic y, instances, FP16)
FORMS = [(128, 64, True, False, 1, False), (1, 40, True, True, 1, False), (3, 5, False, True, 1, False),
         (31, 33, False, False, 2, False), (33, 31, True, True, 1, False), (129, 9, True, False, 1, False),
         (127, 128, False, True, 1, False), (256, 96, True, True, 3, False), (264, 52, False, False, 2, True),
         (640, 520, True, True, 1, True), (483, 800, True, False, 2, False)]


def _state(L, form, strip, steps, rates, inout):
    nx, ny, px, py, nb, half = form
    r = np.random.default_rng(3)
    y, x = np.mgrid[:ny, :nx]
    phi0, phi1 = [], []
    for _ in range(nb):
        d = min(nx, ny) / 4 - np.hypot(x - nx * r.uniform(.3, .7), y - ny * r.uniform(.3, .7))
        s = min(nx, ny) / 6 - np.hypot(x - nx * r.random(), y - ny * r.random())
        phi0.append(0.5 + 0.5 * np.tanh(s / 2))
        phi1.append((1 - phi0[-1]) * (0.5 + 0.5 * np.tanh(d / 2)))
    prm = [L.lbm_default_params(theta_deg=60.0 + 20 * k, rho=(2.0, 2.0, 1.0), mu=(0.1, 0.1, 0.05), body_force=(1e-6, 2e-6, 0),
                                **rates) for k in range(nb)]
    ctx = L.Context(L.LBM_D2Q9, nx, ny, 1, periodic=(px, py, False), batch=prm, flags=L.LBM_STORE_G_F16 if half else 0)
    try:
        if strip:
            ctx.set_launch(strip)
        ctx.set_solid(np.array(phi0, np.float32))
        ctx.set_phase(np.array(phi1, np.float32))
        if inout:
            ctx.set_inout(3, np.stack([np.full(ny, 0.01), np.zeros(ny)]).astype(np.float32), 0.0, 0.0)
        ctx.step(steps)
        return ctx.get_fields(), ctx.get_state()
    finally:
        ctx.close()


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("rates", [{}, dict(s_free_ch=0.8, s_free_ns=1.2)], ids=["unit", "free"])
def test_tile_form_equals_sweep(lbm_lib, form, rates):
    inout = not form[2] and form[0] >= 4
    a = _state(lbm_lib, form, 0, 21, rates, inout)
    for strip in (5, 16):
        b = _state(lbm_lib, form, strip, 21, rates, inout)
        assert all(np.isfinite(v).all() for v in a[0])
        assert all(np.array_equal(u, v) for u, v in zip(a[0], b[0]))
        assert a[1] == b[1]


def test_tuner_keeps_the_state_and_either_form(lbm_lib):
    L = lbm_lib
    geo, theta = random_disks_droplet(n=128, seed=5)
    out = []
    for tune in (False, True):
        with L.Context(L.LBM_D2Q9, 128, 128, 1, periodic=(True, True, False),
                       params=L.lbm_default_params(theta_deg=theta, kappa=geo.kappa)) as ctx:
            ctx.set_solid(geo.phi0.astype(np.float32))
            ctx.set_phase(geo.phi1.astype(np.float32))
            ctx.step(10)
            if tune:
                before = ctx.get_state()
                ctx.tune(3)
                assert ctx.get_state() == before
            ctx.step(40)
            out.append(ctx.get_state())
    assert out[0] == out[1]
