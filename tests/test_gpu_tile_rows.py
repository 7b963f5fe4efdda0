"""The one-node-per-thread form of the D2Q9 step with tiles of eight rows against the swept form, bitwise, on every kind
of lattice that takes them; the kernel that ran is read from the device's launch records, so that a change of the rule
that chooses it cannot drop the coverage.  And the form on a caller's stream between the caller's own kernels."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# (nx, ny, periodic x, periodic y, instances, FP16, inlet and outlet, tile rows on 152 SMs)
FORMS = [(512, 512, True, True, 1, False, False, 8), (1001, 333, True, True, 1, False, False, 8),
         (1024, 300, True, True, 3, False, False, 8), (1601, 1603, True, True, 1, False, False, 8),
         (700, 301, False, False, 1, False, True, 8), (640, 522, True, False, 1, True, False, 8),
         (520, 505, False, True, 1, True, True, 8), (200, 96, True, True, 1, False, False, 4),
         (200, 97, False, False, 1, True, True, 4)]


def _fields(form):
    nx, ny, _, _, nb, *_ = form
    r = np.random.default_rng(3)
    y, x = np.mgrid[:ny, :nx]
    phi0, phi1 = [], []
    for _ in range(nb):
        d = min(nx, ny) / 4 - np.hypot(x - nx * r.uniform(.3, .7), y - ny * r.uniform(.3, .7))
        s = min(nx, ny) / 6 - np.hypot(x - nx * r.random(), y - ny * r.random())
        phi0.append(0.5 + 0.5 * np.tanh(s / 2))
        phi1.append((1 - phi0[-1]) * (0.5 + 0.5 * np.tanh(d / 2)))
    return np.array(phi0, np.float32), np.array(phi1, np.float32)


def _context(L, form, rates, strip):
    nx, ny, px, py, nb, half, inout, _ = form
    prm = [L.lbm_default_params(theta_deg=60.0 + 20 * k, rho=(2.0, 2.0, 1.0), mu=(0.1, 0.1, 0.05),
                                body_force=(1e-6, 2e-6, 0), **rates) for k in range(nb)]
    ctx = L.Context(L.LBM_D2Q9, nx, ny, 1, periodic=(px, py, False), batch=prm, flags=L.LBM_STORE_G_F16 if half else 0)
    if strip:
        ctx.set_launch(strip)
    if inout:
        ctx.set_inout(3, np.stack([np.full(ny, 0.01), np.zeros(ny)]).astype(np.float32), 0.0, 0.0)
    return ctx


def _run(L, form, rates, strip):
    phi0, phi1 = _fields(form)
    with _context(L, form, rates, strip) as ctx:
        ctx.set_solid(phi0)
        ctx.set_phase(phi1)
        ctx.step(21)                       # replayed graph, single steps and an observed one
        return ctx.get_fields(), ctx.get_state()


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("rates", [{}, dict(s_free_ch=0.8, s_free_ns=1.2)], ids=["unit", "free"])
def test_tile_rows_equal_the_sweep(lbm_lib, form, rates):
    fields, state = _run(lbm_lib, form, rates, 0)
    assert all(np.isfinite(v).all() for v in fields)
    for strip in (5, 16):
        f, s = _run(lbm_lib, form, rates, strip)
        assert all(np.array_equal(u, v) for u, v in zip(fields, f))
        assert state == s


def _launched(work):
    """Names of the kernels that `work` launches, by the profiler's records (it may miss them while it starts)."""
    for _ in range(4):
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            work()
            torch.cuda.synchronize()
        names = {e.key for e in prof.key_averages()}
        if names:
            break
    return names


def test_forms_take_the_kernels_they_name(lbm_lib):
    one = torch.ones(1, device="cuda")
    if not any("kernel" in n for n in _launched(lambda: one.add_(1))):
        pytest.skip("the profiler records no kernels here")
    for form in FORMS:
        phi0, phi1 = _fields(form)
        for strip in (0, 16):
            with _context(lbm_lib, form, {}, strip) as ctx:
                ctx.set_solid(phi0)
                ctx.set_phase(phi1)
                ran = {n for n in _launched(lambda: ctx.step(2)) if "d2q9_" in n}
            want = "d2q9_step" if strip else "d2q9_tile"
            assert ran and all(want in n for n in ran), (form, strip, ran)
            assert strip or all(f"{form[7]}>" in n for n in ran), (form, ran)


@pytest.mark.parametrize("form", [FORMS[0], FORMS[4], FORMS[7]])
def test_tiles_between_kernels_of_the_caller(lbm_lib, form):
    """New solids and phases written by the caller's kernels on the context's stream, without a wait in between."""
    L = lbm_lib
    phi0, phi1 = (torch.tensor(a, device="cuda") for a in _fields(form))
    out = []
    for strip, wait in ((0, False), (16, True)):
        stream = torch.cuda.Stream()
        with _context(L, form, {}, strip) as ctx, torch.cuda.stream(stream):
            stream.wait_stream(torch.cuda.default_stream())
            ctx.set_stream(stream.cuda_stream)
            a, b = torch.empty_like(phi0), torch.empty_like(phi1)
            after = (lambda: torch.cuda.synchronize()) if wait else (lambda: None)
            for k in range(4):
                torch.mul(torch.roll(phi0, k, -1), 1 - 0.01 * k, out=a)
                after()
                ctx.set_solid_device(a.data_ptr())
                if k % 2 == 0:
                    torch.minimum(phi1 * (1 - 0.1 * k), 1 - a, out=b)
                    after()
                    ctx.set_phase_device(b.data_ptr())
                ctx.step(19)
                after()
                a.fill_(float("nan"))      # the caller's buffers are free again once the copies are enqueued
                b.fill_(float("nan"))
            ctx.sync()
            out.append((ctx.get_fields(), ctx.get_state()))
    assert all(np.isfinite(v).all() for v in out[0][0])
    assert all(np.array_equal(u, v) for u, v in zip(out[0][0], out[1][0]))
    assert out[0][1] == out[1][1]
