"""The network's input, loss and projection kernels at the edges of their warps and buffers: ragged node counts, rows of
words that are not whole float4, pointers off 16 bytes, one launch per projection pass against two."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.tensor(a, device="cuda")


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n,h,w", [(1, 1, 1), (3, 5, 7), (2, 16, 16), (2, 33, 31)])
def test_pack_input_is_exact(lbm_lib, n, h, w, shift):
    from paper_2311_05091_gb300 import _nn
    r = np.random.default_rng(3)
    p0, p1 = (r.uniform(0, 1, (n, h, w)).astype(np.float32) for _ in range(2))
    ct = r.uniform(-1, 1, n).astype(np.float32)
    P = n * h * w
    buf = torch.full((shift + P * 16 + 64,), -7.0, device="cuda")
    a, b, c = _dev(p0), _dev(p1), _dev(ct)
    _nn.pack_input(a.data_ptr(), b.data_ptr(), c.data_ptr(), buf.data_ptr() + 4 * shift, n, h, w)
    got = buf.cpu().numpy()
    ref = np.zeros((n, h, w, 16), np.float32)
    ref[..., 0], ref[..., 1], ref[..., 2] = p0, p1, ct[:, None, None]
    assert np.array_equal(got[shift:shift + P * 16], ref.ravel())
    assert np.all(got[:shift] == -7.0) and np.all(got[shift + P * 16:] == -7.0)   # nothing outside


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("P,cpad", [(1, 32), (127, 32), (1000, 16), (129, 20), (300, 17), (65, 1), (64, 4)])
def test_mse_residual_is_exact(lbm_lib, P, cpad, shift):
    from paper_2311_05091_gb300 import _nn
    r = np.random.default_rng(4)
    out = r.normal(0, 0.3, (P, cpad)).astype(np.float32)
    base, target = (r.uniform(0, 1, P).astype(np.float32) for _ in range(2))
    buf = torch.full((shift + P * cpad + 64,), -7.0, device="cuda")
    work, loss = (torch.empty(k, dtype=torch.float64, device="cuda") for k in (64, 1))
    o, b, t = _dev(out), _dev(base), _dev(target)
    _nn.mse_residual(o.data_ptr(), cpad, b.data_ptr(), t.data_ptr(), buf.data_ptr() + 4 * shift, work.data_ptr(), 64,
                     loss.data_ptr(), P)
    d = (base + out[:, 0]) - target                          # float32, the kernel's own order
    ref = np.zeros((P, cpad), np.float32)
    ref[:, 0] = np.float32(2) * d / np.float32(P)
    got = buf.cpu().numpy()
    assert np.array_equal(got[shift:shift + P * cpad], ref.ravel())
    assert np.all(got[:shift] == -7.0) and np.all(got[shift + P * cpad:] == -7.0)
    e = np.sum(d.astype(np.float64) ** 2)
    assert abs(loss.item() - e) <= P * 2.0 ** -52 * e        # P additions in FP64


@pytest.mark.parametrize("n,h,w", [(1, 1, 1), (2, 9, 15), (3, 64, 129), (1, 256, 256)])
def test_projection_is_the_same_in_one_launch_per_pass(lbm_lib, n, h, w):
    """Work of 192 n doubles takes two launches per pass, 384 n one: the same sums in the same order."""
    from paper_2311_05091_gb300 import _nn
    r = np.random.default_rng(5)
    phi0 = np.clip(r.normal(0, 0.5, (n, h, w)), 0, 1).astype(np.float32)
    phi1 = np.clip(r.uniform(0, 1, (n, h, w)), 0, 1 - phi0).astype(np.float32)
    out = r.normal(0, 0.3, (n, h, w, 32)).astype(np.float32)
    o, a, b = _dev(out), _dev(phi0), _dev(phi1)
    fields = []
    for doubles in (192 * n, 384 * n):
        work = torch.full((doubles + 8,), -7.0, dtype=torch.float64, device="cuda")
        f = torch.full((n, h, w), float("nan"), device="cuda")
        _nn.project(o.data_ptr(), 32, a.data_ptr(), b.data_ptr(), f.data_ptr(), work.data_ptr(), doubles, n, h, w)
        assert bool((work[doubles:] == -7.0).all())
        fields.append(f.cpu().numpy())
    assert np.array_equal(fields[0], fields[1])
    assert np.all(fields[1] >= 0) and np.all(fields[1] <= np.maximum(1 - phi0, 0) * (1 + 1e-6))
