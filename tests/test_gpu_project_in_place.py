"""The projection with the field in place of the phase field it starts from, whose sum is then no target to read again in
a later pass: the workspace that allows one launch per pass must not change the result."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("together", [True, False])
@pytest.mark.parametrize("n,h,w", [(1, 9, 15), (2, 64, 129), (1, 256, 256)])
def test_workspace_does_not_change_a_projection_in_place(lbm_lib, n, h, w, together):
    from paper_2311_05091_gb300 import _nn
    r = np.random.default_rng(6)
    P = n * h * w
    phi0 = np.clip(r.normal(0, 0.5, P), 0, 1).astype(np.float32)
    phi1 = np.clip(r.uniform(0, 1, P), 0, 1 - phi0).astype(np.float32)
    o, a = (torch.tensor(v, device="cuda") for v in (r.normal(0, 0.3, (P, 32)).astype(np.float32), phi0))
    fields = []
    for doubles in (192 * n, 384 * n):
        work = torch.full((doubles + 8,), -7.0, dtype=torch.float64, device="cuda")
        buf = torch.zeros(2 * P, device="cuda")
        start, field = buf[:P], buf[:P] if together else buf[P:]   # the same buffer, or the one right behind
        start.copy_(torch.tensor(phi1, device="cuda"))
        _nn.project(o.data_ptr(), 32, a.data_ptr(), start.data_ptr(), field.data_ptr(), work.data_ptr(), doubles, n, h, w)
        assert bool((work[doubles:] == -7.0).all())
        fields.append(field.cpu().numpy())
    assert np.array_equal(fields[0], fields[1])
    assert np.all(fields[0] >= 0) and np.all(fields[0] <= np.maximum(1 - phi0, 0).reshape(-1) * (1 + 1e-6))
