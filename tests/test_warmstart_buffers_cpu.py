"""The buffers that WarmStartNet hands to the kernels (recorded instead of launched: no GPU needed)."""
import pytest
import torch


@pytest.mark.parametrize("n,h,w", [(1, 64, 64), (1, 128, 128), (3, 192, 192), (16, 64, 64), (1, 256, 256)])
def test_prediction_projects_in_one_launch_per_pass(lbm_lib, monkeypatch, n, h, w):
    from paper_2311_05091_gb300 import _nn
    from paper_2311_05091_gb300.warmstart import WarmStartNet
    calls = {}
    for name in ("to_bf16", "flip_transpose", "pack_input", "conv3x3", "pool2", "up2", "add", "project", "mse_residual"):
        monkeypatch.setattr(_nn, name, lambda *a, _n=name, **k: calls.setdefault(_n, []).append(a))
    net = WarmStartNet(widths=(32, 64), n=n, h=h, w=w, device="cpu")
    f = torch.zeros((n, h, w))
    net.predict(f, f, torch.zeros(n), torch.empty_like(f))
    (out, cpad, phi0, phi1, field, work, work_len, pn, ph, pw), = calls["project"]
    assert (pn, ph, pw) == (n, h, w) and work == net.dwork.data_ptr()
    assert work_len == net.dwork.numel() and work_len >= 384 * n
    # the loss partials of a training step share the buffer
    assert net.dwork.numel() >= -(-n * h * w // 128)
