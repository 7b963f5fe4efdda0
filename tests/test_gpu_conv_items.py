"""The forward convolution where one CTA walks several work items: its ring of stages and its two accumulator
sets wrap, blocks of rows run across image borders and the last blocks are ragged."""
import numpy as np
import pytest
import torch

from oracle import nn as onn

pytestmark = pytest.mark.gpu


# one stage per item and more than six items per CTA; two stages per item; four stages, blocks across images of odd
# height; channel tiles of 128 with several tiles per image
@pytest.mark.parametrize("n,h,w,cin,cout", [(14, 256, 250, 16, 32), (5, 200, 256, 64, 32), (31, 33, 31, 128, 64),
                                            (6, 64, 64, 64, 256)])
def test_forward_over_many_items(lbm_lib, n, h, w, cin, cout):
    from paper_2311_05091_gb300 import _nn
    r = np.random.default_rng(7)
    x = r.normal(0, 1, (n, h, w, cin)).astype(np.float32)
    wt = torch.tensor(r.normal(0, 0.2, (9, cout, cin)).astype(np.float32)).bfloat16()
    b = r.normal(0, 0.1, cout).astype(np.float32)
    xd, wd, bd = torch.tensor(x, device="cuda"), wt.cuda(), torch.tensor(b, device="cuda")
    y = torch.full((n, h, w, cout), float("nan"), device="cuda")
    _nn.conv3x3(xd.data_ptr(), wd.data_ptr(), bd.data_ptr(), y.data_ptr(), n, h, w, cin, cout, False)
    got = y.cpu().numpy()
    _nn.check()
    W = wt.float().numpy()
    # float32 accumulation: within 1e-5 of the sum of absolute products, image by image
    for i in {0, n // 2, n - 1}:
        ref = onn.conv3x3(x[i:i + 1], W, b.astype(np.float64))
        bound = onn.conv3x3(np.abs(onn.bf16_round(x[i:i + 1])), np.abs(W), np.abs(b.astype(np.float64)), bf16=False)
        assert np.all(np.abs(got[i:i + 1] - ref) <= 1e-5 * bound + 1e-30)
    assert np.all(np.isfinite(got))


# the weight gradient over several segments of a chunk and several column strips: three, two and one of x's column
# shifts per product, ragged channel tiles on both sides, one and two accumulator sets, images of one row
@pytest.mark.parametrize("n,h,w,cin,cout", [(4, 150, 260, 32, 32), (3, 101, 131, 64, 32), (2, 90, 140, 80, 96),
                                            (5, 64, 64, 128, 64), (9, 1, 300, 48, 16), (3, 33, 32, 256, 144)])
def test_weight_gradient_over_segments_and_strips(lbm_lib, n, h, w, cin, cout):
    from paper_2311_05091_gb300 import _nn
    r = np.random.default_rng(8)
    x = r.normal(0, 1, (n, h, w, cin)).astype(np.float32)
    dy = r.normal(0, 1, (n, h, w, cout)).astype(np.float32)
    xd, dyd = torch.tensor(x, device="cuda"), torch.tensor(dy, device="cuda")
    dw = torch.full((9, cout, cin), float("nan"), device="cuda")
    db = torch.full((cout,), float("nan"), device="cuda")
    work = torch.full((_nn.wgrad_workspace(n, h, w, cin, cout),), float("nan"), device="cuda")
    _nn.conv3x3_wgrad(xd.data_ptr(), dyd.data_ptr(), dw.data_ptr(), db.data_ptr(), work.data_ptr(), work.numel(), n, h,
                      w, cin, cout)
    got, gdb = dw.cpu().numpy(), db.cpu().numpy()
    _nn.check()
    zero = np.zeros((9, cout, cin))
    _, ref, rdb = onn.conv3x3_grads(x, zero, dy)
    _, bound, _ = onn.conv3x3_grads(np.abs(onn.bf16_round(x)), zero, np.abs(onn.bf16_round(dy)), bf16=False)
    # float32 accumulation: within 1e-5 of the sum of absolute products
    assert np.all(np.abs(got - ref) <= 1e-5 * bound + 1e-30)
    assert np.all(np.abs(gdb - rdb) <= 1e-5 * np.abs(dy).sum(axis=(0, 1, 2)))
