"""The weight gradient on shapes and buffers far from the network's: images far taller than wide, tensors on 16 bytes
but not on 32."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _ints(shape, seed, shift=0):
    """Whole numbers in -2 .. 2 (exact in BF16), `shift` floats behind an aligned start."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    k = 1
    for s in shape:
        k *= s
    buf = torch.empty(k + shift, device="cuda")
    buf[shift:] = torch.randint(-2, 3, (k,), generator=g, device="cuda").float()
    return buf[shift:].view(shape)


def _reference(x, dy):
    """[tap][co][ci] and [co].  Every partial sum is a whole number below 2^24, so float32 holds it exactly."""
    n, h, w, cin = x.shape
    assert 4 * n * h * w < 2 ** 24 and not torch.backends.cuda.matmul.allow_tf32
    out = torch.zeros((9, dy.shape[3], cin), device="cuda")
    for tap in range(9):
        ky, kx = tap // 3 - 1, tap % 3 - 1
        ys, xs = slice(max(0, -ky), min(h, h - ky)), slice(max(0, -kx), min(w, w - kx))
        yx, xx = slice(max(0, ky), min(h, h + ky)), slice(max(0, kx), min(w, w + kx))
        for i in range(n):
            out[tap] += dy[i, ys, xs].reshape(-1, dy.shape[3]).T @ x[i, yx, xx].reshape(-1, cin)
    return out, dy.sum(dim=(0, 1, 2))


def _wgrad(x, dy):
    from paper_2311_05091_gb300 import _nn
    (n, h, w, cin), cout = x.shape, dy.shape[3]
    dw = torch.full((9, cout, cin), float("nan"), device="cuda")
    db = torch.full((cout,), float("nan"), device="cuda")
    work = torch.full((_nn.wgrad_workspace(n, h, w, cin, cout),), float("nan"), device="cuda")
    _nn.conv3x3_wgrad(x.data_ptr(), dy.data_ptr(), dw.data_ptr(), db.data_ptr(), work.data_ptr(), work.numel(), n, h, w,
                      cin, cout)
    torch.cuda.synchronize()
    _nn.check()
    return dw, db


# segments that span several images of more than 2^16 rows, with one column and with several
@pytest.mark.parametrize("n,h,w,cin,cout", [(2, 65536, 1, 1536, 768), (2, 65536, 1, 768, 1536), (40, 50000, 2, 64, 32)])
def test_tall_images_are_exact(lbm_lib, n, h, w, cin, cout):
    x, dy = _ints((n, h, w, cin), 1), _ints((n, h, w, cout), 2)
    dw, db = _wgrad(x, dy)
    ref, rdb = _reference(x, dy)
    assert torch.equal(dw, ref) and torch.equal(db, rdb)


# 16-byte loads: either tensor, or both, half a 32-byte sector off; folded and plain channel tiles, one row, strips
@pytest.mark.parametrize("sx,sdy", [(4, 0), (0, 4), (4, 4)])
@pytest.mark.parametrize("n,h,w,cin,cout", [(2, 13, 17, 16, 32), (3, 40, 140, 64, 48), (1, 1, 300, 128, 64),
                                            (2, 33, 31, 80, 144)])
def test_tensors_on_sixteen_bytes(lbm_lib, n, h, w, cin, cout, sx, sdy):
    x, dy = _ints((n, h, w, cin), 3, sx), _ints((n, h, w, cout), 4, sdy)
    assert (x.data_ptr() | dy.data_ptr()) % 32 == 16 and x.is_contiguous()
    dw, db = _wgrad(x, dy)
    ref, rdb = _reference(x, dy)
    assert torch.equal(dw, ref) and torch.equal(db, rdb)
