"""The two-input convolution and its weight gradient against the same calls on the written
concatenation, and the 16-byte element-wise kernels against the two-byte ones."""
import pytest
import torch

from paper_2609_07172_gb300.unet import P, _ok, _st, nn_lib

pytestmark = pytest.mark.gpu


def _bf(*shape, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(*shape, generator=g).to(torch.bfloat16).cuda()


def _cat(up, skip):
    return torch.cat([up.repeat_interleave(2, 1).repeat_interleave(2, 2), skip], 3).contiguous()


# wide images (both inputs read in place), several tiles per row, few rows; narrow and untileable ones
# (concatenation written); weights too large to stay resident
@pytest.mark.parametrize("n,h,w", [(1, 2, 128), (3, 10, 256), (2, 6, 384), (2, 8, 64), (1, 4, 40)])
@pytest.mark.parametrize("cu,cs,cout", [(16, 16, 16), (32, 32, 16), (16, 32, 48), (64, 64, 32), (64, 64, 128)])
def test_cat_convolution_is_the_convolution_of_the_concatenation(n, h, w, cu, cs, cout):
    lib = nn_lib()
    up, skip = _bf(n, h // 2, w // 2, cu, seed=1), _bf(n, h, w, cs, seed=2)
    wt, bias = _bf(9, cout, cu + cs, seed=3), torch.randn(cout, generator=torch.Generator().manual_seed(4)).cuda()
    cat = _cat(up, skip)
    out, ref = [torch.full((n, h, w, cout), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    out32, ref32 = [torch.full((n, h, w, cout), float("nan"), device="cuda") for _ in range(2)]
    work = torch.empty_like(cat)
    _ok(lib.pic_nn_conv3x3_cat(P(up), cu, P(skip), cs, P(wt), P(bias), P(work), P(out), P(out32), cout, n, h, w, 1, _st()))
    _ok(lib.pic_nn_conv3x3(P(cat), cu + cs, P(wt), P(bias), P(ref), P(ref32), cout, n, h, w, 1, _st()))
    assert torch.equal(out, ref) and torch.equal(out32, ref32)
    need = lib.pic_nn_wgrad_scratch_floats(cu + cs, cout, n, h, w)
    scratch = torch.empty(need, device="cuda")
    dy = _bf(n, h, w, cout, seed=5)
    got, want = [(torch.empty(9, cout, cu + cs, device="cuda"), torch.empty(cout, device="cuda")) for _ in range(2)]
    _ok(lib.pic_nn_conv3x3_wgrad_cat(P(up), cu, P(skip), cs, P(dy), cout, n, h, w, P(got[0]), P(got[1]), P(scratch),
                                     need, _st()))
    _ok(lib.pic_nn_conv3x3_wgrad(P(cat), cu + cs, P(dy), cout, n, h, w, P(want[0]), P(want[1]), P(scratch), need, _st()))
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


# 8 and 16 channels take 16-byte accesses; 6 channels, and 8 channels one element off alignment, do not
@pytest.mark.parametrize("c,shift", [(8, 0), (16, 0), (6, 0), (8, 1)])
def test_elementwise_kernels(c, shift):
    lib = nn_lib()
    n, h, w = 3, 6, 10

    def place(t):      # the values at an address `shift` elements past a 16-byte boundary
        buf = torch.empty(t.numel() + 8, dtype=t.dtype, device="cuda")
        v = buf[shift:shift + t.numel()].view(t.shape)
        v.copy_(t)
        return v

    x, y = _bf(n, h, w, c, seed=7), _bf(n, h, w, c, seed=8)
    half = _bf(n, h // 2, w // 2, c, seed=9)
    d = place(y)
    _ok(lib.pic_nn_relu_bwd(P(place(x)), P(d), d.numel(), _st()))
    assert torch.equal(d, torch.where(x > 0, y, torch.zeros_like(y)))
    a = place(x)
    _ok(lib.pic_nn_add(P(a), P(place(y)), a.numel(), _st()))
    assert torch.equal(a, (x.float() + y.float()).to(torch.bfloat16))
    b = x.float().view(n, h // 2, 2, w // 2, 2, c)
    total = b[:, :, 0, :, 0] + b[:, :, 0, :, 1] + b[:, :, 1, :, 0] + b[:, :, 1, :, 1]
    out = place(torch.zeros_like(half))
    _ok(lib.pic_nn_pool2(P(place(x)), P(out), n, h, w, c, 0, _st()))
    assert torch.equal(out, (0.25 * total).to(torch.bfloat16))
    out = place(torch.zeros_like(x))
    _ok(lib.pic_nn_pool2(P(place(half)), P(out), n, h, w, c, 1, _st()))
    spread = half.repeat_interleave(2, 1).repeat_interleave(2, 2)
    assert torch.equal(out, (0.25 * spread.float()).to(torch.bfloat16))
    wide = place(torch.zeros(n, h, w, 2 * c, dtype=torch.bfloat16, device="cuda"))
    _ok(lib.pic_nn_up2(P(place(half)), P(wide), n, h // 2, w // 2, c, 2 * c, 0, _st()))
    _ok(lib.pic_nn_copy_channels(P(place(x)), c, 0, P(wide), 2 * c, c, n * h * w, c, _st()))
    assert torch.equal(wide, torch.cat([spread, x], 3))
    out = place(torch.zeros_like(half))
    _ok(lib.pic_nn_up2(P(place(torch.cat([x, y], 3).contiguous())), P(out), n, h // 2, w // 2, c, 2 * c, 1, _st()))
    assert torch.equal(out, total.to(torch.bfloat16))


@pytest.mark.parametrize("c,used", [(16, 2), (8, 8), (6, 2)])
def test_mse(c, used):
    lib = nn_lib()
    pix = 1003
    g = torch.Generator().manual_seed(c + used)
    pred, target = torch.randn(pix, c, generator=g).cuda(), torch.randn(pix, used, generator=g).cuda()
    dp = torch.full((pix, c), float("nan"), dtype=torch.bfloat16, device="cuda")
    scratch, loss = torch.empty((pix * c + 255) // 256, device="cuda"), torch.empty(1, device="cuda")
    _ok(lib.pic_nn_mse(P(pred), P(target), pix, c, used, P(dp), P(scratch), P(loss), _st()))
    d = pred[:, :used] - target
    grad = torch.zeros(pix, c, device="cuda")
    grad[:, :used] = 2.0 * d / (pix * used)
    assert torch.equal(dp, grad.to(torch.bfloat16))
    ref = d.double().square().mean()
    assert abs(loss.double() - ref) <= 64 * 2.0 ** -24 * ref     # FP32 sums of at most 64 terms in a row


# two rows per tile (wide images, one and several tiles per row) and the two-pass form
@pytest.mark.parametrize("n,h,w", [(1, 2, 128), (3, 10, 256), (2, 6, 64), (1, 4, 40)])
@pytest.mark.parametrize("cin,cout", [(16, 16), (16, 32), (64, 48), (64, 128)])
def test_pooled_convolution_is_convolution_then_pooling(n, h, w, cin, cout):
    lib = nn_lib()
    x, wt = _bf(n, h, w, cin, seed=11), _bf(9, cout, cin, seed=12)
    bias = torch.randn(cout, generator=torch.Generator().manual_seed(13)).cuda()
    out, ref = [torch.full((n, h, w, cout), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    pool, pref = [torch.full((n, h // 2, w // 2, cout), float("nan"), dtype=torch.bfloat16, device="cuda")
                  for _ in range(2)]
    _ok(lib.pic_nn_conv3x3_pool(P(x), cin, P(wt), P(bias), P(out), P(pool), cout, n, h, w, 1, _st()))
    _ok(lib.pic_nn_conv3x3(P(x), cin, P(wt), P(bias), P(ref), None, cout, n, h, w, 1, _st()))
    _ok(lib.pic_nn_pool2(P(ref), P(pref), n, h, w, cout, 0, _st()))
    assert torch.equal(out, ref) and torch.equal(pool, pref)


# an odd number of rows: the last tile's second row lies outside the image
@pytest.mark.parametrize("cin,cout", [(16, 16), (32, 16), (64, 16)])
def test_wide_convolution_with_an_odd_number_of_rows(cin, cout):
    lib = nn_lib()
    n, h, w = 2, 7, 256
    x, wt = _bf(n, h, w, cin, seed=21), _bf(9, cout, cin, seed=22)
    out, ref = [torch.full((n, h, w, cout), float("nan"), device="cuda") for _ in range(2)]
    guard = torch.full((n * h * w * cout + 4096,), float("nan"), device="cuda")
    _ok(lib.pic_nn_conv3x3(P(x), cin, P(wt), None, None, P(guard), cout, n, h, w, 0, _st()))
    _ok(lib.pic_nn_conv3x3_mma_sync(P(x), cin, P(wt), None, None, P(ref), cout, n, h, w, 0, _st()))
    out = guard[:ref.numel()].view(ref.shape)
    assert torch.isnan(guard[ref.numel():]).all()
    # FP32 sums of the same 9 cin exact products in two orders
    assert torch.all((out - ref).abs() <= 9 * cin * 2.0 ** -22 * ref.abs().max())
