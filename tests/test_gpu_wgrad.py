"""Weight and bias gradients of the 3x3 convolution (tensor-core kernel and the scalar one for
channel counts that are no multiple of 8) against a float64 correlation of the same BF16 values."""
import pytest
import torch
import torch.nn.functional as F

from paper_2609_07172_gb300.unet import P, _ok, _st, nn_lib

pytestmark = pytest.mark.gpu


# tiles of 64x8, 32x16 and 16x32 pixels with their remainders; channel blocks of 16 and parts of one
@pytest.mark.parametrize("n,h,w", [(1, 1, 1), (2, 33, 16), (1, 17, 17), (3, 8, 64), (2, 9, 40), (1, 3, 130), (5, 16, 256)])
@pytest.mark.parametrize("cin,cout", [(16, 16), (8, 24), (24, 8), (128, 64), (5, 3)])
def test_wgrad_matches_float64(n, h, w, cin, cout):
    g = torch.Generator().manual_seed(n * 1000 + h * 100 + w + 7 * cin + cout)
    x = torch.randn(n, h, w, cin, generator=g).to(torch.bfloat16).cuda()
    dy = torch.randn(n, h, w, cout, generator=g).to(torch.bfloat16).cuda()
    lib = nn_lib()
    need = lib.pic_nn_wgrad_scratch_floats(cin, cout, n, h, w)
    scratch = torch.full((need + 1,), float("nan"), device="cuda")
    dw = torch.full((9, cout, cin), float("nan"), device="cuda")
    db = torch.full((cout,), float("nan"), device="cuda")
    _ok(lib.pic_nn_conv3x3_wgrad(P(x), cin, P(dy), cout, n, h, w, P(dw), P(db), P(scratch), need, _st()))
    xp = F.pad(x.double(), (0, 0, 1, 1, 1, 1)).cpu()
    d = dy.double().cpu()
    taps = [(xp[:, t // 3:t // 3 + h, t % 3:t % 3 + w].reshape(-1, cin), d.reshape(-1, cout)) for t in range(9)]
    ref = torch.stack([b.T @ a for a, b in taps])
    mag = torch.stack([b.abs().T @ a.abs() for a, b in taps])
    # exact products, FP32 sums: at most 2048 terms one after the other (the scalar kernel; an MMA
    # counts as 16), then the partials, each addition within 2^-23 of the sum of magnitudes
    bound = 2.0 ** -23 * (min(n * h * w, 2048) + 64 + (n * h * w) // 2048)
    assert torch.all((dw.cpu().double() - ref).abs() <= bound * mag)
    assert torch.all((db.cpu().double() - d.reshape(-1, cout).sum(0)).abs() <= bound * d.reshape(-1, cout).abs().sum(0))
    assert torch.isnan(scratch[-1])
