"""Weight gradients: sums over very many pixels."""
import pytest
import torch
import torch.nn.functional as F

from paper_2609_07172_gb300.unet import P, _ok, _st, nn_lib

pytestmark = pytest.mark.gpu


def _wgrad(x, dy):
    n, h, w, cin = x.shape
    cout = dy.shape[-1]
    lib = nn_lib()
    need = lib.pic_nn_wgrad_scratch_floats(cin, cout, n, h, w)
    scratch = torch.empty(need, device="cuda")
    dw = torch.empty(9, cout, cin, device="cuda")
    db = torch.empty(cout, device="cuda")
    _ok(lib.pic_nn_conv3x3_wgrad(P(x), cin, P(dy), cout, n, h, w, P(dw), P(db), P(scratch), need, _st()))
    return dw, db


@pytest.mark.parametrize("n,h,w,cin,cout", [(16384, 16, 16, 64, 128), (2048, 64, 64, 16, 16)])
def test_sums_of_many_pixels(n, h, w, cin, cout):
    """Terms of one sign, so that an accumulator that is cut at every addition drifts.  A warp's accumulator
    takes 32 MMAs at most (each cut by up to 2 units in the last place of the sum), then 8 warps, an eighth of the
    partials of 4096 pixels and the eight eighths are added, each within half a unit."""
    g = torch.Generator(device="cuda").manual_seed(n)
    x = (0.5 + 0.5 * torch.rand(n, h, w, cin, generator=g, device="cuda")).to(torch.bfloat16)
    dy = (0.5 + 0.5 * torch.rand(n, h, w, cout, generator=g, device="cuda")).to(torch.bfloat16)
    dw, db = _wgrad(x, dy)
    parts = (n * h * w + 4095) // 4096
    bound = 2.0 ** -23 * (2 * 32 + 0.5 * (8 + (parts + 7) // 8 + 8))
    for tap in (0, 4, 5):
        ref = torch.zeros(cout, cin, dtype=torch.float64, device="cuda")
        for s in range(0, n, 1024):
            xp = F.pad(x[s:s + 1024].double(), (0, 0, 1, 1, 1, 1))[:, tap // 3:tap // 3 + h, tap % 3:tap % 3 + w]
            ref += dy[s:s + 1024].double().reshape(-1, cout).T @ xp.reshape(-1, cin)
        rel = ((dw[tap].double() - ref).abs() / ref).max().item()
        assert rel <= bound, (tap, rel, bound)
    ref = dy.double().sum((0, 1, 2))
    assert ((db.double() - ref).abs() / ref).max().item() <= bound
