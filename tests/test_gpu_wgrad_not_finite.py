"""Weight gradients where the input or the gradient holds values that are not finite."""
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


@pytest.mark.parametrize("cin,cout", [(16, 16), (8, 24), (5, 3)])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
@pytest.mark.parametrize("where", ["input", "gradient"])
def test_what_does_not_contribute_may_be_anything(where, value, cin, cout):
    """A product enters only where the shifted pixel lies in the image and the gradient is not zero: an infinity in the
    input under zero gradients changes nothing, one in the gradient at the image's corner only the taps that stay inside."""
    n, h, w = 2, 11, 70
    g = torch.Generator().manual_seed(cin)
    x = torch.randint(-8, 9, (n, h, w, cin), generator=g).to(torch.bfloat16).cuda()
    dy = torch.randint(-8, 9, (n, h, w, cout), generator=g).to(torch.bfloat16).cuda()
    if where == "input":
        x[1, 5, 66, 2] = value
        dy[1, 4:7, 65:68] = 0.0
    else:
        dy[0, 0, 0, 1] = value
    dw, db = _wgrad(x, dy)
    xf, df = x.double(), dy.double()
    xf[~torch.isfinite(xf)] = 0.0
    bad = ~torch.isfinite(df)
    df[bad] = 0.0
    xp = F.pad(xf, (0, 0, 1, 1, 1, 1))
    for tap in range(9):
        ref = df.reshape(-1, cout).T @ xp[:, tap // 3:tap // 3 + h, tap % 3:tap % 3 + w].reshape(-1, cin)
        want = torch.ones(cout, cin, dtype=torch.bool, device="cuda")
        if where == "gradient" and tap // 3 >= 1 and tap % 3 >= 1:
            want[1] = False
        got = dw[tap].double()
        assert torch.equal(got[want], ref[want]), tap        # (whole numbers: exact)
        assert not torch.isfinite(got[~want]).any()
    want = ~bad.any(0).any(0).any(0)
    assert torch.equal(db.double()[want], df.sum((0, 1, 2))[want]) and not torch.isfinite(db[~want]).any()
