"""The transforms of values below binary64's normal range (their arithmetic is in integers)."""
import numpy as np
import pytest
import torch

from paper_2609_07172_gb300 import Plan, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("power", [-1022, -1030, -1050])
@pytest.mark.parametrize("nt", [2, 8, 64, 256])
def test_transforms_of_subnormal_values(nt, power):
    p = W.annulus(34, nt, 3, phi_z0=0.0)
    rng = np.random.default_rng(nt)
    x = rng.uniform(-1.0, 1.0, p.shape)
    small = np.ldexp(x, power)
    with Plan(p) as plan:
        got = plan.analyze(torch.from_numpy(small).cuda()).cpu().numpy()
        back = plan.inverse(torch.from_numpy(np.ldexp(np.stack([x[:, :1].transpose(0, 2, 1), 0 * x[:, :1].transpose(0, 2, 1)], -1).repeat(
            nt // 2 + 1, 2), power)).cuda()).cpu().numpy()
    m = np.fft.rfft(np.ldexp(small, 1000), axis=1).transpose(0, 2, 1) / nt     # (normal here, the inputs' own rounding included)
    want = np.ldexp(np.stack([m.real, m.imag], -1), -1000)
    # one rounding to a multiple of 2^-1074, and the transform's own error
    bound = 2.0 ** -1074 + np.ldexp(np.abs(np.ldexp(small, 1000)).max() * 2.0 ** -48, -1000)
    assert np.abs(got - want).max() <= bound and np.abs(want).max() > 0
    spec = np.ldexp(x[:, :1], power)
    h = np.ldexp(spec, 1000).transpose(0, 2, 1).repeat(nt // 2 + 1, 2)
    phi = np.ldexp(np.fft.irfft(h, n=nt, axis=2) * nt, -1000).transpose(0, 2, 1)
    assert np.abs(back - phi).max() <= 2.0 ** -1074 + np.ldexp(nt * np.abs(np.ldexp(spec, 1000)).max() * 2.0 ** -48, -1000)
