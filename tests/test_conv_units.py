"""The convolutions' work units: volumes whose tiles, planes and stages end raggedly in each
way the launches choose between (units of one tile and of many, odd and even; columns of 1 to
16 planes; rings of 2 to 6 stages), against the FP64 oracle within the bound of
tests/test_denoiser.py (one BF16 rounding and the FP32 accumulation).  Each runs several
times: a stage read before or after its time shows as a difference between runs."""
import numpy as np
import pytest

from oracle import denoiser as od

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_1711_03244_gb300 import build
    build.build()
    import paper_1711_03244_gb300 as m
    m.load()
    return m


# (n, d, h, w): 16 and 32 wide, the denoiser's coarse levels; 64 wide, where the ring of the
# widest layer has two stages
@pytest.mark.parametrize("shape", [(1, 5, 7, 16), (2, 9, 11, 32), (2, 18, 22, 64), (3, 16, 16, 32), (1, 1, 3, 48)])
@pytest.mark.parametrize("cin,cout", [(96, 32), (32, 96), (64, 64), (32, 64), (64, 32), (32, 32), (16, 48), (48, 16)])
def test_conv_units_match_oracle(g, cin, cout, shape):
    import torch
    rng = np.random.default_rng(700 + cin + 3 * cout + shape[-1])
    x = od.bf16_round(torch.as_tensor(rng.normal(size=shape + (cin,)))).numpy()
    w = od.bf16_round(torch.as_tensor(rng.normal(size=(27, cout, cin)) / np.sqrt(27 * cin))).numpy()
    b = rng.normal(size=cout).astype(np.float32)
    got = [g.mcx_debug_conv3d(0, x, w, b) for _ in range(4)]
    for r in got[1:]:
        assert np.array_equal(r, got[0])
    xt, wt = torch.tensor(x), torch.tensor(w)
    ref = np.maximum(od.conv3d(xt, wt, torch.tensor(b, dtype=torch.float64)).numpy(), 0)
    s_abs = od.conv3d(xt.abs(), wt.abs()).numpy() + np.abs(b)
    bound = 2.0 ** -8 * np.abs(ref) + 1.01 * 27 * cin * 2.0 ** -22 * s_abs
    assert np.all(np.abs(got[0].astype(np.float64) - ref) <= bound)
