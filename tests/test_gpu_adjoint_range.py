"""A tile's motion gradient whose sum leaves FP32's range is infinite: the sums carry each addition's
rounding error along, and infinity less itself would make the error, and with it the sum, no number."""
import numpy as np
import pytest
import torch

import oracle
import paper_1905_03277_gb300 as hm
from test_gpu_adjoint import oparams

pytestmark = pytest.mark.gpu

# (scale, tile, parts of the tile's sum that leave the range each: a phase's in the region kernels, a column's in
# the per-pixel ones)
CASES = [((1, 1), 16, 4), ((3, 2), 16, 9), ((2, 1), 16, 16), ((4, 3), 64, 21)]


@pytest.mark.parametrize("case", CASES, ids=str)
def test_sum_beyond_the_range_is_infinite(case):
    """Every pixel's contribution is finite and of one sign, their sum is not: a ramp along x, gradients
    near the end of FP32's range."""
    scale, tile, parts = case
    hm.build()
    dev = torch.device("cuda:0")
    n, h, w = 2, 128, 128
    raw = np.broadcast_to(np.minimum(4 + 40 * np.arange(w), 4095).astype(np.uint16), (n, h, w)).copy()
    ty, tx = hm.n_tiles(h, w, tile)
    mv = np.zeros((n, ty, tx, 2), np.float32)
    mv[1] = (0.45, 0.02)
    p = hm.MergeParams(k_detail=0.5, k_denoise=1.0, d_th=1.0, d_tr=0.5, k_stretch=1.0, k_shrink=1.0, t=0.1, s1=50.0, s2=50.0,
                       m_th=3.0, noise_a=50.0, noise_b=4000.0, tile=tile)
    g = np.zeros((3,) + hm.out_size(h, w, scale), np.float32)
    g[:, :tile * scale[0] // scale[1], :16 * scale[0] // scale[1]] = 2.5e38 / raw[0, 0, 17]  # times any value in reach: finite
    burst, motion = torch.from_numpy(raw).to(dev), torch.from_numpy(mv).to(dev)
    rgb, den = hm.merge(burst, motion, p, scale, with_den=True)
    _, gm = hm.merge_backward(burst, motion, p, rgb, den, torch.from_numpy(g).to(dev), scale)
    _, want = oracle.merge_backward(raw, mv, oparams(p), g, scale=scale, tile=tile)
    assert want[1, 0, 0, 0] / parts > 2 * float(np.finfo(np.float32).max)
    got = gm.cpu().numpy()[1, 0, 0]
    assert got[0] == np.inf and not np.isnan(got[1])
