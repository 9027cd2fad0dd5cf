"""The adjoint where a frame that robustness rejects (Rhat = 0) has samples far nearer than those
that count: its normalised weights and their products with Omega^-1 d leave FP32's range, and 0
times them is not a number.  The FP64 oracle, in whose range they are, gives it no part.  The bars
are the adjoint's own: 1e-3 relative."""
import numpy as np
import pytest
import torch

import oracle
import paper_1905_03277_gb300 as hm
from test_gpu_adjoint import assert_adjoint_close, oparams

pytestmark = pytest.mark.gpu

SHIFTS = [(0, 0), (2, 0), (-2, 2)]  # of the frames that count: whole Bayer periods
PARAMS = dict(k_detail=0.1, k_denoise=1.0, d_th=0.0, d_tr=1.0, k_stretch=1.2, k_shrink=1.1, t=0.12, s1=12.0, s2=2.0,
              m_th=3.0, noise_a=0.5, noise_b=9.0)
CASES = [  # (scale, tile)
    ((1, 1), 16),
    ((1, 1), 32),
    ((3, 2), 16),
    ((2, 1), 16),
    ((1, 1), 8),    # the per-pixel kernel
    ((4, 3), 16),
]


def rejected_burst(seed, h, w, tile):
    """Three frames of one scene at even shifts (so that a channel's samples are a px and more from most
    pixels) and a fourth, far brighter one at an odd shift and a fraction that differs from tile to tile
    (so that its samples of the same channels lie next to the pixels)."""
    rng = np.random.default_rng(seed)
    ph, pw = h + 32, w + 32
    y, x = np.mgrid[0:ph, 0:pw]
    scene = 900 + 250 * np.sin(0.55 * x + 0.21 * y) + 200 * np.sin(0.17 * x - 0.63 * y) + rng.normal(size=(ph, pw)) * 40
    scene = np.clip(np.round(scene), 50, 1900).astype(np.uint16)
    raw, (ty, tx) = np.empty((4, h, w), np.uint16), hm.n_tiles(h, w, tile)
    mv = np.zeros((4, ty, tx, 2), np.float32)
    for f, (dx, dy) in enumerate(SHIFTS):  # a sample at q lies on the base frame at q - v
        raw[f] = scene[16 - dy:16 - dy + h, 16 - dx:16 - dx + w]
        if f:
            mv[f] = np.array([dx, dy]) + rng.uniform(0.005, 0.02, size=(ty, tx, 2)) * rng.choice([-1, 1], size=(ty, tx, 2))
    raw[3] = scene[16:16 + h, 16:16 + w] + 2100
    mv[3] = 1 + rng.uniform(-0.5, 0.5, size=(ty, tx, 2))
    return raw, mv


@pytest.mark.parametrize("case", CASES, ids=str)
def test_rejected_near_samples_add_nothing(case):
    scale, tile = case
    hm.build()
    dev = torch.device("cuda:0")
    h, w = 80, 112
    raw, mv = rejected_burst(5, h, w, tile)
    p = hm.MergeParams(**PARAMS, tile=tile)
    c = oracle.merge(raw, mv, oparams(p), scale=scale, ref=0, tile=tile)
    g = ((c - c.mean(axis=(1, 2), keepdims=True)) / 100).astype(np.float32)  # no sum cancels: a bar on the kernels
    burst, motion = torch.from_numpy(raw).to(dev), torch.from_numpy(mv).to(dev)
    rgb, den = hm.merge(burst, motion, p, scale, 0, with_den=True)
    gp, gm = hm.merge_backward(burst, motion, p, rgb, den, torch.from_numpy(g).to(dev), scale, 0)
    ogp, ogm = oracle.merge_backward(raw, mv, oparams(p), g, scale=scale, ref=0, tile=tile)
    assert np.all(ogm[3] == 0) and np.abs(ogp[:6]).min() > 0
    assert_adjoint_close(gp, gm, ogp, ogm, 0)
