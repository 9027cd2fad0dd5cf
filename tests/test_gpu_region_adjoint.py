"""The adjoint's block-per-region kernels (scales 1, 3/2 and 2, tiles of 16 px and more) against the
FP64 oracle adjoint at their edges: frames smaller than a region and ragged against it, the extra
first region of scales above 1, more frames than the ring of constants holds, windows and texels
outside the frame, scales given in other than lowest terms, and the 8-px tiles and other scales
left to the per-pixel kernels.  The bars are the adjoint's own: 1e-3 relative."""
import numpy as np
import pytest
import torch

import burstgen
import oracle
import paper_1905_03277_gb300 as hm
from test_gpu_adjoint import assert_adjoint_close, oparams

pytestmark = pytest.mark.gpu

CASES = [  # (n, h, w, scale, tile, ref, motion spread in px)
    (2, 10, 6, (2, 1), 16, 0, 0.3),
    (2, 6, 14, (3, 2), 16, 1, 1.5),
    (3, 18, 34, (1, 1), 16, 0, 3.0),
    (3, 16, 48, (2, 1), 16, 2, 12.0),
    (4, 50, 30, (3, 2), 32, 1, 9.0),
    (18, 34, 50, (2, 1), 16, 17, 2.0),
    (19, 20, 36, (1, 1), 64, 7, 2.0),
    (17, 36, 20, (3, 2), 16, 0, 6.0),
    (3, 40, 56, (6, 4), 32, 1, 2.0),
    (3, 40, 56, (2, 2), 16, 2, 2.0),
    (3, 40, 56, (3, 2), 8, 0, 4.0),
    (3, 40, 56, (4, 3), 16, 1, 4.0),
]


@pytest.mark.parametrize("case", CASES, ids=str)
def test_region_adjoint_edges_match_oracle(case):
    n, h, w, scale, tile, ref, spread = case
    hm.build()
    dev = torch.device("cuda:0")
    raw = burstgen.make_burst(dict(n=n, h=h, w=w, gain=1.0, read=3.0, motion="global", scale=(1, 1)), seed=23)["raw"]
    rng = np.random.default_rng(n * 1000 + h)
    ty, tx = hm.n_tiles(h, w, tile)
    mv = (rng.normal(size=(n, ty, tx, 2)) * spread).astype(np.float32)
    mv[ref] = 0
    p = hm.MergeParams(k_detail=0.3, k_denoise=3.0, d_th=0.004, d_tr=0.05, k_stretch=3.0, k_shrink=1.8, t=0.12,
                       s1=12.0, s2=1.1, m_th=3.0, noise_a=0.02, noise_b=0.5, tile=tile)
    ho, wo = hm.out_size(h, w, scale)
    g = rng.normal(size=(3, ho, wo))
    burst, motion = raw.to(dev), torch.from_numpy(mv).to(dev)
    rgb, den = hm.merge(burst, motion, p, scale, ref, with_den=True)
    gp, gm = hm.merge_backward(burst, motion, p, rgb, den, torch.from_numpy(g).float().to(dev), scale, ref)
    ogp, ogm = oracle.merge_backward(raw.numpy(), mv, oparams(p), g, scale=scale, ref=ref, tile=tile)
    assert_adjoint_close(gp, gm, ogp, ogm, ref)
