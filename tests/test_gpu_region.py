"""The accumulation's block-per-region kernel (scales 1, 3/2 and 2, tiles of 16 px and more)
against the oracle at its edges: frames smaller than a region and ragged against it, the extra
first region of scales above 1, more frames than its ring of constants holds, windows and texels
outside the frame, scales given in other than lowest terms, and the 8-px tiles it leaves to the
per-pixel kernels.  The bars are the merge's own: 1e-4 WL per pixel, 1e-6 WL in the mean."""
import numpy as np
import pytest
import torch

import burstgen
import oracle
import paper_1905_03277_gb300 as hm
from _parity import assert_merge_close, oparams

pytestmark = pytest.mark.gpu

CASES = [  # (n, h, w, scale, tile, ref, motion spread in px)
    (1, 4, 6, (2, 1), 16, 0, 0.0),
    (2, 6, 4, (3, 2), 16, 1, 1.5),
    (3, 18, 34, (1, 1), 16, 0, 3.0),
    (3, 16, 48, (2, 1), 16, 2, 40.0),
    (4, 50, 30, (3, 2), 32, 1, 9.0),
    (17, 34, 50, (2, 1), 16, 16, 2.0),
    (35, 20, 36, (1, 1), 64, 7, 2.0),
    (26, 36, 20, (3, 2), 16, 0, 6.0),
    (3, 40, 56, (4, 2), 16, 0, 2.0),
    (3, 40, 56, (6, 4), 32, 1, 2.0),
    (3, 40, 56, (2, 2), 16, 2, 2.0),
    (3, 40, 56, (3, 2), 8, 0, 4.0),
    (3, 40, 56, (2, 1), 8, 1, 4.0),
    (3, 40, 56, (1, 1), 8, 1, 4.0),
    (3, 40, 56, (4, 3), 16, 1, 4.0),
]


@pytest.mark.parametrize("case", CASES, ids=str)
def test_region_edges_match_oracle(case):
    n, h, w, scale, tile, ref, spread = case
    hm.build()
    dev = torch.device("cuda:0")
    raw = burstgen.make_burst(dict(n=n, h=h, w=w, gain=1.0, read=3.0, motion="global", scale=(1, 1)), seed=17)["raw"]
    rng = np.random.default_rng(n * 1000 + h)
    ty, tx = hm.n_tiles(h, w, tile)
    mv = (rng.normal(size=(n, ty, tx, 2)) * spread).astype(np.float32)
    mv[:, 0, 0] = np.round(mv[:, 0, 0] * 4) / 4  # window centres and texel cells on their boundaries
    mv[ref] = 0
    p = hm.MergeParams(noise_a=1.0, noise_b=9.0, tile=tile, t=-0.3)  # R >= 0.3: every frame counts
    rgb, den = hm.merge(raw.to(dev), torch.from_numpy(mv).to(dev), p, scale, ref, with_den=True)
    want = oracle.merge(raw.numpy(), mv, oparams(p), scale=scale, ref=ref, tile=tile)
    assert_merge_close(rgb.cpu().numpy(), want)
    assert torch.isfinite(den).all()
    for chunk in (1, 3):
        got, gden = hm.merge_chunked(raw.to(dev), torch.from_numpy(mv).to(dev), p, scale, ref, chunk_frames=chunk,
                                     with_den=True)
        assert torch.equal(got, rgb) and torch.equal(gden, den)
