"""The adjoint's robustness path at the boundary of rejection.  The forward finds R with the SFU's
exponential, the adjoint its derivative with expf, so R = s exp(-d) - t can be 0 in one and a last
place above 0 in the other.  Where the forward rejects a frame whose samples lie far nearer than those
that count, dL/dRhat has no bound; it must not reach s2, t or the motion as infinity or NaN."""
import numpy as np
import pytest
import torch

import paper_1905_03277_gb300 as hm

pytestmark = pytest.mark.gpu

THIN = dict(k_detail=0.1, k_denoise=1.0, d_th=1.0, d_tr=1.0, k_stretch=1.0, k_shrink=1.0, s1=1.5, s2=1.5, m_th=3.0,
            noise_a=0.0, noise_b=16.0)


def thresholds():
    """(flat difference between the frames, its thresholds t around s exp(-d), in steps of a last place)."""
    for delta in range(1, 20):
        # Eq. 5-6 for a flat difference: variances 16 (green 8), d_md^2 two ninths of them
        d = sum((delta ** 3 / (delta ** 2 + v * 2 / 9)) ** 2 for v in (16, 8, 16)) / 40
        t = np.float32(1.5 * np.exp(-d))
        if 1e-6 < t < 1:
            t = t * np.float32(1 - 64 * 2.0 ** -23)
            ts = []
            for _ in range(160):
                t = np.nextafter(t, np.float32(2))
                ts.append(float(t))
            yield delta, ts


@pytest.mark.parametrize("scale,tile", [((1, 1), 16), ((3, 2), 16), ((2, 1), 16), ((1, 1), 8), ((4, 3), 16)])
def test_rejection_boundary_stays_finite(scale, tile):
    hm.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(2)
    ty, tx = hm.n_tiles(64, 64, tile)
    mv = np.zeros((2, ty, tx, 2), np.float32)
    mv[1] = 1 + rng.uniform(-0.4, 0.4, size=(ty, tx, 2))
    mv = torch.from_numpy(mv).to(dev)
    rejected = 0
    for delta, ts in thresholds():
        raw = np.full((2, 64, 64), 1000, np.uint16)
        raw[1] += delta
        burst = torch.from_numpy(raw).to(dev)
        for t in ts:
            p = hm.MergeParams(t=t, tile=tile, **THIN)
            if (hm.merge_stages(burst, mv, p, 0)[1][1] > 0).any():
                continue
            rejected += 1
            rgb, den = hm.merge(burst, mv, p, scale, 0, with_den=True)
            assert float(den.min()) < -128  # the base frame's sums: a sample at the pixel weighs over 2^128 of them
            gp, gm = hm.merge_backward(burst, mv, p, rgb, den, torch.ones_like(rgb), scale, 0)
            assert torch.isfinite(gp).all() and torch.isfinite(gm).all(), (delta, t)
            assert (gp[6:] == 0).all() and (gm == 0).all(), (delta, t)  # nothing of a rejected frame
    assert rejected >= 100
