"""The sums behind a tile's motion gradient carry the rounding errors of their additions.  Scene and
frames repeat exactly, so two pixels a period apart contribute the same numbers; with gradients +1 and
-1 they cancel, and what is left is a third pixel's, 2^-24 of them: a sum that rounds it away is off by
all of it.  Against the FP64 oracle at the adjoint's bar, 1e-3 relative."""
import numpy as np
import pytest
import torch

import oracle
import paper_1905_03277_gb300 as hm
from test_gpu_adjoint import oparams

pytestmark = pytest.mark.gpu

# The +1, the -1 and the 2^-24 pixel, by half-res pixel of an inner tile.  R clamped at 1 leaves the
# pixels' own path, in which a thread takes (u, 0) and (u, 1).  Where R is open too, the texels that
# the first and the last reach (3 away at most) are other ones, of one 8 x 8 block's columns or rows.
PLACES = {
    "clamped": (16, 8, [(1, 0), (5, 0), (1, 1)]),
    "open, one row": (32, 16, [(1, 3), (1, 11), (7, 3)]),
    "open, one column": (32, 16, [(3, 1), (11, 1), (3, 7)]),
}
CASES = [(scale, place) for place in PLACES for scale in ((1, 1), (3, 2), (2, 1))]


def periodic_burst(seed, h, w, period):
    rng = np.random.default_rng(seed)
    cell = 1200 + rng.integers(-300, 300, size=(period, period))
    raw = np.stack([np.tile(cell + rng.integers(-12, 13, size=cell.shape), (h // period, w // period)) for _ in range(2)])
    return raw.astype(np.uint16)


@pytest.mark.parametrize("case", CASES, ids=str)
def test_small_contribution_beside_cancelling_ones(case):
    scale, place = case
    tile, period, at = PLACES[place]
    hm.build()
    dev = torch.device("cuda:0")
    h = w = 4 * max(tile, 32)
    raw = periodic_burst(3, h, w, period)
    ty, tx = hm.n_tiles(h, w, tile)
    mv = np.zeros((2, ty, tx, 2), np.float32)
    mv[1] = (0.40, -0.30)
    s = 12.0 if place == "clamped" else 0.8
    p = hm.MergeParams(k_detail=0.5, k_denoise=2.0, d_th=0.01, d_tr=0.1, k_stretch=2.0, k_shrink=1.5, t=0.1, s1=s, s2=s,
                       m_th=3.0, noise_a=4.0, noise_b=25.0, tile=tile)
    S, first = 2 * scale[0] // scale[1], 0 if scale == (1, 1) else 1  # output pixels of a half-res pixel, the first one
    g = np.zeros((3,) + hm.out_size(h, w, scale), np.float32)
    for (u, v), value in zip(at, (1.0, -1.0, 2.0 ** -24)):
        g[:, S * (ty // 2 * tile // 2 + v) + first, S * (tx // 2 * tile // 2 + u) + first] = value
    burst, motion = torch.from_numpy(raw).to(dev), torch.from_numpy(mv).to(dev)
    rgb, den = hm.merge(burst, motion, p, scale, 0, with_den=True)
    _, gm = hm.merge_backward(burst, motion, p, rgb, den, torch.from_numpy(g).to(dev), scale, 0)
    _, want = oracle.merge_backward(raw, mv, oparams(p), g, scale=scale, ref=0, tile=tile)
    got, want = gm.cpu().numpy().astype(np.float64)[1, ty // 2, tx // 2], want[1, ty // 2, tx // 2]
    assert np.all(np.abs(want) > 0)
    assert got == pytest.approx(want, rel=1e-3)
