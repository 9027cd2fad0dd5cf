"""The staged block matching (levels with many tiles) against the oracle: each tile size and radius
it serves, level rows that start on 16-byte boundaries and rows that do not, ragged last tiles, and
both sides of the white level up to which a row's squared differences fit 32 bits.  Vectors are
whole numbers and equal."""
import numpy as np
import pytest
import torch

import burstgen
import oracle
import paper_1905_03277_gb300 as hm

pytestmark = pytest.mark.gpu

CASES = [  # (n, h, w, tile, radius, white level)
    (14, 1090, 1290, 32, (1, 4, 4, 4), 4095),
    (13, 1088, 1344, 32, (1, 7, 2, 4), 4095),
    (13, 1090, 1290, 32, (1, 4, 3, 4), 5000),
    (12, 1250, 1302, 16, (1, 3, 2, 4), 4095),
    (11, 1280, 1344, 16, (1, 5, 4, 4), 4095),
    (11, 1282, 1402, 16, (1, 6, 4, 4), 6000),
    (12, 700, 740, 8, (1, 4, 2, 3), 4095),
]


@pytest.mark.parametrize("case", CASES, ids=str)
def test_staged_search_matches_oracle(case):
    n, h, w, tile, radius, wl = case
    hm.build()
    raw = burstgen.make_burst(dict(n=n, h=h, w=w, gain=1.0, read=3.0, motion="global", scale=(1, 1)), seed=41)["raw"]
    if wl > 4095:  # the whole of the range
        raw = (raw.to(torch.float32) * (wl / 4095.0)).to(torch.int32).to(raw.dtype)
    ap = hm.AlignParams(tile=tile, radius=radius)
    motion, vectors = hm.align(raw.to("cuda:0"), 0, ap, with_int=True, white_level=wl)
    want, _, _, _ = oracle.align(raw.numpy(), ref=0, tile=tile, radius=radius)
    assert np.array_equal(vectors.cpu().numpy(), want)
    assert torch.isfinite(motion).all()
