"""The merge's outputs are the quotients of its running sums, correctly rounded, down to the smallest
sums: a channel whose only near samples come from a frame that robustness leaves a weight of 2^-118 and
less.  The sums are those that a bounded-memory merge keeps in its workspace before a last chunk that
adds nothing."""
import ctypes

import numpy as np
import pytest
import torch

import paper_1905_03277_gb300 as hm
from paper_1905_03277_gb300 import _lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [(1, 1), (3, 2), (2, 1)])
def test_outputs_are_the_sums_quotients(scale):
    tile = 16
    hm.build()
    L, dev = _lib.load(), torch.device("cuda:0")
    n, h, w = 3, 256, 320
    rng = np.random.default_rng(1)
    raw = np.full((n, h, w), 1000, np.int64)
    raw[1] += 34 + rng.integers(-3, 4, size=(h, w))  # R = exp(-3 x 34^2 / 40), t = 0
    raw[2] += 2500                                   # rejected
    raw = torch.from_numpy(raw.astype(np.uint16)).to(dev)
    ty, tx = hm.n_tiles(h, w, tile)
    mv = np.zeros((n, ty, tx, 2), np.float32)
    mv[1] = 1 + rng.uniform(-0.45, 0.45, size=(ty, tx, 2))  # an odd shift: its samples of a channel fall between the base's
    mv = torch.from_numpy(mv).to(dev)
    p = hm.MergeParams(k_detail=0.1, k_denoise=1.0, d_th=1.0, d_tr=1.0, k_stretch=1.0, k_shrink=1.0, t=0.0, s1=1.0, s2=1.0,
                       m_th=3.0, noise_a=0.0, noise_b=16.0, tile=tile)
    d, pc = _lib.BurstDesc(n, h, w, w, 0, 0, 4095, 0), p.c()
    nbytes = L.hmfsr_merge_chunked_workspace_size(ctypes.byref(d), tile, scale[0], scale[1], 1)
    buf = torch.zeros(nbytes + 256, dtype=torch.uint8, device=dev)
    ws = buf[(-buf.data_ptr()) % 256:][:nbytes]
    ho, wo = hm.out_size(h, w, scale)
    rgb = torch.empty((3, ho, wo), dtype=torch.float32, device=dev)
    _lib.check(L.hmfsr_merge_chunked(raw.data_ptr(), ctypes.byref(d), mv.data_ptr(), ctypes.byref(pc), scale[0], scale[1], 1,
                                     rgb.data_ptr(), None, ws.data_ptr(), nbytes,
                                     torch.cuda.current_stream().cuda_stream), "hmfsr_merge_chunked")
    size = 9 * ho * wo * 4  # the workspace ends with the sums: numerators, denominators, shifts
    sums = ws[nbytes - -(-size // 256) * 256:][:size].view(torch.float32).view(9, ho, wo).cpu().numpy()
    want = sums[0:3] / sums[3:6]
    assert sums[3:6].min() < 2.0 ** -100 and np.isfinite(want).all()
    assert np.array_equal(rgb.cpu().numpy(), want)
    assert torch.equal(hm.merge(raw, mv, p, scale), rgb)
