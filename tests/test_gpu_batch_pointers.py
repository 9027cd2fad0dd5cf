"""A batch plan run on other buffers than before (hmfsr_batch_run): every mode reads the bursts and
writes the outputs and motions of this call, also where a refused call came in between."""
import pytest
import torch

import burstgen
import paper_1905_03277_gb300 as hm

pytestmark = pytest.mark.gpu

SHAPES = [(4, 96, 128), (3, 64, 80), (5, 80, 64)]


def inputs(seed, dev):
    return [burstgen.make_burst(dict(n=n, h=h, w=w, gain=1.0, read=3.0, motion="global", scale=(1, 1)), seed=seed + k,
                                device=dev)["raw"] for k, (n, h, w) in enumerate(SHAPES)]


def buffers(plan, dev):
    rgbs = plan.outputs(dev)
    mvs = [torch.empty((n,) + hm.n_tiles(h, w, 16) + (2,), dtype=torch.float32, device=dev) for n, h, w in SHAPES]
    for t in rgbs + mvs:
        t.fill_(float("nan"))
    return rgbs, mvs


@pytest.fixture(scope="module")
def two():
    hm.build()
    dev = torch.device("cuda:0")
    out = []
    for seed in (310, 320):
        bursts = inputs(seed, dev)
        mvs = [hm.align(b) for b in bursts]
        out.append((bursts, mvs, [hm.merge(b, m, hm.MergeParams(noise_a=1.0, noise_b=9.0)) for b, m in zip(bursts, mvs)]))
    return dev, out


def check(got, want):
    for a, b in zip(got, want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("mode", [0, 1, 3])
def test_second_buffers(two, mode):
    dev, ((bursts, mvs, rgbs), (bursts2, mvs2, rgbs2)) = two
    plan = hm.BatchPlan(SHAPES, hm.MergeParams(noise_a=1.0, noise_b=9.0))
    plan.set_mode(mode)
    o, m = buffers(plan, dev)
    plan.run(bursts, o, m, wait=True)
    check(o + m, rgbs + mvs)
    o2, m2 = buffers(plan, dev)
    plan.run(bursts2, o2, m2, wait=True)
    check(o2 + m2, rgbs2 + mvs2)
    check(o + m, rgbs + mvs)  # the first call's outputs are left alone
    for t in o2:  # one pointer differs, a motion field's
        t.fill_(float("nan"))
    m3 = [m2[0], torch.full_like(m2[1], 7.0), m2[2]]
    plan.run(bursts2, o2, m3, wait=True)
    check(o2 + m3, rgbs2 + mvs2)


@pytest.mark.parametrize("mode", [0, 2])
def test_refused_call_between(two, mode):
    dev, ((bursts, mvs, rgbs), (bursts2, _, rgbs2)) = two
    plan = hm.BatchPlan(SHAPES, hm.MergeParams(noise_a=1.0, noise_b=9.0))
    plan.set_mode(mode)
    o, m = buffers(plan, dev)
    for _ in range(2):
        plan.run(bursts, o, m, wait=True)
    odd = torch.zeros(bursts[1].numel() + 1, dtype=bursts[1].dtype, device=dev)[1:].view(bursts[1].shape)
    with pytest.raises(RuntimeError, match="invalid argument"):  # 2-byte aligned
        plan.run([bursts2[0], odd, bursts[2]], o, m)
    plan.run([bursts2[0], bursts[1], bursts[2]], o, m, wait=True)
    check(o, [rgbs2[0], rgbs[1], rgbs[2]])
