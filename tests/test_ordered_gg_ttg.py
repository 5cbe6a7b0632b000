"""The ordered program of g g -> t t~ g: its tables, and helicity subsets whose
groups leave lanes and events of a CTA idle, against the oracle's partial
helicity sums (bars as for g g -> t t~ g g: relative to the full sum, whose
amplitudes a subset's rounding is the size of)."""
import numpy as np
import pytest
import torch

from helpers import FP64_CAP, MIXED_MAX_REL, MIXED_MEDIAN_REL, oracle_conditioning
from paper_2106_12631_gb300 import inputs as I
from paper_2106_12631_gb300.gen import procgen


def test_items_write_each_slot_once_and_read_inside():
    proc = procgen.Process(procgen.PROCS[3])
    em = procgen.Emitter(proc)
    for leg in range(proc.n):
        em.momentum_phys(leg)
    em.emit()
    sp = procgen.program(proc, em)
    sp.emit_tables(3)
    cur, x, sc = [], [], []
    for t, a, b, c, flag, out, ins, k0, k1, pr in sp.levels[0] + sp.levels[1] + sp.xitems:
        two = t in (sp.T_ROW2, sp.T_COL2, sp.T_G3)
        (sc if t == sp.T_DOT else cur if t < sp.T_ROW2 else x).append(out)
        if two:
            x.append(out + 8)
        if t < 3:
            continue
        in3 = (a & 255) | (b & 255) << 8
        reads = list(ins[:3] if two else ins[:2])
        if two:
            reads += sp.ext[in3][0]
        elif t == sp.T_VB:
            reads += [ins[2], in3]
        assert all(0 <= r < sp.nslots for r in reads)
        assert k0 < len(em.mom) and k1 < len(em.mom) and pr < len(em.props)
    assert sorted(cur) == list(range(sp.nslots))
    assert sorted(x) == list(range(sp.xcap))
    assert sorted(sc) == list(range(sp.nsc))


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["fp64", "mixed"])
@pytest.mark.parametrize("ng,nevt", [(1, 7), (3, 1), (5, 2501), (19, 613), (31, 9)])
def test_helicity_subsets(orc, ng, nevt, mode):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12631_gb300 import mg
    mom, _ = orc.rambo(3, I.uniforms(700 + ng, 12, nevt), 1500.0)
    me_o, ph = orc.me(3, mom, per_helicity=True, nthreads=16)
    _, d_rot = oracle_conditioning(orc, 3, mom, nthreads=16)
    mask = np.zeros(32, np.int32)
    mask[np.random.default_rng(ng).permutation(32)[:ng]] = 1
    want = ph[mask == 1].sum(axis=0)
    got = mg.sigmakin(3, torch.from_numpy(mom).cuda(), torch.from_numpy(mask).cuda(), mode=mode)
    torch.cuda.synchronize()
    err = np.abs(got.cpu().numpy() - want)
    if mode == "fp64":
        # d_rot, from two rotations, may underestimate an event's conditioning:
        # all but one event in 500 within 4 d_rot, every one within the cap
        tol = np.minimum(np.maximum(1e-12, 4 * d_rot), FP64_CAP)
        assert np.mean(err > tol * me_o) <= 1 / 500 and np.all(err <= FP64_CAP * me_o)
    else:
        assert np.all(err <= MIXED_MAX_REL * me_o) and np.median(err / me_o) <= MIXED_MEDIAN_REL
