"""The ordered program of g g -> t t~ g g (currents summed per gluon ordering,
then contracted) and the block form of its colour sum.

* The colour matrix's blocks reproduce J^dagger C J exactly (integers).
* The generated items write every slot and scalar once and read inside their
  regions.
* Helicity subsets of sizes that leave lanes and events of a CTA idle, at
  event counts around whole groups, against the oracle's partial helicity
  sums: FP64 within the event's conditioning bar, mixed within the stated
  mixed bound.
"""
import numpy as np
import pytest
import torch

from helpers import MIXED_MAX_REL, MIXED_MEDIAN_REL, fp64_tol, oracle_conditioning
from paper_2106_12631_gb300 import inputs as I
from paper_2106_12631_gb300.gen import procgen


def ordered():
    proc = procgen.Process(procgen.PROCS[4])
    em = procgen.Emitter(proc)
    for leg in range(proc.n):
        em.momentum_phys(leg)
    em.emit()
    sp = procgen.program(proc, em)
    sp.emit_tables(4)
    return em, sp


def test_colour_blocks_are_the_colour_sum():
    em, _ = ordered()
    orbits, blocks = procgen.colour_blocks(em.perms, em.cnum)
    rng = np.random.default_rng(4)
    J = rng.integers(-9, 10, 24) + 1j * rng.integers(-9, 10, 24)
    want = (J.conj() @ em.cnum @ J).real
    got = 0
    for x, chi in enumerate(procgen.KLEIN_CHARACTERS):
        y = np.array([sum(chi[k] * J[o[k]] for k in range(4)) for o in orbits])
        got += (y.conj() @ np.array(blocks[x]) @ y).real
    assert got == 4 * want
    assert sorted(s for o in orbits for s in o) == list(range(24))


def test_items_write_each_slot_once_and_read_inside():
    _, sp = ordered()
    cur, x, sc = [], [], []
    for it in sp.levels[0] + sp.levels[1] + sp.xitems:
        t, a, b, c, flag, out, ins, k0, k1, pr = it
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
        assert k0 < len(sp.em.mom) and k1 < len(sp.em.mom) and pr < len(sp.em.props)
    assert sorted(cur) == list(range(sp.nslots))
    assert sorted(x) == list(range(sp.xcap))
    assert sorted(sc) == list(range(sp.nsc))


@pytest.mark.gpu
@pytest.mark.parametrize("ng,nevt,mode", [(ng, nevt, mode) for ng, nevt in ((1, 5), (3, 1), (37, 613), (63, 4))
                                          for mode in ("fp64", "mixed")] + [(64, 1217, "mixed")])
def test_helicity_subsets(orc, ng, nevt, mode):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12631_gb300 import mg
    mom, _ = orc.rambo(4, I.uniforms(900 + ng, 16, nevt), 1500.0)
    me_o, ph = orc.me(4, mom, per_helicity=True, nthreads=16)
    _, d_rot = oracle_conditioning(orc, 4, mom, nthreads=16)
    mask = np.zeros(64, np.int32)
    mask[np.random.default_rng(ng).permutation(64)[:ng]] = 1
    part = ph[mask == 1].sum(axis=0)
    want = part
    got = mg.sigmakin(4, torch.from_numpy(mom).cuda(), torch.from_numpy(mask).cuda(), mode=mode)
    torch.cuda.synchronize()
    err = np.abs(got.cpu().numpy() - want)
    # a subset's rounding is that of its own amplitudes, of the size of the full
    # sum's where the subset is small: the bars are relative to the full sum
    if mode == "fp64":
        assert np.all(err <= fp64_tol(d_rot) * me_o)
    else:
        assert np.all(err <= MIXED_MAX_REL * me_o) and np.median(err / me_o) <= MIXED_MEDIAN_REL


@pytest.mark.gpu
@pytest.mark.parametrize("proc,mode", [(p, m) for p in (1, 2, 3, 4) for m in ("fp64", "mixed")])
def test_batch_size_does_not_change_an_event(proc, mode):
    """How a batch is split into groups and pairs of events (one unit per CTA for
    the smallest, full groups over several rounds, an odd last event) changes no
    event's result: each batch equals the start of the largest one, bit for bit."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12631_gb300 import mg
    ecm = 500.0 if proc == 1 else 1500.0
    most = 20011 if proc < 3 else 2611
    mom, _ = mg.rambo_seeded(proc, most, ecm, seed=61 + proc)
    mask = mg.filter_helicities(proc, mom[:, :, :16].contiguous())
    want = mg.sigmakin(proc, mom, mask, mode=mode)
    for n in (1, 2, 3, 151, 152, 153, 303, 305, 607, 609, 1215, 1217, 2433, most - 1):
        got = mg.sigmakin(proc, mom[:, :, :n].contiguous(), mask, mode=mode)
        torch.cuda.synchronize()
        assert torch.equal(got, want[:n]), n


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 5000, 1 << 20, (1 << 20) + 1])
def test_unweight_block_counts(orc, n):
    """Unweighting with one block, a ragged last block, the most blocks that find
    maximum and offsets by themselves, and one more: the oracle's indices."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12631_gb300 import mg
    rng = np.random.default_rng(n)
    me, wgt = rng.exponential(size=n), rng.uniform(0.5, 1.5, n)
    u = I.uniforms(n + 7, 64, n)[63]
    idx, count = mg.unweight(torch.from_numpy(me).cuda(), torch.from_numpy(wgt).cuda(), seed=n + 7)
    torch.cuda.synchronize()
    want = np.asarray(orc.unweight(me, wgt, u))
    k = int(count.item())
    assert k == len(want)
    np.testing.assert_array_equal(idx[:k].cpu().numpy(), want)
