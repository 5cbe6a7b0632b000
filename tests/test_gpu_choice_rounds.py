"""Helicity and flow choices where CTAs take full groups over several rounds.

The same events in batches that leave every CTA one unit, and in one batch of
several full rounds with an odd last event: the same matrix elements, helicities
and flows, bit for bit.  (A group's staged flow weights lie where the next
group's currents go, so a missing barrier would show here.)  The small batches
are compared with the oracle elsewhere.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

# several rounds of the CTAs that fit an SM, times 152 SMs, times events per group
CASES = [(1, 60001, 256), (2, 60001, 128), (3, 15001, 128), (4, 3751, 64)]


@pytest.mark.parametrize("mode", ["fp64", "mixed", "mixed_tc"])
@pytest.mark.parametrize("proc,nevt,small", CASES)
def test_choices_do_not_depend_on_the_batch(proc, nevt, small, mode):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12631_gb300 import mg
    mom, _ = mg.rambo_seeded(proc, nevt, 500.0 if proc == 1 else 1500.0, seed=311 + proc)
    mask = mg.filter_helicities(proc, mom[:, :, :16].contiguous())
    rec = mom.permute(2, 0, 1).contiguous()
    g = torch.Generator(device="cuda").manual_seed(proc)
    u, v = (torch.rand(nevt, dtype=torch.float64, device="cuda", generator=g) for _ in range(2))
    whole = mg.matrix_elements_batch(proc, rec, mask, mode=mode, hel_rnd=u, col_rnd=v)
    parts = [mg.matrix_elements_batch(proc, rec[i:i + small], mask, mode=mode, hel_rnd=u[i:i + small],
                                      col_rnd=v[i:i + small]) for i in range(0, nevt, small)]
    torch.cuda.synchronize()
    for k, name in enumerate(("me", "hel", "col")):
        assert torch.equal(whole[k], torch.cat([p[k] for p in parts])), name
    assert len(torch.unique(whole[1])) > 1 and (proc == 1 or len(torch.unique(whole[2])) > 1)
