"""RAMBO's energy constraint from far above threshold down to it.

sum_f sqrt(m_f^2 + |k_f|^2) of the final three-momenta, formed in the host's
extended precision, is the collision energy to rounding at every energy.  In
units of u ecm, u = 2^-53: an energy as the constraint evaluates it carries
2.5 u of its value (two products and an addition under the root, half of them
through it, and the root), their sum another NF u, the root found and the
momenta's own rounding half a unit: (3 + NF) u.  A Newton iteration that ends at
rounding adds nothing.  The massless momenta that the constraint scales are
boosted with a factor gamma, which amplifies their rounding by gamma^2: 16 u
gamma^2 of the energy above threshold.
"""
import numpy as np
import pytest
import torch

from helpers import rambo_gamma
from paper_2106_12631_gb300 import inputs as I

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
NF = {2: 2, 3: 3, 4: 4}


def energy_defect(mom, ecm, mt):
    k = mom[2:].astype(np.longdouble)
    m = np.array([mt, mt] + [0.0] * (k.shape[0] - 2), dtype=np.longdouble)
    e = np.sqrt((k[:, 1:] ** 2).sum(axis=1) + m[:, None] ** 2).sum(axis=0)
    return np.abs(e - np.longdouble(ecm)) / ecm


def bar(rnd, nf, above, ecm):
    return U * (3 + nf + 16 * rambo_gamma(rnd, nf) ** 2 * above / ecm)


@pytest.mark.parametrize("proc", [2, 3, 4])
@pytest.mark.parametrize("above", [1154.0, 10.0, 0.1, 1e-3, 1e-5, 1e-6, 3e-7, 1e-7, 3e-8, 1e-8])  # GeV above 2 m_t
def test_energy_to_rounding(proc, above):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12631_gb300 import mg
    mt = I.SM_PARAMS["mt"]
    ecm = 2 * mt + above
    rnd = I.uniforms(500 + proc, 4 * NF[proc], 40001)
    mom, wgt = mg.rambo(proc, torch.from_numpy(rnd).cuda(), ecm)
    torch.cuda.synchronize()
    err = energy_defect(mom.cpu().numpy(), ecm, mt) / bar(rnd, NF[proc], above, ecm)
    assert err.max() <= 1, err.max()
    assert bool(torch.isfinite(wgt).all())


@pytest.mark.parametrize("scale", [1e-42, 1e42])
def test_energies_outside_fp32(scale):
    """The same process in units in which its energies leave FP32's range."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12631_gb300 import mg
    p = mg.get_params()
    rnd = torch.from_numpy(I.uniforms(600, 12, 1001)).cuda()
    try:
        mg.set_params(**dict(p, mt=p["mt"] * scale))
        mom, _ = mg.rambo(3, rnd, 1500.0 * scale)
    finally:
        mg.set_params(**p)
    torch.cuda.synchronize()
    err = energy_defect(mom.cpu().numpy() / scale, 1500.0, p["mt"]) / bar(rnd.cpu().numpy(), 3, 1154.0, 1500.0)
    assert err.max() <= 1, err.max()
