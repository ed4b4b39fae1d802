"""The built-in flexible-water term on the device against the oracle, at the list shapes its
warp-per-row kernel can get wrong: one molecule (no O-O pair but its images), a box smaller than
the cutoff, rows of several queue fills, and a brick grid larger than the launch.

F_short is the difference of the shadow forces with and without the term: both carry the same
Coulomb forces (FP64, of a few eV/A), so the difference is good to about 1e-13 of the largest
force and 1e-10 of the largest short-range force is the bound."""

import numpy as np
import pytest

from gpu_util import cuda_or_skip, dev_tensor
from oracle import short_range
from workloads import water_box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_mol,r_cut,skin", [(1, 1.2, 0.2), (9, 4.0, 0.5), (64, 9.0, 1.0), (216, 9.0, 1.0),
                                              (1001, 6.0, 0.5), (1728, 5.0, 0.3)])
def test_water_term_matches_oracle(n_mol, r_cut, skin):
    qg = cuda_or_skip()
    w = water_box(n_mol, seed=100 + n_mol)
    t = dev_tensor
    rng = np.random.default_rng(n_mol)
    R = w.R + 0.03 * rng.standard_normal(w.R.shape)  # off the rigid geometry
    n0 = t(0.05 * rng.standard_normal(w.n_atoms))
    got = {}
    for model in (qg.QEQ_SHORT_NONE, qg.QEQ_SHORT_WATER):
        s = qg.System(qg.make_params(w.n_atoms, w.box, r_cut=r_cut, skin=skin, mesh=(16, 16, 16),
                                     short_range=model))
        md = qg.ShadowMD(s, t(w.chi), t(w.eta), t(w.sigma), t(w.mass), t(R), t(np.zeros_like(R)), n0)
        md.init()
        got[model] = (md.F.cpu().numpy(), md.energy_dict()["short"])
        s.close()
    e, F = short_range.water_short_range(R, w.box, r_cut)
    dF = got[qg.QEQ_SHORT_WATER][0] - got[qg.QEQ_SHORT_NONE][0]
    assert np.abs(dF - F).max() <= 1e-10 * np.abs(F).max()
    assert abs(got[qg.QEQ_SHORT_WATER][1] - e) <= 1e-10 * max(abs(e), 1.0)
