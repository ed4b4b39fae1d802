"""Shadow evaluations at atom counts around the blocks of the atom-wise reductions (256 atoms a
block, no more blocks than that needs), against the oracle: charges, kernel update and energies.
FP64, sums of at most a few hundred terms of one sign scale: 1e-10 relative."""

import numpy as np
import pytest

from gpu_util import cuda_or_skip, dev_tensor, rel_max
from oracle import ewald, qeq
from workloads import water_box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_mol,r_cut", [(1, 4.0), (85, 6.0), (86, 6.0), (171, 6.0)])
def test_evaluation_at_block_edges(n_mol, r_cut):
    qg = cuda_or_skip()
    w = water_box(n_mol, seed=n_mol)
    mesh = (16, 16, 16)
    n0 = 0.1 * np.random.default_rng(n_mol).standard_normal(w.n_atoms)
    V0 = 0.01 * np.random.default_rng(n_mol + 1).standard_normal(w.R.shape)
    s = qg.System(qg.make_params(w.n_atoms, w.box, r_cut=r_cut, skin=0.5, mesh=mesh, krylov_rank=2))
    t = dev_tensor
    md = qg.ShadowMD(s, t(w.chi), t(w.eta), t(w.sigma), t(w.mass), t(w.R), t(V0), t(n0))
    md.init()

    def coul(R, x, need_field=True):
        o = ewald.coulomb_apply(R, x, w.sigma, w.box, 0.34, r_cut, recip="pme", mesh=mesh, order=4,
                                gaussian_self=True)
        return o["v"], o["E"]

    st = qeq.ShadowSystem(coul, w.chi, w.eta, w.mass, rank=2, dt=0.5, k_d=5).init_state(w.R, V0, n0)
    e = md.energy_dict()
    assert rel_max(md.q.cpu().numpy(), st["q"]) < 1e-10
    assert rel_max(md.F.cpu().numpy(), st["F"]) < 1e-10
    assert np.abs(md.Kf.cpu().numpy() - st["Kf"]).max() < 1e-9 * np.abs(st["q"]).max()
    assert abs(e["kinetic"] - st["e_kin"]) < 1e-10 * st["e_kin"]
    assert abs(e["shadow_potential"] - st["e_pot"]) < 1e-10 * abs(st["e_pot"])
    s.close()
