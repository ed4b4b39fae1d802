"""Applies from kept pair values (every iteration of a solve after the first) against the operator
itself: the residual of the solved charges, formed with the public apply, which computes its pairs,
must be what the solve reports.  Boxes that the tile repeats, rows that end inside a stripe, pairs of
the exact path and of the correction queue, and a single atom.

FP64: both operators are good to 1e-14 of the terms, so the two residuals differ by less than 1e-12 of
|chi|.  FP32-mixed: the same pair values and order, other operators within 1e-5 (the mode's bound)."""

import numpy as np
import pytest

from gpu_util import cuda_or_skip, dev_tensor
from workloads import water_box

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,tol,slack", [("fp64", 1e-11, 1e-12), ("fp32_mixed", 1e-5, 1e-5)])
@pytest.mark.parametrize("kind,n_mol,r_cut", [("water", 1, 2.2), ("water", 33, 6.0), ("water", 216, 9.0),
                                              ("water", 1500, 5.5), ("uniform", 150, 5.0), ("wide", 100, 7.0)])
def test_solve_residual(precision, tol, slack, kind, n_mol, r_cut):
    qg = cuda_or_skip()
    w = water_box(n_mol, seed=n_mol)
    R, sigma, box = w.R, w.sigma.copy(), w.box
    rng = np.random.default_rng(n_mol)
    if kind == "uniform":
        R = rng.uniform(0, 1, R.shape) * box
    if kind == "wide":
        sigma = rng.uniform(0.5, 3.5, w.n_atoms)
    eta = w.eta + 20.0  # a well conditioned system for any geometry
    s = qg.System(qg.make_params(w.n_atoms, box, r_cut=r_cut, skin=0.5, mesh=(24, 24, 24), precision=precision))
    t = dev_tensor
    Rd, sd = t(R), t(sigma)
    s.neighbor_build(Rd)
    q = torch.zeros(w.n_atoms, dtype=torch.float64, device="cuda")
    info = qg.qeq_solve(s.ctx, Rd, t(w.chi), t(eta), sd, q, tol)
    assert info["rel_residual"] <= 2 * tol
    v, _, _, _ = s.apply(Rd, q, sd)
    r = -w.chi - (eta * q.cpu().numpy() + v.cpu().numpy() + info["lambda"])
    assert np.linalg.norm(r) / np.linalg.norm(w.chi) <= info["rel_residual"] + slack
    s.close()
