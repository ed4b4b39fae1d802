"""One GMRES cycle of k iterations against the least-squares minimum over the same Krylov space, with
the matrix written out: k at and beside the eight vectors that a pass of dot products takes, at
vector lengths (atoms + 1) on and past a block.  The residual reported is that of the final iterate."""

import numpy as np
import pytest

from gpu_util import cuda_or_skip, dev_tensor
from oracle import ewald
from workloads import water_box

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
MESH, RC, ALPHA = (24, 24, 24), 6.0, 0.34


@pytest.mark.parametrize("molecules", [40, 85, 86])
def test_cycle_minimises_over_its_krylov_space(molecules):
    qg = cuda_or_skip()
    w = water_box(molecules, seed=molecules)
    n = w.n_atoms
    A = np.zeros((n + 1, n + 1))
    A[:n, :n] = ewald.phi_matrix(w.R, w.sigma, w.box, ALPHA, RC, recip="pme", mesh=MESH, order=4,
                                 gaussian_self=True) + np.diag(w.eta)
    A[:n, n] = A[n, :n] = 1.0
    b = np.append(-w.chi, 0.0)
    M = np.append(w.eta + ewald.K_E * np.sqrt(2 / np.pi) / w.sigma, 1.0)
    s = qg.System(qg.make_params(n, w.box, alpha=ALPHA, r_cut=RC, skin=0.5, mesh=MESH, order=4))
    s.neighbor_build(dev_tensor(w.R))
    V = [b / np.linalg.norm(b)]
    for k in range(1, 18):
        x = A @ (V[-1] / M)
        for _ in range(2):
            x = x - np.array(V).T @ (np.array(V) @ x)
        V.append(x / np.linalg.norm(x))
        if k not in (1, 7, 8, 9, 15, 16, 17):
            continue
        AV = A @ (np.array(V[:k]) / M).T
        y = np.linalg.lstsq(AV, b, rcond=None)[0]
        ref = np.linalg.norm(b - AV @ y) / np.linalg.norm(b)
        q = torch.zeros(n, dtype=torch.float64, device="cuda")
        info = qg.qeq_solve(s.ctx, dev_tensor(w.R), dev_tensor(w.chi), dev_tensor(w.eta),
                            dev_tensor(w.sigma), q, tol=1e-15, restart=k, max_iter=k)
        assert info["iterations"] == k
        # the applies agree with the written-out matrix to better than 1e-9
        assert abs(info["rel_residual"] - ref) < 1e-9 + 1e-6 * ref, (k, info["rel_residual"], ref)
    s.close()
