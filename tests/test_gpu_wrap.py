"""Wrapping and binning at the places where the reciprocal's product does not decide the floor: atoms
on box and cell faces and one ulp to either side, and atoms more than 2^20 boxes away.  The list of
the wrapped atoms must be the brute-force one (the oracle wraps by x - L floor(x / L))."""

import numpy as np
import pytest

from gpu_util import canonical_rows_gpu, canonical_rows_oracle, cuda_or_skip, dev_tensor
from oracle import neighbors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [9.0, 10.3, 17.77])
def test_faces_and_far_atoms(L):
    qg = cuda_or_skip()
    rng = np.random.default_rng(int(L * 100))
    n, r_list = 240, 3.1
    box = np.array([L, 1.1 * L, 0.9 * L])
    R = rng.uniform(0, 1, (n, 3)) * box
    k = rng.integers(-3, 4, (60, 3))
    R[:60] = k * (box / 6)  # on faces of the box and of cells
    R[20:40] = np.nextafter(R[20:40], np.inf)
    R[40:60] = np.nextafter(R[40:60], -np.inf)
    R[60:80, 0] += box[0] * rng.integers(2 ** 20, 2 ** 22, 20)
    s = qg.System(qg.make_params(n, box, r_cut=2.8, skin=0.3, mesh=(16, 16, 16)))
    s.neighbor_build(dev_tensor(R))
    rows = canonical_rows_gpu(*s.neighbor_export())
    assert rows == canonical_rows_oracle(*neighbors.brute_force_pairs(R, box, r_list))
    s.close()
