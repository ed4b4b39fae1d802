"""The grouped emit of small systems: its list against brute force at row groups, cells and candidate
counts around its edges (one atom, 32 candidates, a cell of more rows than a group, bricks of one and
of two cells), and the regrowth of rows that do not fit."""

import numpy as np
import pytest

from gpu_util import canonical_rows_gpu, canonical_rows_oracle, cuda_or_skip, dev_tensor
from oracle import neighbors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,box,r_list,width", [
    (1, (5.0, 5.0, 5.0), 4.0, 0), (2, (9.0, 6.0, 7.0), 4.0, 0), (31, (8.0, 8.0, 8.0), 3.0, 0),
    (33, (7.9, 12.1, 8.3), 4.0, 0), (129, (9.0, 9.0, 9.0), 2.2, 16), (500, (10.0, 10.0, 10.0), 5.0, 0),
    (1500, (30.0, 11.0, 21.0), 4.5, 32), (4000, (36.0, 36.0, 36.0), 4.0, 0)])
def test_grouped_list_is_exact(n, box, r_list, width):
    qg = cuda_or_skip()
    rng = np.random.default_rng(n)
    box = np.array(box)
    R = rng.uniform(-0.3, 1.3, (n, 3)) * box
    R[: n // 3] = R[0] + 0.3 * rng.standard_normal((n // 3, 3))  # a crowded cell
    s = qg.System(qg.make_params(n, box, r_cut=r_list - 0.3, skin=0.3, mesh=(16, 16, 16), max_neighbors=width))
    s.neighbor_build(dev_tensor(R))
    rows = canonical_rows_gpu(*s.neighbor_export())
    assert rows == canonical_rows_oracle(*neighbors.brute_force_pairs(R, box, r_list))
    s.close()


def test_skin_wider_than_the_near_class():
    """r_list^2 / 3 > r_cut^2: the near radius lies beyond the cutoff."""
    qg = cuda_or_skip()
    rng = np.random.default_rng(5)
    box = np.array([11.0, 12.0, 13.0])
    R = rng.uniform(0, 1, (900, 3)) * box
    s = qg.System(qg.make_params(900, box, r_cut=1.8, skin=1.9, mesh=(16, 16, 16)))
    s.neighbor_build(dev_tensor(R))
    rows = canonical_rows_gpu(*s.neighbor_export())
    assert rows == canonical_rows_oracle(*neighbors.brute_force_pairs(R, box, 3.7))
    s.close()
