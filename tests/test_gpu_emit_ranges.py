"""The brick search of large systems against the per-atom search: the same pairs in every row, for
sparse boxes (many short and empty ranges), crowded cells and a box two cells wide."""

import numpy as np
import pytest

from gpu_util import cuda_or_skip, dev_tensor

pytestmark = pytest.mark.gpu


def _rows(s):
    counts, nbr, shift = (np.asarray(a) for a in s.neighbor_export())
    key = np.full(nbr.shape, -1, dtype=np.int64)
    live = np.arange(nbr.shape[1])[None, :] < counts[:, None]
    code = ((shift[..., 0].astype(np.int64) + 2) * 5 + shift[..., 1] + 2) * 5 + shift[..., 2] + 2
    key[live] = (nbr.astype(np.int64) * 125 + code)[live]
    return counts, [np.sort(k[:c]) for k, c in zip(key, counts)]


@pytest.mark.parametrize("box,r_list,crowd", [
    ((60.0, 60.0, 60.0), 3.0, 0), ((150.0, 150.0, 150.0), 5.0, 0), ((80.0, 80.0, 80.0), 4.0, 300),
    ((400.0, 40.0, 9.0), 4.4, 0)])
def test_large_lists_agree_with_the_atom_search(box, r_list, crowd):
    qg = cuda_or_skip()
    n = 50_000  # above the sizes of the grouped form
    rng = np.random.default_rng(n + crowd)
    box = np.array(box)
    R = rng.uniform(-0.2, 1.2, (n, 3)) * box
    R[:crowd] = R[0] + 0.5 * rng.standard_normal((crowd, 3))
    got = []
    for method in ("brick", "atom"):
        s = qg.System(qg.make_params(n, box, r_cut=r_list - 0.4, skin=0.4, mesh=(16, 16, 16)))
        qg.qeq_set_neighbor_method(s.ctx, method)
        s.neighbor_build(dev_tensor(R))
        got.append(_rows(s))
        s.close()
    assert np.array_equal(got[0][0], got[1][0])
    assert all(np.array_equal(a, b) for a, b in zip(got[0][1], got[1][1]))
