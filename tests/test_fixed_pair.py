"""The fixed-point pair functions of the FP64 real-space kernel, on the host (the same source as on
the device) against mpmath: every octave, cutoffs that scale lengths up and down, close pairs, wide
and narrow charges, and the pairs that are left to the exact path.

Bounds, in lengths scaled so that r_cut' is in (4, 8]: each of erfc(a r) / r and its correction is
good to 2^-51 of the bare 1 / r' (squared distance to 3 units of 2^-54, reciprocal widths to 2^-51)
plus 2^-53 of fixed-point truncation, so f is within 2^-50 / r' + 2^-52 and gc r within
2^-49 / r'^2 + 2^-52."""

import math

import numpy as np
import pytest

import paper_2503_21176_gb300 as qg
from paper_2503_21176_gb300 import _lib

mp = pytest.importorskip("mpmath")


def _reference(alpha, d, si, sj):
    mp.mp.dps = 40
    r = mp.sqrt(sum(mp.mpf(float(x)) ** 2 for x in d))
    g = mp.sqrt(mp.mpf(float(si)) ** 2 + mp.mpf(float(sj)) ** 2)
    f, df = mp.mpf(0), mp.mpf(0)
    for a, sign in ((mp.mpf(alpha), 1), (1 / g if g > 0 else None, -1)):
        if a is None:
            continue
        e = mp.erfc(a * r) / r
        f += sign * e
        df -= sign * (e + 2 * a / mp.sqrt(mp.pi) * mp.exp(-(a * r) ** 2)) / r
    return f, df / r, r


@pytest.mark.parametrize("alpha,r_cut,sigmas", [
    (0.34, 8.0, (0.45, 0.70)), (0.34, 9.0, (0.45, 0.70)), (0.30, 7.3, (0.3, 1.5)), (0.5, 4.0, (0.0, 0.4)),
    (0.25, 12.0, (0.05, 2.5)), (3.4, 0.8, (0.045, 0.07)), (0.9, 3.0, (0.0, 0.0))])
def test_fixed_pairs_match_mpmath(alpha, r_cut, sigmas):
    e = math.ceil(math.log2(r_cut / 8.0) - 1e-12)
    lam = 2.0 ** e
    rng = np.random.default_rng(int(100 * r_cut))
    n = 700
    u = rng.standard_normal((n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    r = np.exp(rng.uniform(math.log(0.36 * lam), math.log(r_cut), n))
    d = u * r[:, None]
    d[:30, 1:] = 0.0  # along an axis
    r = np.linalg.norm(d, axis=1)
    si = rng.uniform(*sigmas, n)
    sj = rng.uniform(*sigmas, n)
    f, gc, path = _lib.qeq_fixed_pair_eval(alpha, r_cut, d, si, sj)
    gamma = np.hypot(si, sj)
    far = (r > 0.51 * gamma) & (r > 0.36 * lam)  # the tables' ranges
    assert (path[far & (r < 0.9999 * r_cut)] == 1).all()
    for k in np.nonzero(path == 1)[0]:
        rf, rg, rr = _reference(alpha, d[k], si[k], sj[k])
        rp = float(rr) / lam
        assert abs(float(mp.mpf(f[k]) - rf)) * lam <= 2.0 ** -50 / rp + 2.0 ** -52
        assert abs(float((mp.mpf(gc[k]) - rg) * rr)) * lam ** 2 <= 2.0 ** -49 / rp ** 2 + 2.0 ** -52


def test_paths_at_the_edges():
    """Exact path nearer than the tables reach, at the cutoff, and for very wide charges; none beyond."""
    r = np.array([1e-9, 0.2, 0.35, 0.36, 3.0, 7.99, 8.0 - 1e-9, 8.0, 8.0 + 1e-9, 8.01, 15.0])
    d = np.stack([r, 0 * r, 0 * r], axis=1)
    _, _, path = _lib.qeq_fixed_pair_eval(0.34, 8.0, d, 0.0, 0.0)
    assert path.tolist() == [0, 0, 0, 1, 1, 1, 0, 0, 0, -1, -1]
    _, _, path = _lib.qeq_fixed_pair_eval(0.34, 8.0, d[3:6], [9.0, 9.0, np.inf], 0.0)
    assert path.tolist() == [0, 0, 0]
    _, _, path = _lib.qeq_fixed_pair_eval(0.34, 8.0, d[3:6], np.nan, 0.5)
    assert path.tolist() == [1, 1, 1]
    with pytest.raises(qg.QeqError):
        _lib.qeq_fixed_pair_eval(-1.0, 8.0, d, 0.0, 0.0)
