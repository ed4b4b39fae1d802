"""The FP64 apply at the inputs its fixed-point real space has to scale, hand over or refuse:
cutoffs on both sides of a power of two, boxes that the tile repeats, atoms closer than its tables
reach, widths from none to wider than the cutoff, charges far from 1 or of very unequal size, pairs
exactly at the cutoff, and a skin too large for its coordinates (k_real64 then).

The oracle's own summation and FFT are good to about 1e-14 of the largest value; the bound is the
1e-12 that leaves for the sums of both sides."""

import numpy as np
import pytest

from gpu_util import cuda_or_skip, dev_tensor
from oracle import ewald
from workloads import rocksalt_lattice, water_box

pytestmark = pytest.mark.gpu


def _check(R, q, sigma, box, alpha, r_cut, skin, mesh, order=4, gaussian_self=True, tol=1e-12):
    qg = cuda_or_skip()
    s = qg.System(qg.make_params(len(q), box, alpha=alpha, r_cut=r_cut, skin=skin, mesh=mesh, order=order,
                                 gaussian_self=gaussian_self))
    s.neighbor_build(dev_tensor(R))
    ref = ewald.coulomb_apply(R, q, sigma, box, alpha, r_cut, recip="pme", mesh=mesh, order=order,
                              gaussian_self=gaussian_self)
    for _ in range(2):  # the second apply finds the first one's charge scale cleared
        v, E, F, en = s.apply(dev_tensor(R), dev_tensor(q), dev_tensor(sigma))
        vmax = np.abs(ref["v"]).max()  # the scale of fields that cancel by symmetry too
        for got, want, scale in ((v, ref["v"], vmax), (E, ref["E"], vmax), (F, ref["F"], vmax * np.abs(q).max())):
            assert np.abs(got.cpu().numpy() - want).max() <= tol * max(np.abs(want).max(), scale)
        assert abs(float(en[0]) - ref["energy"]) <= tol * abs(q @ (q / np.maximum(sigma, 0.1))) * 20
    vp = np.full(len(q), np.nan)
    out = dev_tensor(vp)
    qg.qeq_coulomb_apply(s.ctx, dev_tensor(R), dev_tensor(q), dev_tensor(sigma), out)  # potential only
    assert np.abs(out.cpu().numpy() - ref["v"]).max() <= tol * np.abs(ref["v"]).max()
    s.close()


def _charges(n, seed, scale=0.4):
    q = scale * np.random.default_rng(seed).standard_normal(n)
    return q - q.mean()


@pytest.mark.parametrize("n_mol,r_cut,skin,order", [
    (20, 4.0, 0.4, 4), (60, 4.01, 0.5, 4), (216, 8.0, 1.0, 4), (216, 8.01, 1.0, 5), (216, 9.0, 1.0, 6),
    (700, 6.0, 0.5, 4), (1501, 5.5, 1.0, 4), (1, 2.2, 0.3, 4)])
def test_water(n_mol, r_cut, skin, order):
    w = water_box(n_mol, seed=n_mol)
    _check(w.R, _charges(w.n_atoms, n_mol), w.sigma, w.box, 0.34, r_cut, skin, (24, 24, 24), order)


@pytest.mark.parametrize("scale", [1e-150, 1e-6, 1e5, 1e150])
def test_charge_scales(scale):
    w = water_box(100, seed=3)
    _check(w.R, _charges(w.n_atoms, 4, scale), w.sigma, w.box, 0.34, 6.0, 1.0, (20, 20, 20))


def test_one_large_charge():
    w = water_box(100, seed=3)
    q = _charges(w.n_atoms, 4, 1e-3)
    q[17] = 40.0
    _check(w.R, q, w.sigma, w.box, 0.34, 6.0, 1.0, (20, 20, 20))


@pytest.mark.parametrize("sigma", [(0.0, 0.0), (0.05, 0.3), (0.5, 3.0), (4.0, 9.0)])
def test_widths(sigma):
    w = water_box(100, seed=5)
    s = np.random.default_rng(6).uniform(*sigma, w.n_atoms)
    s[::7] = sigma[0]
    _check(w.R, _charges(w.n_atoms, 7), s, w.box, 0.34, 7.0, 1.0, (20, 20, 20), gaussian_self=sigma[0] > 0)


def test_uniform_atoms_reach_the_exact_path():
    """Atoms at random: pairs down to a few hundredths of an Angstrom."""
    rng = np.random.default_rng(8)
    box = np.array([13.0, 17.0, 11.0])
    R = rng.uniform(-0.5, 1.5, (600, 3)) * box
    _check(R, _charges(600, 9), np.full(600, 0.4), box, 0.4, 5.0, 0.5, (16, 20, 16))


def test_pairs_exactly_at_the_cutoff():
    """Lattice spacing 2, r_cut 4: shells at the cutoff are excluded, as in FP64."""
    R, q, L = rocksalt_lattice(4, 2.0)
    _check(R, q, np.full(len(q), 0.3), np.array([L] * 3), 0.5, 4.0, 0.5, (24, 24, 24), gaussian_self=False)


def test_large_skin_takes_the_general_kernel():
    w = water_box(216, seed=11)
    _check(w.R, _charges(w.n_atoms, 12), w.sigma, w.box, 0.34, 4.1, 6.0, (24, 24, 24))
