"""The c != 0 kernels by Taylor tables (pm_green.cuh) against the oracle's Hankel functions,
over the tables' whole range and both its ends: K~ and R~ of a unit density at one node are
w_j K and w_j R at every node without a correction for that node's patch.

Tolerance: the functions at the cells' centres are good to 1.4e-14, the argument's rounding
turns the phase (or scales the decay) by |k| r 2^-52, and as much again for the oracle's:
K to 4e-14 (1 + |k| r) of its modulus, R (sums of up to five such terms) to ten times that of the
largest."""

import numpy as np
import pytest

from workloads import cubed_sphere

pytestmark = pytest.mark.gpu

CS = [1e-9, -1e-9, 1e-5, -1e-5, 0.3, -0.3, 4.0, -4.0, 60.0, -60.0, 260.0, -250.0, 1100.0, -1000.0,
      5000.0, 1e-9j, -1e-6 + 1e-7j, 4.0 + 1.0j, 4.0 - 1.0j, -3.0 + 2.0j, 60.0 + 80.0j,
      90.0 - 20.0j, -100.0 + 5.0j]


@pytest.fixture(scope="module")
def surface():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_12501_gb300 as pm
    ctx = pm.Context(0)
    sf = cubed_sphere(2, 3, axes=(1.0, 0.9, 1.1))
    S = pm.Surface.from_fixture(ctx, sf)
    yield sf, S
    S.close()
    ctx.close()


@pytest.mark.parametrize("c", CS)
def test_pairs(surface, c):
    from oracle.kernels import scaled_pair_c, wavenumber
    sf, S = surface
    x, n = sf.nodes, sf.normals
    a = 1.0 + 0.2 * x[:, 0]
    ga = np.zeros((sf.N, 3))
    cv = c * (1.0 + 0.1 * x[:, 1])
    S.set_coeff_c(a, ga, cv)
    rp, bp, _, _ = S.get_near(corrections=False)
    k = wavenumber(cv, a)
    for j in (0, 100, sf.N - 1):
        e = np.zeros(sf.N)
        e[j] = 1.0
        K, R = S.apply_c(e, "K"), S.apply_c(e, "R")
        far = np.array([j // 9 not in bp[rp[i]:rp[i + 1]] for i in range(sf.N)])
        assert far.sum() > 20
        pair = [scaled_pair_c(x[i], n[i], sf.curvature[i], a[i], ga[i], cv[i], x[j], k[j])
                for i in np.flatnonzero(far)]
        wR, wK = (sf.weights[j] / a[j] * np.array([p[q] for p in pair]) for q in (0, 1))
        tol = 4e-14 * (1.0 + abs(k[j]) * np.linalg.norm(x[far] - x[j], axis=1))
        assert (np.abs(K[far] - wK) <= tol * np.abs(wK)).all()
        assert np.abs(R[far] - wR).max() <= 10 * tol.max() * np.abs(wR).max()


# R entry by entry, with a gradient of a: each of its terms is g, g' or q g times factors good to a
# few 2^-53, so an entry may be off by twice K's tolerance (the derivative's and the oracle's) of
# the sum of its terms' moduli, the cosines taken as 1
@pytest.mark.parametrize("c", CS)
def test_remainder_entries(surface, c):
    from oracle.kernels import green_scaled, scaled_pair_c, wavenumber
    sf, S = surface
    x, n, H = sf.nodes, sf.normals, sf.curvature
    a = 1.0 + 0.2 * x[:, 0]
    ga = 0.2 * (np.array([1.0, 0.0, 0.0]) - n * n[:, :1])
    cv = c * (1.0 + 0.1 * x[:, 1])
    S.set_coeff_c(a, ga, cv)
    rp, bp, _, _ = S.get_near(corrections=False)
    k = wavenumber(cv, a)
    for j in (0, 57, 140, sf.N - 1):
        e = np.zeros(sf.N)
        e[j] = 1.0
        R = S.apply_c(e, "R")
        far = np.flatnonzero([j // 9 not in bp[rp[i]:rp[i + 1]] for i in range(sf.N)])
        r = np.linalg.norm(x[far] - x[j], axis=1)
        g, g1, _ = (np.abs(v) for v in green_scaled(r, k[j]))
        want = np.array([scaled_pair_c(x[i], n[i], H[i], a[i], ga[i], cv[i], x[j], k[j])[0] for i in far])
        q = abs(k[j]) ** 2
        terms = ((np.linalg.norm(ga[far], axis=1) + 2.0 * a[far] * np.abs(H[far]) + 2.0 * a[far] / r) * g1
                 + (np.abs(cv[far]) + 2.0 * a[far] * q) * g)
        tol = 4e-14 * (1.0 + abs(k[j]) * r)
        weight = sf.weights[j] / a[j]
        assert (np.abs(R[far] - weight * want) <= 2.0 * tol * weight * terms).all()
