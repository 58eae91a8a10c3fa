"""Solves of the c != 0 and open-surface systems form a dense matrix where the device has room
for it, and go pair by pair where it has not (PM_FAKE_HBM_BYTES = 0): both give the same
solution.  Each stops at a relative residual of 1e-12, so with the operators' inverses below
about 10 in norm the two agree to 1e-10 with room to spare."""

import numpy as np
import pytest

from workloads import cubed_sphere
from workloads import bvp as bands

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_12501_gb300 as pm
    c = pm.Context(0)
    yield c
    c.close()


def both(monkeypatch, solve):
    dense = solve()
    monkeypatch.setenv("PM_FAKE_HBM_BYTES", "0")
    pairs = solve()
    monkeypatch.delenv("PM_FAKE_HBM_BYTES")
    for d, p in zip(dense, pairs):
        assert np.abs(d - p).max() <= TOL * np.abs(p).max()


# 54 to 600 nodes: less than a block's rows and sources, one more, and a remainder of both
@pytest.mark.parametrize("m,p,kind", [(1, 3, "real"), (1, 5, "negative"), (1, 5, "complex"),
                                      (1, 7, "mixed"), (2, 5, "real")])
def test_wave_solve(ctx, monkeypatch, m, p, kind):
    import paper_2401_12501_gb300 as pm
    s = cubed_sphere(m, p, axes=(1.0, 1.5, 2.0))
    x = s.nodes
    c = {"real": 4.0 + x[:, 1], "negative": -4.0 - x[:, 0] ** 2, "complex": 4.0 + 1j * x[:, 2],
         "mixed": np.where(x[:, 2] > 0, 3.0, 2.0 + 0.5j)}[kind]
    S = pm.Surface.from_fixture(ctx, s)
    S.set_coeff_c(1.0 + 0.2 * x[:, 2] ** 2, None, c)
    f = np.cos(x[:, 0]) + 1j * x[:, 1]

    def solve():
        u, _, sigma = S.solve_c(f, tol=1e-12, return_sigma=True)
        return u, sigma

    both(monkeypatch, solve)
    S.close()


@pytest.mark.parametrize("kind,n,p,M", [("neumann", 4, 5, 12), ("dirichlet", 4, 6, 36),
                                        ("dirichlet", 3, 7, 135), ("neumann", 3, 6, 129)])
def test_edge_solve(ctx, monkeypatch, kind, n, p, M):
    edge_solve(ctx, monkeypatch, kind, n, p, M, 4)


# F M a multiple of 4 with M even (a Nyquist function) and odd, one tile of points and a
# remainder; F M not a multiple of 4, below and above a block's 128 nodes
@pytest.mark.parametrize("kind,M,F", [("neumann", 6, 6), ("dirichlet", 9, 8), ("neumann", 129, 8),
                                      ("dirichlet", 66, 8), ("dirichlet", 9, 6), ("neumann", 135, 6)])
def test_edge_columns(ctx, monkeypatch, kind, M, F):
    edge_solve(ctx, monkeypatch, kind, 3, 6, M, F)


def edge_solve(ctx, monkeypatch, kind, n, p, M, F):
    import paper_2401_12501_gb300 as pm
    band = bands.torus_band(2, n, p, M, F)
    co = (bands.band_coefficient(band) if kind == "neumann" else bands.constant_band_coefficient(band))
    S = pm.Surface.from_fixture(ctx, band.surface)
    S.set_coeff(co.a, co.grad_a)
    patch, uv = bands.edge_patches(band)
    ae, ao = ((bands.edge_a(band), bands.edge_a(band, True)) if kind == "neumann"
              else (np.ones(band.M), np.ones(F * band.M)))
    b = pm.BoundaryValueProblem(S, band.curves, ae, ao, patch, uv, kind=kind)
    rng = np.random.default_rng(5)
    sigma, mu = rng.standard_normal(S.N), rng.standard_normal(b.Me)
    f, fg = b.apply(sigma, mu)          # consistent data: the solution is (sigma, mu)

    def solve():
        u, _, s, m = b.solve(f, fg, tol=1e-12)
        return s, m

    both(monkeypatch, solve)
    b.close()
    S.close()


# data whose norm is undefined or overflows: no relative residual can be met, whichever way the
# operator is applied
@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e200])
@pytest.mark.parametrize("hbm", [None, "0"])
def test_undefined_data_do_not_converge(ctx, monkeypatch, bad, hbm):
    import paper_2401_12501_gb300 as pm
    from paper_2401_12501_gb300._lib import PmError
    if hbm is not None:
        monkeypatch.setenv("PM_FAKE_HBM_BYTES", hbm)
    s = cubed_sphere(1, 4, axes=(1.0, 1.5, 2.0))
    S = pm.Surface.from_fixture(ctx, s)
    S.set_coeff_c(np.ones(s.N), None, np.full(s.N, 3.0))
    f = np.ones(s.N)
    f[5] = bad
    with pytest.raises(PmError, match="NOT_CONVERGED"):
        S.solve_c(f)
    S.close()

    band = bands.torus_band(2, 3, 5, 6, 4)
    co = bands.constant_band_coefficient(band)
    S = pm.Surface.from_fixture(ctx, band.surface)
    S.set_coeff(co.a, co.grad_a)
    patch, uv = bands.edge_patches(band)
    b = pm.BoundaryValueProblem(S, band.curves, np.ones(band.M), np.ones(4 * band.M), patch, uv,
                                kind="dirichlet")
    f, fg = np.ones(S.N), np.ones(b.Me)
    for v in (f, fg):
        v[2] = bad
        with pytest.raises(PmError, match="NOT_CONVERGED"):
            b.solve(f, fg)
        v[2] = 1.0
    b.close()
    S.close()


# matrices of 6.1 GB with 12.1 GB free: more than half, so the pairs are summed at every step;
# with 64 GB free they are evaluated once
@pytest.mark.parametrize("free,dense", [(12.1e9, False), (64e9, True)])
def test_matrix_takes_half_of_the_free_memory_at_most(ctx, monkeypatch, free, dense):
    import paper_2401_12501_gb300 as pm
    from paper_2401_12501_gb300._lib import PM_PHASE_DIRECT64
    s = cubed_sphere(6, 8, axes=(1.0, 1.5, 2.0))
    S = pm.Surface.from_fixture(ctx, s)
    S.set_coeff_c(np.ones(s.N), None, np.full(s.N, 3.0))
    monkeypatch.setenv("PM_FAKE_HBM_BYTES", str(int(free)))
    S.profile()
    _, info = S.solve_c(s.nodes[:, 0] + 0j, tol=1e-3)
    _, sums = S.profile_read(PM_PHASE_DIRECT64)
    assert info.iterations > 1 and (sums == 1) == dense
    S.close()
