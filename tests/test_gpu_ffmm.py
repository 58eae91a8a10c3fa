"""Float-float sums of 8 and more right-hand sides on the tensor cores (pm_ffmm.cu) against the
float64 sums, column by column, and batches of operators on one geometry (the
shared coefficient-free matrices from five on) against single solves.

Tolerance of the sums: an entry is good to some 2^-44 (lazy float-float arithmetic), its fixed
point to 2^-53 of the largest, which is within 2^10 of the typical one here; both add up at
random over at most 2,000 sources: 1e-12 of the column's largest value leaves a factor of ten."""

import numpy as np
import pytest

from workloads import cubed_sphere, torus
from workloads.coefficients import smooth_random_coefficient
from workloads.rhs import random_harmonic_rhs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_12501_gb300 as pm
    c = pm.Context(0)
    yield c
    c.close()


def _operator(ctx, s, seed):
    import paper_2401_12501_gb300 as pm
    c = smooth_random_coefficient(s, seed)
    op = pm.Surface.from_fixture(ctx, s)
    op.set_coeff(c.a, c.grad_a)
    return op


# 54 to 1,944 nodes: below a tile of 64 targets and a stage of 128 sources, one over, several
@pytest.mark.parametrize("make", [lambda: cubed_sphere(1, 3), lambda: cubed_sphere(1, 5, axes=(1, 1.5, 2)),
                                  lambda: cubed_sphere(1, 8, axes=(1, 1.5, 2)),
                                  lambda: torus(9, 6, 6)])
@pytest.mark.parametrize("nrhs", [8, 17, 65])
def test_columns_match_float64(ctx, make, nrhs):
    s = make()
    op = _operator(ctx, s, 3)
    rng = np.random.default_rng(nrhs)
    F = rng.standard_normal((nrhs, s.N)) * 10.0 ** rng.integers(-30, 30, (nrhs, 1))
    F[1] = 0.0
    F[2, 1:] = 0.0                     # one source
    for apply in (op.apply_R, op.apply_K):
        got, want = apply(F, "ff"), apply(F, "fp64")
        scale = np.abs(want).max(1, keepdims=True)
        assert (np.abs(got - want) <= 1e-12 * scale).all()
    op.close()


def test_undefined_strengths_stay_in_their_column(ctx):
    s = cubed_sphere(1, 5)
    op = _operator(ctx, s, 1)
    F = np.ones((9, s.N))
    F[4, 7] = np.nan
    y = op.apply_R(F, "ff")
    assert np.isnan(y[4]).any()
    assert np.isfinite(np.delete(y, 4, 0)).all()
    op.close()


@pytest.mark.parametrize("nops,nrhs", [(4, 9), (5, 3), (8, 9), (17, 2)])
def test_operators_on_one_geometry(ctx, nops, nrhs):
    import paper_2401_12501_gb300 as pm
    s = cubed_sphere(1, 7, axes=(1.0, 1.5, 2.0))
    ops = [_operator(ctx, s, 0)]
    for k in range(1, nops):
        c = smooth_random_coefficient(s, k)
        ops.append(ops[0].clone())
        ops[-1].set_coeff(c.a, c.grad_a)
    rhs = [np.stack([random_harmonic_rhs(s, 10 * k + r) for r in range(nrhs)]) for k in range(nops)]
    us, _ = pm.solve_multi(ops, rhs, tol=1e-11)
    for op, F, U in zip(ops, rhs, us):
        for f, u in zip(F, U):
            ref, _ = op.solve(f, tol=1e-11)
            # both to a residual of 1e-11: 1e-9 covers operators with an inverse up to 50
            assert np.abs(u - ref).max() <= 1e-9 * np.abs(ref).max()
    for op in ops:
        op.close()
