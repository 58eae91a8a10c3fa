"""Float-float sums of 8 and 17 right-hand sides on surfaces whose nodes lie unevenly, or far from
the origin, against the float64 sums.

Tolerances.  Graded patches: as for even ones (test_gpu_ffmm.py), an entry is good to some 2^-44
of itself and the errors add up at random over at most 2,200 sources: 1e-12 of the column's largest
value, whatever the ratio of the node distances.  Offset surfaces: float-float coordinates carry
2^-48 of their size, which bounds what any of the sums can give; all form the same differences of
the same coordinates, so the columns may be twice as far off as one at a time, and those 1e-12."""

import numpy as np
import pytest

from workloads import cubed_sphere, star_surface
from workloads.coefficients import smooth_random_coefficient
from workloads.surfaces import _FACES, Surface, _level_set_curvatures, gauss_legendre

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


def _graded(levels, p=6, axes=(1.0, 1.5, 2.0)):
    """An ellipsoid of one patch a face, the first halved `levels` times towards a corner."""
    q = np.pi / 4
    boxes = [(f, -q, q, -q, q) for f in range(1, 6)]
    a0, a1, b0, b1 = -q, q, -q, q
    for _ in range(levels):
        am, bm = 0.5 * (a0 + a1), 0.5 * (b0 + b1)
        boxes += [(0, am, a1, b0, bm), (0, a0, am, bm, b1), (0, am, a1, bm, b1)]
        a1, b1 = am, bm
    boxes.append((0, a0, a1, b0, b1))
    t, wt = gauss_legendre(p)
    D = np.asarray(axes)
    parts = []
    for f, a0, a1, b0, b1 in boxes:
        c0, e1, e2 = (np.asarray(v, dtype=np.float64) for v in _FACES[f])
        xi = (0.5 * (a0 + a1) + 0.5 * (a1 - a0) * t)[:, None, None] + 0.0 * t[None, :, None]
        eta = (0.5 * (b0 + b1) + 0.5 * (b1 - b0) * t)[None, :, None] + 0.0 * t[:, None, None]
        c = c0 + np.tan(xi) * e1 + np.tan(eta) * e2
        cn = np.linalg.norm(c, axis=-1, keepdims=True)
        ys = c / cn
        tangents = []
        for d, h in ((e1 / np.cos(xi) ** 2, 0.5 * (a1 - a0)), (e2 / np.cos(eta) ** 2, 0.5 * (b1 - b0))):
            tangents.append((d - ys * np.sum(ys * d, -1, keepdims=True)) / cn * h * D)
        n = ys / D
        n /= np.linalg.norm(n, axis=-1, keepdims=True)
        H, kg = _level_set_curvatures(ys * D, D)
        w = wt[:, None] * wt * np.linalg.norm(np.cross(*tangents), axis=-1)
        parts.append((ys * D, n, np.concatenate(tangents, -1), H, w, kg))
    x, n, tn, H, w, kg = (np.concatenate([v.reshape(p * p, -1) for v in vs]) for vs in zip(*parts))
    return Surface(kind="graded", npatch=len(boxes), p=p, nodes=x, normals=n, tangents=tn,
                   curvature=H.ravel(), weights=w.ravel(), gauss_curvature=kg.ravel())


def _operator(ctx, s):
    import paper_2401_12501_gb300 as pm
    c = smooth_random_coefficient(s, 3)
    op = pm.Surface.from_fixture(ctx, s)
    op.set_coeff(c.a, c.grad_a)
    return op


def _columns(s, nrhs):
    F = np.random.default_rng(nrhs).standard_normal((nrhs, s.N))
    F[1] = 1.0
    far = np.linalg.norm(s.nodes - s.nodes[-1], axis=1)
    F[2] *= far > np.median(far)          # nothing near the small patches
    return F


# nodes as close as 1e-2, 1e-4, 1e-5 and 1e-6 of the surface's size
@pytest.mark.parametrize("levels", [4, 11, 14, 18])
@pytest.mark.parametrize("nrhs", [8, 17])
def test_graded_patches(ctx, levels, nrhs):
    s = _graded(levels)
    op = _operator(ctx, s)
    F = _columns(s, nrhs)
    for apply in (op.apply_R, op.apply_K):
        got, want = apply(F, "ff"), apply(F, "fp64")
        assert (np.abs(got - want) <= 1e-12 * np.abs(want).max(1, keepdims=True)).all()
    op.close()


@pytest.mark.parametrize("offset", [1e4, 1e6])
@pytest.mark.parametrize("nrhs", [8, 17])
def test_offset_surfaces(ctx, offset, nrhs):
    s = cubed_sphere(2, 8, axes=(1.0, 1.5, 2.0))
    s.nodes = s.nodes + offset * np.array([1.0, 0.7, -0.3])
    op = _operator(ctx, s)
    F = _columns(s, nrhs)
    for apply in (op.apply_R, op.apply_K):
        got, want = apply(F, "ff"), apply(F, "fp64")
        one = np.stack([apply(f, "ff") for f in F])
        scale = np.abs(want).max(1)
        assert (np.abs(got - want).max(1) <= 2 * np.abs(one - want).max(1) + 1e-12 * scale).all()
    op.close()


# below 128 nodes eight columns run as seven do (the tensor-core sums are slower there): same bits
@pytest.mark.parametrize("make", [lambda: cubed_sphere(1, 3), lambda: cubed_sphere(1, 4)])
def test_small_surfaces_keep_the_pair_sums(ctx, make):
    s = make()
    op = _operator(ctx, s)
    F = _columns(s, 8)
    for apply in (op.apply_R, op.apply_K):
        assert np.array_equal(apply(F, "ff")[:7], apply(F[:7], "ff"))
    op.close()


# the star's kinks at its poles leave a few rows with entries far above their mean, beside which the
# rest of the row must stay as good; such a surface is even enough for the tensor-core sums, so its
# bits are not those of seven columns
def test_kinked_star(ctx):
    s = star_surface(8, 8)
    op = _operator(ctx, s)
    F = _columns(s, 8)
    F[3] *= np.abs(s.nodes[:, 2]) < 0.9 * np.linalg.norm(s.nodes, axis=1)      # nothing near the kinks
    got, want = op.apply_R(F, "ff"), op.apply_R(F, "fp64")
    assert (np.abs(got - want) <= 1e-12 * np.abs(want).max(1, keepdims=True)).all()
    assert not np.array_equal(got[:7], op.apply_R(F[:7], "ff"))
    op.close()
