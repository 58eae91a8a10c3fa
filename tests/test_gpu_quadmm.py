"""The near-field weights are formed for eight (target, patch) columns at a time (k_qm): which
columns share a group, which lanes a partial group leaves empty and where its sums are kept
follow from the order of the patches.  None of it may show: each column is scaled, multiplied
and added up by itself, so a surface with its patches in another order has the same correction
blocks, bit for bit.  That the blocks are the right ones, the oracle's tests say."""

from types import SimpleNamespace

import numpy as np
import pytest

from workloads import cubed_sphere, ellipsoid_coefficient
from workloads.trisurfaces import tri_ellipsoid

pytestmark = pytest.mark.gpu
AXES = (1.0, 1.5, 2.0)


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_12501_gb300 as pm
    c = pm.Context(0)
    yield c
    c.close()


def blocks(ctx, fields, co, order, n):
    """{(node, patch): (R block, K block)}, nodes and patches by their number in `fields`."""
    import paper_2401_12501_gb300 as pm
    rows = (order[:, None] * n + np.arange(n)).ravel()
    data = {k: v[rows] if isinstance(v, np.ndarray) and len(v) == len(rows) else v
            for k, v in fields.items()}
    s = pm.Surface.from_fixture(ctx, SimpleNamespace(**data))
    s.set_coeff(co.a[rows], co.grad_a[rows])
    rp, bp, cR, cK = s.get_near()
    out = {(rows[i], order[bp[b]]): (cR[b], cK[b])
           for i in range(len(rows)) for b in range(rp[i], rp[i + 1])}
    s.close()
    return out


# n nodes a patch: one k-step of 16 and part of it, whole ones, one more node, the largest; 6 and
# 20 patches: a group that is not full, and whole ones with a rest
@pytest.mark.parametrize("shape,p", [("quad", 2), ("quad", 4), ("quad", 5), ("quad", 8), ("quad", 9),
                                     ("quad", 11), ("tri", 2), ("tri", 5), ("tri", 6), ("tri", 8)])
def test_patch_order_changes_no_bit(ctx, shape, p):
    surf = cubed_sphere(1, p, axes=AXES) if shape == "quad" else tri_ellipsoid(0, p, axes=AXES)
    names = ["npatch", "p", "nodes", "normals", "tangents", "curvature", "weights"]
    fields = {k: getattr(surf, k) for k in names + (["ref_u", "ref_v", "ref_w"] if shape == "tri" else [])}
    n = surf.N // surf.npatch
    co = ellipsoid_coefficient(surf)
    first = blocks(ctx, fields, co, np.arange(surf.npatch), n)
    other = blocks(ctx, fields, co, np.random.default_rng(p).permutation(surf.npatch), n)
    assert first.keys() == other.keys()
    for key, (R, K) in first.items():
        assert np.isfinite(R).all() and np.isfinite(K).all()
        assert np.array_equal(R, other[key][0]) and np.array_equal(K, other[key][1]), key
