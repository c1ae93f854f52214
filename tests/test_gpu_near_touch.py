"""Touching pairs with factorised sums (k_near_touch) against the direct kernel (k_near_quad), which takes
over when a geometry knot lies inside an element: the same surface with a knot inserted at 0.3 (no element
boundary: direct kernel) and at 0.5 (an element boundary: factorised, two spans per patch direction).  All p, all kinds of
touching pairs with their symmetries (sphere, cube), singular rules from 2 points to the largest that
fits, and one beyond (direct kernel, against the library's own block symmetry only through the oracle
tests).  Tolerance as in the parity tests: the rules are the same, the sums are in another order."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu

TOL64 = 1e-11


def insert_knot(patch, t):
    """The same rational patch with the knot t inserted once in both directions (Boehm)."""
    H = np.concatenate([patch["cp"] * patch["w"][..., None], patch["w"][..., None]], -1)
    knots = []
    for d, axis in ((0, 1), (1, 0)):
        deg, k = patch["deg"][d], patch["knots"][d]
        C = np.moveaxis(H, axis, 0)
        s = np.searchsorted(k, t, side="right") - 1
        out = []
        for i in range(C.shape[0] + 1):
            if i <= s - deg:
                out.append(C[i])
            elif i > s:
                out.append(C[i - 1])
            else:
                a = (t - k[i]) / (k[i + deg] - k[i])
                out.append(a * C[i] + (1 - a) * C[i - 1])
        H = np.moveaxis(np.stack(out), 0, axis)
        knots.append(np.insert(k, s + 1, t))
    return {"deg": patch["deg"], "knots": tuple(knots), "cp": np.ascontiguousarray(H[..., :3] / H[..., 3:]),
            "w": np.ascontiguousarray(H[..., 3])}


@pytest.mark.parametrize("mk,p,m,gs", [(G.sphere, 1, 1, 0), (G.sphere, 2, 1, 0), (G.cube, 3, 1, 0), (G.sphere, 4, 1, 0),
                                       (G.cube, 1, 2, 2), (G.sphere, 2, 1, 3), (G.cube, 3, 1, 8), (G.cube, 1, 1, 6)],
                         ids=lambda v: getattr(v, "__name__", str(v)))
def test_factorised_blocks_match_direct_blocks(mk, p, m, gs):
    from paper_1807_03097_gb300 import Solver

    def blocks(patches):
        s = Solver(patches, p=p, level_m=m, kappa=2.0, q=2, eta=1.6, quad_singular=gs)
        far, near = s.blocks()
        b = s.near_blocks()
        s.close()
        return near, b

    geo = mk()
    n0, direct = blocks([insert_knot(q, 0.3) for q in geo])
    for other in (geo, [insert_knot(q, 0.5) for q in geo]):
        n1, b = blocks(other)
        assert np.array_equal(n0, n1)
        scale = np.abs(direct).max(axis=(1, 2))
        assert (np.abs(b - direct).max(axis=(1, 2)) / scale).max() < TOL64
