"""Touching pairs at the limit of k_near_touch's rules (two points a thread: 2 x 128 for p <= 2, 2 x 256 beyond)
against the oracle with the same rule: the largest rule that fits (6; 8) and the first that does not (7; 9), which
k_near_quad takes.  A rule let through beyond the limit would drop points.  Tolerance of the parity tests."""
import numpy as np
import pytest

import oracle as O
from workloads import geometry as G

pytestmark = pytest.mark.gpu

TOL64 = 1e-11


@pytest.mark.parametrize("p,g", [(1, 6), (1, 7), (2, 6), (2, 7), (3, 8), (3, 9), (4, 9)])
def test_blocks_at_the_limit_of_the_rule(p, g):
    from paper_1807_03097_gb300 import Solver

    kw = dict(p=p, kappa=2.0, q=2, eta=1.6)
    s = Solver(G.cube(), level_m=0, quad_singular=g, **kw)
    r = O.Problem(G.cube(), m=0, g_sing=g, **kw)
    at = {tuple(e): k for k, e in enumerate(r.near_pairs())}
    a, b = s.near_blocks(), r.near_blocks()[[at[tuple(e)] for e in s.blocks()[1]]]
    s.close()
    assert np.abs(a - b).max() < TOL64 * np.abs(b).max()
