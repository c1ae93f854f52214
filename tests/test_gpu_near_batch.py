"""Near-field product of several right-hand sides (k_near_apply_multi) against the single-vector product.
Without admissible pairs the superspace product of a batch is the near field alone.  Both
add FP32 block products of 2 nb terms and compensated block sums, so they differ by at most
(2 nb + 4) 2^-24 of the absolute sums (below 2e-5 of the largest row for smooth rows; random vectors stay
under 1e-6); 8 x 8 blocks keep every rounding error and agree to 1e-11."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu


# one lane group per four right-hand sides: ragged quads, sources split over groups, several grid rows
@pytest.mark.parametrize("p,R", [(1, 2), (1, 7), (1, 33), (2, 3), (2, 13), (2, 64), (3, 5), (3, 32), (3, 64), (4, 6), (4, 19)])
def test_batched_near_field_matches_single(p, R):
    from paper_1807_03097_gb300 import Solver

    s = Solver(G.cube(), p=p, level_m=1, kappa=1.0, q=3, eta=1e-3, precision=1)
    assert s.nfar == 0
    rng = np.random.default_rng(31 + R)
    x = rng.standard_normal((R, s.nsup)) + 1j * rng.standard_normal((R, s.nsup))
    y = s.matvec_superspace(x)
    z = np.stack([s.near_apply(v) for v in x])
    assert np.abs(y - z).max() / np.abs(z).max() < (1e-11 if p == 1 else 2e-5)
    s.close()
