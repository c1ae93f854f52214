"""Near-field product of 8 x 8 blocks in the mixed form (k_near_apply_8): FP32 blocks, x* as hi + lo, every
rounding error of products and sums kept.  With fixed blocks the product is then linear to the
rounding of the compensation terms: at most about 40 blocks x 8 columns x 4 products of 2^-47 relative
to the absolute sums, 1e-11 of the largest row (sums in plain FP32 reach 1e-7)."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mk,m", [(G.sphere, 0), (G.cube, 1), (G.torus, 1), (G.sphere, 3)], ids=lambda v: getattr(v, "__name__", str(v)))
def test_near_product_is_linear(mk, m):
    from paper_1807_03097_gb300 import Solver

    s = Solver(mk(), p=1, level_m=m, kappa=0.5, q=3, eta=1.6, precision=1)
    rng = np.random.default_rng(97)
    x, y = (rng.standard_normal(s.nsup) + 1j * rng.standard_normal(s.nsup) for _ in range(2))
    z = s.near_apply(x + y)
    assert np.abs(z - s.near_apply(x) - s.near_apply(y)).max() / np.abs(z).max() < 1e-11
    assert np.abs(s.near_apply(2.0 ** 40 * x) - 2.0 ** 40 * s.near_apply(x)).max() == 0.0
    s.close()
