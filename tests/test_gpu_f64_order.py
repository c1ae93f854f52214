"""FP64 product with evaluated coupling matrices (m2l_store = 1): the M2L, whose blocks all start at once and then stay on
their SMs, starts when the near field on the second stream is done (beside it the blocks crowd some of the SMs
and take up to 1.8 times as long).  Read from the recorded phases: both are times since the end of the
gather, the near field's to its end, the moments' to the start of the M2L."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,m,R", [(2, 3, 1), (2, 3, 3), (1, 4, 2)])
def test_m2l_starts_after_the_near_field(p, m, R):
    from paper_1807_03097_gb300 import Solver

    s = Solver(G.sphere(), p=p, level_m=m, kappa=5.0, q=3, eta=1.6, precision=0, m2l_store=1)
    assert s.nfar > 0
    rng = np.random.default_rng(71)
    x = rng.standard_normal((R, s.ndof)) + 1j * rng.standard_normal((R, s.ndof))
    for _ in range(3):
        s.matvec(x if R > 1 else x[0])
        t = s.last_timings()
        assert t["moments_m2m"] >= t["near"] - 2e-3  # resolution of the events
    s.close()
