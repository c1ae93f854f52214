"""A lockstep solve keeps one M2L kernel while its systems drop out, down to the last one (k_m2l_tc for three and four systems
at 81 nodes).  Copies of a system against the system among zero right-hand sides, which drop out at once: up to
four right-hand sides take the same sums in the same order in every kernel of the product, so the iterates are
the same bit by bit, unless the last system changes to another kernel."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mk,p,m,kappa,R", [(G.cube, 1, 2, 2.0, 4), (G.sphere, 1, 2, 1.0, 3), (G.sphere, 2, 2, 2.0, 4)],
                         ids=lambda v: getattr(v, "__name__", str(v)))
def test_last_system_keeps_the_kernel(mk, p, m, kappa, R):
    from paper_1807_03097_gb300 import Solver

    s = Solver(mk(), p=p, level_m=m, kappa=kappa, q=8, eta=1.6, precision=1, gmres_tol=1e-5)
    b = s.rhs(*G.plane_waves(1, 7))[0]
    x, info, st = s.solve(np.stack([b] * R))
    alone = np.zeros((R, s.ndof), dtype=complex)
    alone[2] = b
    y, info1, st1 = s.solve(alone)
    assert st == 0 and st1 == 0 and info.iterations == info1.iterations
    assert np.array_equal(x[0], x[2]) and np.array_equal(y[2], x[2]) and not y[0].any()
    s.close()
