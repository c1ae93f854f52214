"""The stages around the M2L in their forms: leaves with their parents in one block (FP32 always, FP64 from
152 x 4 leaves on) or on their own, roots that are leaves (m = 0), whose children are leaves (m = 1), and
deeper; split source lists or not; one vector and batches beyond one group of T launches' lanes.  The
FP64 product (pinned to the oracle by the parity tests in its small form) against the mixed product of
the same vectors within the mixed form's 2e-6 (its kernels' error bound, see test_gpu_m2l_mma.py, with
room for the tensor-core batch's accumulators of 3e-6 from 8 right-hand sides on)."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu

CASES = [(G.sphere, 1, 0, 3, 1), (G.sphere, 2, 1, 4, 3), (G.multicell, 1, 1, 3, 2), (G.torus, 1, 2, 5, 1),
         (G.torus, 3, 2, 3, 20), (G.cube, 1, 4, 2, 1), (G.cube, 2, 3, 12, 2)]


@pytest.mark.parametrize("mk,p,m,q,nrhs", CASES, ids=[f"{c[0].__name__}_p{c[1]}_m{c[2]}_q{c[3]}_r{c[4]}" for c in CASES])
def test_fp64_and_mixed_products_agree(mk, p, m, q, nrhs):
    from paper_1807_03097_gb300 import Solver

    kw = dict(p=p, level_m=m, kappa=2.0, q=q, eta=1.6)
    a, b = Solver(mk(), precision=0, **kw), Solver(mk(), precision=1, **kw)
    rng = np.random.default_rng(98)
    x = rng.standard_normal((nrhs, a.ndof)) + 1j * rng.standard_normal((nrhs, a.ndof))
    ya, yb = a.matvec(x), b.matvec(x if nrhs > 1 else x[0]).reshape(nrhs, -1)
    tol = 2e-6 if nrhs < 8 else 5e-6
    for i in range(nrhs):
        assert np.linalg.norm(ya[i] - yb[i]) / np.linalg.norm(ya[i]) < tol, i
    a.close()
    b.close()
