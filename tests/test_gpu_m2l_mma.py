"""Mixed M2L of one and a few right-hand sides (k_m2l_mma) against the FP64 oracle, at the edges of its
16-row tiles and 64-node chunks (4 to 289 interpolation nodes, one to seven warps a block, split
and whole source lists, full and ragged groups of right-hand sides) and in its general form (phases
reduced explicitly, lengths not scaled by the wavenumber).

Tolerance of the product (relative 2-norm): an entry's error is at most about 2^-20.5 from the hardware
sine and cosine, 2^-22 from the split operands and 2^-22 from the reciprocal square root, together
1.2e-6, plus the phase: kappa times a few units of 2^-24 of the cluster radius (below 0.8 here)."""
import numpy as np
import pytest

import oracle as O
from workloads import geometry as G

pytestmark = pytest.mark.gpu

CASES = [
    # geometry, m, kappa, q, right-hand sides
    (G.sphere, 2, 1.0, 1, 1), (G.sphere, 2, 1.0, 3, 7), (G.cube, 2, 2.0, 4, 3), (G.sphere, 2, 2.0, 5, 5),
    (G.torus, 1, 2.0, 6, 5), (G.sphere, 2, 1.0, 8, 4), (G.sphere, 2, 1.0, 9, 4), (G.sphere, 1, 3.0, 12, 8),
    (G.sphere, 1, 3.0, 16, 2), (G.torus, 2, 3.0, 7, 1),
    (G.sphere, 2, 1e-7, 4, 1), (G.sphere, 1, 400.0, 6, 3),  # general form: tiny kappa, large phases
]


@pytest.mark.parametrize("mk,m,kappa,q,nrhs", CASES, ids=[f"{c[0].__name__}_m{c[1]}_k{c[2]}_q{c[3]}_r{c[4]}" for c in CASES])
def test_mixed_m2l_vs_oracle(mk, m, kappa, q, nrhs):
    from paper_1807_03097_gb300 import Solver

    s = Solver(mk(), p=1, level_m=m, kappa=kappa, q=q, eta=1.6, precision=1)
    r = O.Problem(mk(), p=1, m=m, kappa=kappa, q=q, eta=1.6)
    assert s.nfar > 0
    rng = np.random.default_rng(90 + q)
    x = rng.standard_normal((nrhs, s.ndof)) + 1j * rng.standard_normal((nrhs, s.ndof))
    tol = 1.2e-6 + 4 * kappa * 0.8 * 2.0 ** -24
    y, yr = s.matvec(x if nrhs > 1 else x[0]).reshape(nrhs, -1), r.fmm_matvec(x)
    for i in range(nrhs):
        assert np.linalg.norm(y[i] - yr[i]) / np.linalg.norm(yr[i]) < tol, i
    s.close()
