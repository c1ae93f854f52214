"""Rounding error of the near-field product of several right-hand sides (18 x 18 and larger blocks in FP32) against
64 bits.  The blocks are summed with compensation, so what counts is the sum over a block's columns.  The reference
is one rounding of a running sum per column (complex product rounded once, then added), emulated here on the same
blocks; the kernel keeps the two halves of the complex product in two running sums, each of half the variance and
rounded once per column, which comes to the same.  Two roundings of one running sum per column would be sqrt(2)
times that, 1.2 with the roundings of blocks and vectors; the root mean square over 7e3 and more entries is
certain to about 1 %: bound 1.1."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,R", [(2, 8), (2, 5), (3, 8), (4, 4)])
def test_rounding_error_of_the_batched_near_field(p, R):
    from paper_1807_03097_gb300 import Solver

    s = Solver(G.cube(), p=p, level_m=1, kappa=1.0, q=3, eta=1e-3, precision=1)
    assert s.nfar == 0
    rng = np.random.default_rng(53)
    x = rng.standard_normal((R, s.nsup)) + 1j * rng.standard_normal((R, s.nsup))
    got = s.matvec_superspace(x)
    B, near = s.near_blocks(), s.blocks()[1]
    s.close()
    nb = B.shape[1]
    X = x.reshape(R, -1, nb)[:, near[:, 1]].transpose(1, 2, 0)  # [pair][column][right-hand side]
    exact, plain = np.zeros((2, x.shape[1] // nb, nb, R), dtype=complex)
    np.add.at(exact, near[:, 0], np.matmul(B, X))
    Bf, Xf = B.astype(np.complex64).astype(complex), X.astype(np.complex64).astype(complex)
    run = np.zeros((len(near), nb, R), dtype=np.complex64)
    for c in range(nb):
        run = run + (Bf[:, :, c, None] * Xf[:, None, c]).astype(np.complex64)
    np.add.at(plain, near[:, 0], run.astype(complex))
    y = got.reshape(R, -1, nb).transpose(1, 2, 0)
    assert np.linalg.norm(y - exact) < 1.1 * np.linalg.norm(plain - exact)
