"""FP64 M2L from kept matrices in digits on the FP16 tensor cores (m2l_store = 2) against the form that
evaluates every entry in FP64 (m2l_store = 1), at the edges of its 16-row tiles and 16-node steps
(odd and even node counts from 4 to 289, one to nineteen warps a block, split and whole lists).

Tolerance: both forms add at most about 4e4 products; the digits' fixed point (2^-58 of the largest entry
and source of a list) and the products left out (2^-57) and the FP64 sums of the other form
(2^-53 each, random) stay below 4e4 x 2^-57 = 3e-13 of the largest row."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu

TOL = 3e-13
CASES = [(G.sphere, 2, 1.0, 4), (G.cube, 2, 2.0, 1), (G.cube, 2, 2.0, 2), (G.cube, 3, 0.01, 3), (G.torus, 2, 3.0, 5),
         (G.sphere, 2, 5.0, 7), (G.sphere, 1, 3.0, 11), (G.sphere, 1, 3.0, 16)]


def relmax(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("mk,m,kappa,q", CASES, ids=[f"{c[0].__name__}_m{c[1]}_k{c[2]}_q{c[3]}" for c in CASES])
def test_digits_match_evaluated_entries(mk, m, kappa, q):
    from paper_1807_03097_gb300 import Solver

    kw = dict(p=1, level_m=m, kappa=kappa, q=q, eta=1.6, precision=0)
    a, b = Solver(mk(), m2l_store=1, **kw), Solver(mk(), m2l_store=2, **kw)
    assert a.nfar > 0
    rng = np.random.default_rng(95 + q)
    x = rng.standard_normal(a.ndof) + 1j * rng.standard_normal(a.ndof)
    y = a.matvec(x)
    assert relmax(b.matvec(x), y) < TOL
    for f in (2.0 ** -600, 2.0 ** 600):  # the fixed point follows the size of the input
        assert relmax(b.matvec(x * f) / f, y) < TOL
    one = np.zeros_like(x)
    one[:3] = 1.0  # sources on one cluster, zero elsewhere
    assert relmax(b.matvec(one), a.matvec(one)) < TOL
    assert not b.matvec(np.zeros_like(x)).any()
    bad = x.copy()
    bad[1] = np.nan
    assert np.array_equal(np.isnan(b.matvec(bad)), np.isnan(a.matvec(bad)))
    a.close()
    b.close()
