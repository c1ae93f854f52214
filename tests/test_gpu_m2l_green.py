"""Kernel entries of the kept FP64 matrices (table-driven e^{i kappa r}, iterated 1 / r) against the evaluated
form, which calls the CUDA functions.  Either entry is off by at most a few 2^-53 plus the rounding of the
phase, kappa r 2^-53; 1e-12 + 1e-14 kappa D leaves a factor of 50 for the sums (D the diameter, 2 units).
kappa D = 2e9 is past the range of the table's argument reduction, 2^-50 and 2^50 change the exponents."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unit,kD", [(1.0, 0.5), (1.0, 60.0), (1.0, 2e5), (1.0, 2e9), (2.0 ** -50, 4.0), (2.0 ** 49, 4.0)])
def test_kept_entries_match_evaluated(unit, kD):
    from paper_1807_03097_gb300 import Solver

    kw = dict(p=1, level_m=2, kappa=kD / (2 * unit), q=4, eta=1.6, precision=0)
    a, b = Solver(G.sphere(radius=unit), m2l_store=2, **kw), Solver(G.sphere(radius=unit), m2l_store=1, **kw)
    assert a.nfar > 0
    rng = np.random.default_rng(3)
    x = rng.standard_normal(a.nsup) + 1j * rng.standard_normal(a.nsup)
    y = [s.matvec_superspace(x[None])[0] - s.near_apply(x) for s in (a, b)]
    assert np.abs(y[0] - y[1]).max() / np.abs(y[1]).max() < 1e-12 + 1e-14 * kD
    a.close()
    b.close()
