"""Kept FP64 matrices in digits (m2l_store = 2) in units of length whose squares leave the range of FP32 (2^-75 and
2^64): the fixed point of a target's matrices follows the distances of its list in FP64.  Against the form that evaluates
every entry (m2l_store = 1), with the tolerance of test_gpu_m2l_f64.py; powers of two as units change no
rounding, so the product of the unit sphere only scales.  2^-40 and 2^40 are where the FP32 distances end."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu

TOL = 3e-13


@pytest.mark.parametrize("exponent", [-100, -76, -41, -39, 39, 41, 66, 100])
def test_units_of_length(exponent):
    from paper_1807_03097_gb300 import Solver

    unit = 2.0 ** exponent
    kw = dict(p=1, level_m=2, kappa=2.0 / unit, q=4, eta=1.6, precision=0)
    a, b = Solver(G.sphere(radius=unit), m2l_store=1, **kw), Solver(G.sphere(radius=unit), m2l_store=2, **kw)
    assert a.nfar > 0
    rng = np.random.default_rng(61)
    x = rng.standard_normal(a.ndof) + 1j * rng.standard_normal(a.ndof)
    y, z = a.matvec(x), b.matvec(x)
    assert np.abs(y - z).max() / np.abs(y).max() < TOL
    a.close()
    b.close()
