"""Tensor-core M2L in split FP16 (k_m2l_tc): tile sizes, source groups, field scales.

Tolerances: 1e-5 of the FP64 form per right-hand side (the bound of the mixed form).  Scaling a right-hand
side by a power of two scales every operand and its scale factor, so the product scales exactly."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu


def _rel(y, z):
    return np.linalg.norm(y - z) / np.linalg.norm(z)


# nodes 4 ... 121: one to 16 groups of 8 source nodes (whole and ragged), row tiles of 64, 96 and 128;
# 8, 17 and 33 right-hand sides: part of a block of 64 fields, two and three blocks
@pytest.mark.parametrize("q,R,kappa", [(1, 8, 1.0), (2, 8, 2.0), (3, 17, 1.0), (5, 8, 2.0), (7, 33, 2.0), (8, 8, 3.0),
                                       (9, 17, 3.0), (10, 8, 3.0), (4, 8, 1.0)])
def test_split_fp16_m2l_against_fp64_form(q, R, kappa):
    from paper_1807_03097_gb300 import Solver

    kw = dict(p=1, level_m=2, kappa=kappa, q=q, eta=1.6)
    s, d = Solver(G.sphere(), precision=1, m2l_batch=2, **kw), Solver(G.sphere(), precision=0, **kw)
    assert s.nfar > 0
    rng = np.random.default_rng(7 + q)
    x = rng.standard_normal((R, s.ndof)) + 1j * rng.standard_normal((R, s.ndof))
    y = s.matvec(x)
    for r in range(0, R, 5):
        assert _rel(y[r], d.matvec(x[r])) < 1e-5
    # right-hand sides of very different size side by side: a zero one, and powers of two of the first
    x[1] = 0.0
    x[2], x[3], x[4] = 2.0 ** 40 * x[0], 2.0 ** -40 * x[0], 2.0 ** -90 * x[0]
    z = s.matvec(x)
    assert np.array_equal(z[0], y[0]) and not z[1].any()
    assert np.array_equal(z[2], 2.0 ** 40 * y[0]) and np.array_equal(z[3], 2.0 ** -40 * y[0])
    assert _rel(2.0 ** 90 * z[4], y[0]) < 1e-5
    s.close()
    d.close()


# entries of one field over 2^40
@pytest.mark.parametrize("q", [5, 10])
def test_fields_with_a_wide_range(q):
    from paper_1807_03097_gb300 import Solver

    kw = dict(p=1, level_m=2, kappa=2.0, q=q, eta=1.6)
    s, d = Solver(G.torus(), precision=1, m2l_batch=2, **kw), Solver(G.torus(), precision=0, **kw)
    rng = np.random.default_rng(q)
    x = rng.standard_normal((8, s.ndof)) * 2.0 ** rng.integers(-40, 1, (8, s.ndof)) + 0j
    y = s.matvec(x)
    for r in range(8):
        assert _rel(y[r], d.matvec(x[r])) < 1e-5
    s.close()
    d.close()


# geometries in other units: the kernel's scale follows the distances; 2^-22 and 2^22: kappa outside
# [1e-6, 1e6], lengths not scaled by it
@pytest.mark.parametrize("unit", [2.0 ** -22, 2.0 ** -10, 2.0 ** 22])
def test_units_of_length(unit):
    from paper_1807_03097_gb300 import Solver

    kw = dict(p=1, level_m=2, kappa=2.0 / unit, q=5, eta=1.6, m2l_batch=2)
    s = Solver(G.sphere(radius=unit), precision=1, **kw)
    kw.pop("m2l_batch")
    d = Solver(G.sphere(radius=unit), precision=0, **kw)
    rng = np.random.default_rng(5)
    x = rng.standard_normal((8, s.ndof)) + 1j * rng.standard_normal((8, s.ndof))
    y = s.matvec(x)
    for r in range(0, 8, 3):
        assert _rel(y[r], d.matvec(x[r])) < 1e-5
    s.close()
    d.close()
