"""Mean error of the mixed form's far part (k_m2l_mma).  The tensor core shortens what it reads and what it
accumulates, so all contributions to a sum err to the same side; the mean is known and given back.  At low wavenumbers, where
the kernel's own phase errors are small, the product's far part must not be longer or shorter than the FP64 form's
by one unit of 2^-23 of every term, 8.6e-8 over evenly distributed logarithms (2^-23 / (2 ln 2)): the projection of
the error on the far part itself."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mk,p,m,kappa,q", [(G.sphere, 1, 1, 0.5, 6), (G.sphere, 1, 2, 0.5, 9), (G.cube, 2, 2, 0.5, 6),
                                            (G.sphere, 2, 3, 1.0, 6), (G.cube, 1, 3, 1.0, 6), (G.torus, 1, 2, 1.0, 4)],
                         ids=lambda v: getattr(v, "__name__", str(v)))
def test_far_part_is_not_shortened(mk, p, m, kappa, q):
    from paper_1807_03097_gb300 import Solver

    kw = dict(p=p, level_m=m, kappa=kappa, q=q, eta=1.6)
    s, d = Solver(mk(), precision=1, **kw), Solver(mk(), precision=0, **kw)
    assert s.nfar > 0
    rng = np.random.default_rng(1)
    x = rng.standard_normal((4, s.nsup)) + 1j * rng.standard_normal((4, s.nsup))
    far = np.stack([d.matvec_superspace(v) - d.near_apply(v) for v in x])
    err = np.stack([s.matvec_superspace(v) - s.near_apply(v) for v in x]) - far
    assert abs(np.vdot(far, err).real / np.vdot(far, far).real) < 8.6e-8
    s.close()
    d.close()
