"""Kept FP64 matrices in the plain form (k_m2l_f64_stored), which runs where it fits in half of the free memory and the
digits, four times as large at q = 1, do not: the rest of the device memory is held by another allocation.
Against evaluated entries; tolerance as between the two other forms (sums of at most 4e4 products in FP64)."""
import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu


def test_plain_matrices_where_digits_do_not_fit():
    torch = pytest.importorskip("torch")
    from paper_1807_03097_gb300 import Solver

    kw = dict(p=1, level_m=5, kappa=5.0, q=1, eta=1.6, precision=0)
    a = Solver(G.sphere(), m2l_store=1, **kw)
    rng = np.random.default_rng(67)
    x = rng.standard_normal(a.ndof) + 1j * rng.standard_normal(a.ndof)
    y = a.matvec(x)
    live, plain = a.device_bytes()[0], 256 * a.nfar
    # free memory as the second setup decides: between twice the plain matrices and twice the digits (4 plain)
    torch.cuda.synchronize()
    room = torch.cuda.mem_get_info()[0] - live - 4 * plain
    assert room > 0
    held = torch.empty(room, dtype=torch.uint8, device="cuda")
    b = Solver(G.sphere(), m2l_store=0, **kw)
    kept = b.device_bytes()[0] - live
    z = b.matvec(x)
    b.close()
    del held
    torch.cuda.empty_cache()
    assert plain <= kept < 1.2 * plain, (kept, plain)
    assert np.abs(y - z).max() / np.abs(y).max() < 3e-13
    c = Solver(G.sphere(), m2l_store=0, **kw)  # with the memory free: digits
    assert c.device_bytes()[0] - live > 3 * plain
    assert np.abs(y - c.matvec(x)).max() / np.abs(y).max() < 3e-13
    c.close()
    a.close()
