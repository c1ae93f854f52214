"""Lockstep solves of independent contexts on several host threads.  Their products take other amounts of
dynamic shared memory (blocks of 18 x 18 and 32 x 32 with 4, 8, 12 and 16 right-hand sides), and the limit that a
launch is checked against belongs to the kernel, not to a context: a thread must never lower it under
another's launch.  Every solve ends by its iteration limit, with the same iterates as alone."""
import threading

import numpy as np
import pytest

from workloads import geometry as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,counts", [(2, (8, 16, 12, 8)), (3, (4, 8, 4, 8)), (2, (8, 16) * 6)])
def test_solves_on_several_threads(p, counts):
    from paper_1807_03097_gb300 import Solver

    solvers = [Solver(G.sphere(), p=p, level_m=1, kappa=1.0, q=3, eta=1.6, precision=1, gmres_tol=1e-30,
                      gmres_restart=10, gmres_maxit=200) for _ in counts]
    b = [s.rhs(*G.plane_waves(r, 3)) for s, r in zip(solvers, counts)]
    alone = [s.solve(v) for s, v in zip(solvers, b)]
    failed, start = [], threading.Barrier(len(counts))

    def work(i):
        start.wait()
        try:
            for _ in range(8):
                x, info, st = solvers[i].solve(b[i])
                assert st == alone[i][2] and np.array_equal(x, alone[i][0])
        except Exception as e:  # noqa: BLE001
            failed.append((counts[i], str(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(counts))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[0]
    for s in solvers:
        s.close()
