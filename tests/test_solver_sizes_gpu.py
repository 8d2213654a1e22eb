"""GPU test of the solvers on both sides of the rule for the inner-loop passes with four
cases per thread: (nodes, R) just below and above it, with a number of four-case groups
that is a power of two or not, and blocks made smaller for the mesh.

Bar: the residual ||f - K u|| / ||f|| of every case, computed with the oracle's matrix, meets
the tolerance of the solve (1e-8; 1 % for the rounding of the stopping test's own product).
"""
import numpy as np
import pytest

from _util import ensure_lib

import oracle
from paper_1710_08679_gb300 import meshgen as mg

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("solver", ["fcg_mixed", "fcg_mg"])
@pytest.mark.parametrize("n,R", [(5, 64), (8, 16), (8, 20), (10, 8), (10, 12)])
def test_solve_at_the_four_case_rule(solver, n, R):
    ensure_lib()
    from paper_1710_08679_gb300 import fe
    m = mg.plain_box(n=n)
    K = oracle.assemble(m)
    f = mg.random_vectors(m.n_nodes, R, seed=70 + R) * m.free[:, None, :]
    u, stats, _ = fe.Mesh.from_mesh(m).solve(torch.from_numpy(f).cuda(), solver=solver, tol=1e-8)
    res = f - oracle.spmv(K, u.cpu().numpy())
    for r in range(R):
        assert stats[r]["relres"] <= 1e-8
        assert np.linalg.norm(res[:, r]) <= 1.01e-8 * np.linalg.norm(f[:, r]), r
