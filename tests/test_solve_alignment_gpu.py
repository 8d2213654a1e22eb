"""GPU test of fe_pcg_solve with u on an 8-byte boundary: the products of the start (u holds
an initial guess) and of the confirmation read u by 16-byte loads in the gather and
float-float kernels, so they must not be given such a u.

Bars: those of the other solver tests (relative residual 1e-8, solution 1e-6).
"""
import ctypes

import numpy as np
import pytest

from _util import ensure_lib, rel_l2

import oracle
from paper_1710_08679_gb300 import meshgen as mg

torch = pytest.importorskip("torch")

GATHER, GATHER_DF, DF_LEAN = 2, 3, 7


@pytest.mark.gpu
@pytest.mark.parametrize("solver", ["pcg64", "fcg_mixed"])
@pytest.mark.parametrize("variant", [GATHER, GATHER_DF, DF_LEAN])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("guess", [False, True])
def test_u_on_an_8_byte_boundary(solver, variant, shift, guess):
    ensure_lib()
    from paper_1710_08679_gb300 import fe
    R = 4
    m, _ = mg.crust_block(shape=(5, 3, 4), h=1000.0, jitter=0.15, seed=2)
    K = oracle.assemble(m)
    f = mg.random_vectors(m.n_nodes, R, seed=7) * m.free[:, None, :]
    ref = oracle.direct_solve(K, f)
    M = fe.Mesh.from_mesh(m)
    M.set_variant(R, "f64", variant, 16)
    F = torch.from_numpy(f).cuda()
    u = torch.zeros(F.numel() + shift, dtype=torch.float64, device="cuda")[shift:]
    assert u.data_ptr() % 16 == 8 * shift
    if guess:
        u.copy_(torch.from_numpy(ref * (1.0 + 1e-3 * mg.random_vectors(m.n_nodes, R, seed=8))).cuda().reshape(-1))
    o = fe.SolveOpts()
    fe.load().fe_solve_opts_default(ctypes.byref(o))
    o.solver, o.tol = fe.SOLVERS[solver], 1e-8
    stats = (fe.SolveStats * R)()
    torch.cuda.synchronize()
    st = fe.load().fe_pcg_solve(M.handle, R, F.data_ptr(), u.data_ptr(), ctypes.byref(o), stats, None)
    torch.cuda.synchronize()
    assert st == fe.FE_OK and all(s.relres <= 1e-8 for s in stats)
    assert rel_l2(u.view(F.shape).cpu().numpy(), ref) <= 1e-6
