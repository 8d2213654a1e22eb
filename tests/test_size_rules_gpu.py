"""GPU parity, against the CPU oracle, of the kernels that are chosen by the size of a
call: the FP64 direct product on both sides of its rule (four lanes per element, one
lane per element and share of the cases), the sensitivities with an element's cases
spread over lanes, the warp-specialised product for R that is no power of two, the
4-case passes of the inner loops and the PCG iterations run as one device-side loop.

Bars: those of the other parity tests (FP64 products 1e-12, FP32 products 2e-6 per
case, sensitivities 1e-12, solutions 1e-6 from a solve to 1e-8).
"""
import numpy as np
import pytest

from _util import ensure_lib, rel_l2

import oracle
from paper_1710_08679_gb300 import meshgen as mg

torch = pytest.importorskip("torch")

TOL64, TOL32 = 1e-12, 2e-6
DIRECT, WS, WS2 = 0, 6, 8

MESHES = {
    "box1": lambda: mg.plain_box(n=1, jitter=0.0),
    "ragged": lambda: mg.crust_block(shape=(5, 3, 4), h=1000.0, jitter=0.15, seed=2)[0],
    "box8": lambda: mg.plain_box(),
    "crust20": lambda: mg.crust_block(shape=(20, 20, 10), h=1000.0, jitter=0.15, seed=5)[0],
}


@pytest.fixture(scope="module", params=list(MESHES))
def case(request):
    ensure_lib()
    from paper_1710_08679_gb300 import fe
    m = MESHES[request.param]()
    return m, oracle.assemble(m), fe.Mesh.from_mesh(m)


def cuda(a, dtype=torch.float64):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dtype).cuda()


# from 6 items (box1, R = 1) over one warp per SM sub-partition (box8) to many (crust20)
@pytest.mark.gpu
@pytest.mark.parametrize("R", [1, 2, 5, 7, 17])
def test_direct_fp64_product(case, R):
    m, K, M = case
    x = mg.random_vectors(m.n_nodes, R, seed=40 + R)
    M.set_variant(R, "f64", DIRECT, 48)
    y = M.ebe(cuda(x)).cpu().numpy()
    ref = oracle.spmv(K, x)
    for r in range(R):
        assert rel_l2(y[:, r], ref[:, r]) <= TOL64, r
    fixed = m.free == 0
    for r in range(R):   # constrained DOFs: (I - P) x
        assert np.array_equal(y[:, r][fixed], x[:, r][fixed])


# even R: two cases per thread
@pytest.mark.gpu
@pytest.mark.parametrize("R", [1, 2, 5, 6, 14, 30])
def test_direct_fp32_product(case, R):
    m, K, M = case
    x = mg.random_vectors(m.n_nodes, R, seed=50 + R).astype(np.float32).astype(np.float64)
    M.set_variant(R, "f32", DIRECT, 48)
    y = M.ebe(cuda(x, torch.float32)).double().cpu().numpy()
    ref = oracle.spmv(K, x)
    for r in range(R):
        assert rel_l2(y[:, r], ref[:, r]) <= TOL32, r
    fixed = m.free == 0
    for r in range(R):
        assert np.array_equal(y[:, r][fixed], x[:, r][fixed])


@pytest.mark.gpu
@pytest.mark.parametrize("R", [1, 2, 5, 16, 33])
def test_sensitivities(case, R):
    m, _, M = case
    u = mg.random_vectors(m.n_nodes, R, seed=60 + R)
    lam = mg.random_vectors(m.n_nodes, R, seed=160 + R)
    g = M.adjoint_grad(cuda(u), cuda(lam)).cpu().numpy()
    assert rel_l2(g, oracle.adjoint_grad(m, u, lam)) <= TOL64


@pytest.mark.gpu
@pytest.mark.parametrize("R,variant,tile", [(12, WS, 32), (12, WS2, 16), (20, WS, 16), (24, WS, 16), (24, WS2, 8),
                                            (28, WS, 16)])
def test_warp_specialised_product(case, R, variant, tile):
    m, K, M = case
    x = mg.random_vectors(m.n_nodes, R, seed=80 + R).astype(np.float32).astype(np.float64)
    M.set_variant(R, "f32", variant, tile)
    assert M.get_variant(R, "f32") == (variant, tile)
    y = M.ebe(cuda(x, torch.float32))
    M.device_status()   # no bounded wait of the kernel gave up
    y = y.double().cpu().numpy()
    ref = oracle.spmv(K, x)
    for r in range(R):
        assert rel_l2(y[:, r], ref[:, r]) <= TOL32, r


# R = 12, 20: groups of 4 cases whose number is no power of two; 5 and 6: the one- and
# two-case passes; 32: the largest. `shift`: u on an 8-byte boundary only.
@pytest.mark.gpu
@pytest.mark.parametrize("R,shift", [(4, 0), (5, 0), (6, 0), (6, 1), (12, 0), (20, 0), (32, 0)])
@pytest.mark.parametrize("solver", ["fcg_mixed", "fcg_mg"])
def test_inner_and_outer_passes(solver, R, shift):
    ensure_lib()
    import ctypes

    from paper_1710_08679_gb300 import fe
    m = MESHES["ragged"]()
    K = oracle.assemble(m)
    f = mg.random_vectors(m.n_nodes, R, seed=7) * m.free[:, None, :]
    f[:, R - 1] = 0.0   # a case that is finished at the start
    M = fe.Mesh.from_mesh(m)
    F = cuda(f)
    u = torch.zeros(F.numel() + shift, dtype=torch.float64, device="cuda")[shift:]
    o = fe.SolveOpts()
    fe.load().fe_solve_opts_default(ctypes.byref(o))
    o.solver, o.tol = fe.SOLVERS[solver], 1e-8
    stats = (fe.SolveStats * R)()
    torch.cuda.synchronize()
    st = fe.load().fe_pcg_solve(M.handle, R, F.data_ptr(), u.data_ptr(), ctypes.byref(o), stats, None)
    torch.cuda.synchronize()
    assert st == fe.FE_OK
    u = u.view(F.shape).cpu().numpy()
    ref = oracle.direct_solve(K, f)
    for r in range(R - 1):
        assert stats[r].relres <= 1e-8 and rel_l2(u[:, r], ref[:, r]) <= 1e-6, r
    assert not np.any(u[:, R - 1])


# cases that converge one after the other leave and re-enter the device-side loop
@pytest.mark.gpu
@pytest.mark.parametrize("R", [1, 3, 6])
def test_pcg_loop_matches_single_iterations(R):
    ensure_lib()
    from paper_1710_08679_gb300 import fe
    m = MESHES["ragged"]()
    K = oracle.assemble(m)
    f = mg.random_vectors(m.n_nodes, R, seed=9) * m.free[:, None, :]
    ref = oracle.direct_solve(K, f)
    M = fe.Mesh.from_mesh(m)
    outer = []
    for use_graph in (True, False):
        u, stats, _ = M.solve(cuda(f), solver="pcg64", tol=1e-8, use_graph=use_graph)
        assert rel_l2(u.cpu().numpy(), ref) <= 1e-6
        assert all(s["relres"] <= 1e-8 for s in stats)
        outer.append([s["outer"] for s in stats])
    assert all(abs(a - b) <= 1 for a, b in zip(*outer)), outer   # sums in another order
    _, stats, st = M.solve(cuda(f), solver="pcg64", tol=1e-8, max_outer=5, raise_on_fail=False)
    assert st == fe.FE_ENOCONV and all(s["outer"] == 5 for s in stats)   # the cap ends the loop
