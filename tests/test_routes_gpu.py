"""GPU parity of launches that the other tests do not reach: products recorded in a caller's
graph (there the product kernels are ordinary launches behind the zero pass), the level-1
product with one block of a row in flight, and the smallest tile of the warp-specialised
kernel for 12 cases. Bars: those of the other parity tests.
"""
import numpy as np
import pytest

from _util import ensure_lib, rel_l2

import oracle
from paper_1710_08679_gb300 import meshgen as mg

torch = pytest.importorskip("torch")

TOL64, TOL32 = 1e-12, 2e-6
DIRECT, GATHER, WS = 0, 2, 6


def box(n):
    ensure_lib()
    from paper_1710_08679_gb300 import fe
    m = mg.plain_box(n=n)
    return m, fe.Mesh.from_mesh(m)


@pytest.mark.gpu
@pytest.mark.parametrize("R,dtype,variant", [(1, "f32", DIRECT), (6, "f32", DIRECT), (1, "f64", DIRECT),
                                             (5, "f64", DIRECT), (4, "f64", GATHER), (16, "f32", WS)])
def test_product_in_a_callers_graph(R, dtype, variant):
    m, M = box(8)
    K = oracle.assemble(m)
    M.set_variant(R, dtype, variant, 32)
    tdt = torch.float32 if dtype == "f32" else torch.float64
    x = torch.zeros((m.n_nodes, R, 3), dtype=tdt, device="cuda")
    y = torch.empty_like(x)
    M.ebe(x, out=y)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        M.ebe(x, out=y)
    for seed in (1, 2):
        h = torch.from_numpy(mg.random_vectors(m.n_nodes, R, seed=seed)).to(tdt)
        x.copy_(h)
        g.replay()
        torch.cuda.synchronize()
        assert rel_l2(y.double().cpu().numpy(), oracle.spmv(K, h.double().numpy())) <= \
            (TOL32 if dtype == "f32" else TOL64)
    M.device_status()


@pytest.mark.gpu
@pytest.mark.parametrize("R", [16, 60, 64])
def test_level1_product_on_both_sides_of_its_rule(R):
    ensure_lib()
    from paper_1710_08679_gb300 import fe
    m, _ = mg.crust_block(shape=(28, 24, 14), h=1000.0, jitter=0.15, seed=5)
    cm = oracle.coarse_mesh(m)
    x = mg.random_vectors(cm.vertex.size, R, seed=R).astype(np.float32)
    y = fe.Mesh.from_mesh(m).coarse_apply(torch.from_numpy(x).cuda()).double().cpu().numpy()
    assert rel_l2(y, oracle.spmv(oracle.assemble4(cm), x.astype(np.float64))) <= TOL32


@pytest.mark.gpu
def test_smallest_warp_specialised_tile_for_12_cases():
    m, M = box(8)
    x = mg.random_vectors(m.n_nodes, 12, seed=3).astype(np.float32)
    M.set_variant(12, "f32", WS, 16)
    assert M.get_variant(12, "f32") == (WS, 16)
    y = M.ebe(torch.from_numpy(x).cuda())
    M.device_status()
    assert rel_l2(y.double().cpu().numpy(), oracle.spmv(oracle.assemble(m), x.astype(np.float64))) <= TOL32
