"""GPU test of the float-float FP64 products' accuracy (both kernels): compiled for the device
the element routine must keep the error terms that test_float_float_cpu.py checks, and the
node sums theirs.

Bar: 2^-48 ||(|K| |x|)||, one unit in the last of the 48 bits of the products that a result
sums up. The products' rounding errors, several of that size each and independent of each
other, add up to a third of the bar for random vectors and a ninth of it for translated
fields (evaluated on the host in the same arithmetic); an error term left out exceeds it.
"""
import numpy as np
import pytest

from _util import ensure_lib

import oracle
from paper_1710_08679_gb300 import meshgen as mg

torch = pytest.importorskip("torch")

GATHER_DF, DF_LEAN = 3, 7


@pytest.mark.gpu
@pytest.mark.parametrize("variant", [GATHER_DF, DF_LEAN])
@pytest.mark.parametrize("R", [2, 16])
@pytest.mark.parametrize("shape", [(5, 3, 4), (12, 10, 6)])
def test_error_of_the_float_float_products(shape, R, variant):
    ensure_lib()
    from paper_1710_08679_gb300 import fe
    m, _ = mg.crust_block(shape=shape, h=1000.0, jitter=0.15, seed=6)
    K = oracle.assemble(m)
    absK = abs(K.to_scipy())
    M = fe.Mesh.from_mesh(m)
    M.set_variant(R, "f64", variant, 12)
    rng = np.random.default_rng(R)
    scale = m.coords.max(axis=0)
    fields = {"random": mg.random_vectors(m.n_nodes, R, seed=90 + R),
              "translated": 1.0 + np.einsum("ni,irj->nrj", m.coords / scale, 1e-2 * rng.standard_normal((3, R, 3)))}
    for name, x in fields.items():
        x = np.ascontiguousarray(x * m.free[:, None, :])
        y = M.ebe(torch.from_numpy(x).cuda()).cpu().numpy()
        ref = oracle.spmv(K, x)
        for r in range(R):
            bar = 2.0 ** -48 * np.linalg.norm(absK @ np.abs(x[:, r].ravel()))
            assert np.linalg.norm(y[:, r] - ref[:, r]) <= bar, (name, r)
