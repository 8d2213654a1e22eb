"""What users of this framework have it do: element-by-element (EBE) products, the coarse
level's products and transfers, element sensitivities and whole solves, through
paper_1710_08679_gb300.fe, on the meshes of the repository's configurations.

Every case is a mesh ("model", "nx", "ny", "nz": hexahedra, six 10-node tetrahedra each),
a number of load cases R and a kind of work:
  ebe       y = K x in FP32 (inner loops) or FP64 (outer loop, true residuals, plain CG);
  coarse    the level-1 (4-node) operator of the inner loops, assembled, FP32;
  transfer  restriction to level 1 and prolongation back, FP32;
  adjoint   element sensitivities of R state / adjoint pairs, FP64;
  solve     fe_pcg_solve from a zero guess, FP64 in and out.
The mesh handle and the tuner's kernel choice (Mesh.tune) are what a program makes once
and keeps for every product and solve on that mesh, so handles are shared by the states of
one mesh; right-hand sides and vectors are made from the seed.
"""
import functools
import math

import numpy as np
import torch

from paper_1710_08679_gb300 import fe
from paper_1710_08679_gb300 import meshgen as mg

DTYPES = {"f32": torch.float32, "f64": torch.float64}


def _ebe(name, model, n, R, dtype):
    return dict(name=name, kind="ebe", model=model, nx=n[0], ny=n[1], nz=n[2], R=R, dtype=dtype)


def listed():
    crust, box, slab = (70, 70, 35), (8, 8, 8), (41, 33, 18)
    dim = dict(nx=70, ny=70, nz=35)
    return [
        # one case on the 15k-DOF box: launch and latency bound, as in small inversions' inner loops
        _ebe("ebe_f32_r1_box8", "box", box, 1, "f32"),
        # the plain FP64 block-Jacobi CG of one double couple on the same box (a whole call)
        dict(name="solve_pcg64_r1_box8", kind="solve", model="box", nx=8, ny=8, nz=8, R=1, solver="pcg64", tol=1e-8),
        # an inner product of one case (the adjoint solve's) on the 83k-element box of the gradient workload
        _ebe("ebe_f32_r1_box24", "box", (24, 24, 24), 1, "f32"),
        # the backward step of that workload: sensitivities of all elements
        dict(name="adjoint_r16_box24", kind="adjoint", model="box", nx=24, ny=24, nz=24, R=16),
        # batch sizes that are no power of two: the last batch of a run, a dozen slips, five gauges
        _ebe("ebe_f32_r12_slab", "crust", slab, 12, "f32"),
        _ebe("ebe_f64_r5_slab", "crust", slab, 5, "f64"),
        # the 4.2M-DOF crust block: inner product, outer product and true residual of a 16-case batch,
        # the single-case FP64 product of the plain solver and of late confirmations
        _ebe("ebe_f32_r16_crust", "crust", crust, 16, "f32"),
        _ebe("ebe_f64_r16_crust", "crust", crust, 16, "f64"),
        _ebe("ebe_f64_r1_crust", "crust", crust, 1, "f64"),
        # level-1 operator (some 400 applications a solve) and transfers of that batch
        dict(name="coarse_r16_crust", kind="coarse", model="crust", R=16, **dim),
        dict(name="transfer_r16_crust", kind="transfer", model="crust", R=16, **dim),
        # the batched two-level mixed-precision solve of 16 slip distributions (a whole call)
        dict(name="solve_mg_r16_crust", kind="solve", model="crust", R=16, solver="fcg_mg", tol=1e-10, **dim),
    ]


def _spread(rng, lo, hi):
    return lo * math.exp(rng.random() * math.log(hi / lo))


def draw(rng):
    kind = rng.choice(["ebe", "ebe", "ebe", "ebe", "coarse", "transfer", "adjoint", "solve"])
    hexes = _spread(rng, 500, 171500 if kind == "ebe" else 40000)
    model = rng.choice(["crust", "crust", "box"])
    aspect = (1.0, 1.0) if model == "box" else (rng.uniform(0.6, 1.0), rng.uniform(0.4, 0.7))
    n = (hexes / (aspect[0] * aspect[1])) ** (1.0 / 3.0)
    nx, ny, nz = max(4, int(n)), max(4, int(n * aspect[0])), max(4, int(n * aspect[1]))
    c = dict(kind=kind, model=model, nx=nx, ny=ny, nz=nz, R=max(1, int(_spread(rng, 1, 32.99))))
    if kind == "ebe":
        c["dtype"] = rng.choice(["f32", "f64"])
    if kind == "solve":
        # FP64 CG runs to 1e-8; its iterates have no FP32 part, unlike the two-level solver's
        if rng.random() < 0.5:
            k = rng.randint(5, 8)
            c.update(model="box", nx=k, ny=k, nz=k, R=rng.randint(1, 8), solver="pcg64", tol=1e-8)
        else:
            c.update(model="crust", nx=max(nx, 24), ny=max(ny, 20), nz=max(nz, 12), R=rng.choice([4, 8, 12, 16]),
                     solver="fcg_mg", tol=1e-10)
    return c


# ---------------------------------------------------------------------------
# meshes and handles (kept by a program for as long as it works on the mesh)
# ---------------------------------------------------------------------------
class _Handle:
    def __init__(self, model, nx, ny, nz):
        self.iface = None
        if model == "box":   # the two-layer 8 km box, sources inside
            self.mesh = mg.box_mesh((nx, ny, nz), (8000.0, 8000.0, 8000.0), jitter=0.10, seed=0)
            mg.set_two_layers(self.mesh, 4000.0)
        else:                # the four-layer crust block of 1 km hexahedra with a dipping interface
            self.mesh, self.iface = mg.crust_block((nx, ny, nz))
        self.gpu = fe.Mesh.from_mesh(self.mesh)
        self.tuned = set()
        self.sources = None

    def tune(self, R, dtype):
        if (R, dtype) not in self.tuned:
            self.gpu.tune(R, dtype)
            self.tuned.add((R, dtype))

    def base_sources(self):
        """Sixteen unit sources f [N, 16, 3]: dip-slip patches on the interface of a crust block,
        double couples in a box."""
        if self.sources is None:
            m = self.mesh
            if self.iface is None:
                lx, ly, lz = m.lattice_shape()
                at = [(a, b) for a in (3, 5, 7, 9) for b in (3, 5, 7, 9)]
                f = np.stack([mg.double_couple(m, (lx * a // 12, ly * b // 12, lz // 2), 1e12) for a, b in at], axis=1)
                self.sources = torch.from_numpy(f).cuda()
            else:
                space = 4000.0 * min(1.0, m.shape[0] / 70.0, m.shape[1] / 70.0)
                out = torch.zeros((m.n_nodes, 16, 3), dtype=torch.float64, device="cuda")
                for r, c in enumerate(mg.patch_grid_cases(m, self.iface, spacing=space)):
                    s = torch.from_numpy(c.slip).cuda()[:, None, :]
                    out[:, r] = -_product(m, s, elems=c.elems)[:, 0]
                self.sources = out * torch.from_numpy(m.free).cuda()[:, None, :]
        return self.sources


@functools.lru_cache(maxsize=4)
def _handle(model, nx, ny, nz):
    return _Handle(model, nx, ny, nz)


def _of(case):
    return _handle(case["model"], case["nx"], case["ny"], case["nz"])


def _normal(shape, seed, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _vectors(case, seed):
    """The inputs of a case, from the seed alone."""
    h, R, kind = _of(case), case["R"], case["kind"]
    n = h.mesh.n_nodes
    if kind == "ebe":
        return [_normal((n, R, 3), seed, DTYPES[case["dtype"]])]
    if kind == "coarse":
        return [_normal((h.gpu.coarse_info()[0], R, 3), seed, torch.float32)]
    if kind == "transfer":
        return [_normal((n, R, 3), seed, torch.float32)]
    if kind == "adjoint":
        return [_normal((n, R, 3), seed), _normal((n, R, 3), seed + 1000003)]
    # solve: every case a distribution of slip (or of couples) over the sixteen unit sources
    g = torch.Generator(device="cuda").manual_seed(seed)
    amount = torch.rand((16, R), generator=g, device="cuda", dtype=torch.float64) ** 4
    return [torch.einsum("nsc,sr->nrc", h.base_sources(), amount).contiguous()]


def prepare(case, seed):
    h, R = _of(case), case["R"]
    if case["kind"] == "ebe":
        h.tune(R, case["dtype"])
    elif case["kind"] == "solve":
        h.tune(R, "f64")
        h.tune(1, "f64")
        if case["solver"] != "pcg64":
            h.tune(R, "f32")
    return dict(case=case, mesh=h.gpu, x=_vectors(case, seed))


def run(state):
    case, m, x = state["case"], state["mesh"], state["x"]
    kind = case["kind"]
    if kind == "ebe":
        return m.ebe(x[0])
    if kind == "coarse":
        return m.coarse_apply(x[0])
    if kind == "transfer":
        r4 = m.coarse_restrict(x[0])
        return r4, m.coarse_prolong(r4)
    if kind == "adjoint":
        return m.adjoint_grad(x[0], x[1])
    return m.solve(x[0], solver=case["solver"], tol=case["tol"])[0]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    nx, ny, nz, R, kind = case["nx"], case["ny"], case["nz"], case["R"], case["kind"]
    E, N = 6 * nx * ny * nz, (2 * nx + 1) * (2 * ny + 1) * (2 * nz + 1)
    N4 = (nx + 1) * (ny + 1) * (nz + 1)
    vec4, vec8 = 12.0 * N * R, 24.0 * N * R

    def ebe(s):   # element data and coordinates once, x read and y written once; multiply-add = 2
        return dict(bytes=E * (40.0 + 2 * s) + N * 3.0 * s + 2 * N * 3.0 * R * s, flops=E * (774.0 * R + 100.0))

    if kind == "ebe":
        return ebe(4 if case["dtype"] == "f32" else 8)
    if kind == "coarse":   # about 15 blocks of 3x3 a row and their columns
        return dict(bytes=15.0 * N4 * 40.0 + 2 * 12.0 * N4 * R, flops=15.0 * N4 * 18.0 * R)
    if kind == "transfer":
        return dict(bytes=2 * vec4 + 2 * 12.0 * N4 * R, flops=6.0 * N * R * 2)
    if kind == "adjoint":
        return dict(bytes=E * 56.0 + N * 24.0 + 2 * vec8 + E * 8.0, flops=E * (834.0 * R + 100.0))
    if case["solver"] == "pcg64":   # some 170 steps on the 8^3 box: a product and eleven vector passes each
        steps = 20.0 * max(nx, ny, nz)
        w = ebe(8)
        return dict(bytes=steps * (w["bytes"] + 9 * vec8), flops=steps * (w["flops"] + 60.0 * N * R))
    # two-level: per outer step some 3.5 level-0 steps and 26 level-1 steps
    a, b, outer = ebe(8), ebe(4), 18.0
    c1 = 15.0 * N4 * 40.0 + 12 * 12.0 * N4 * R
    return dict(bytes=outer * (a["bytes"] + 8 * vec8 + 3.5 * (b["bytes"] + 9 * vec4) + 26 * c1),
                flops=outer * (a["flops"] + 3.5 * b["flops"] + 26 * 15.0 * N4 * 18.0 * R))


# ---------------------------------------------------------------------------
# the same outputs in 64 bits, by plain torch
# ---------------------------------------------------------------------------
_EDGES = ((0, 1), (1, 2), (2, 0), (0, 3), (1, 3), (2, 3))


def _gradients(m, el):
    """Shape-function gradients [4 points, e, 10, 3], weights [e] and Lame constants of elements `el`:
    the 4-point rule, exact for the products of linear gradients of a straight-sided element."""
    conn = torch.from_numpy(np.ascontiguousarray(m.conn[el])).cuda().long()
    xyz = torch.from_numpy(m.coords).cuda()[conn[:, :4]]
    d = xyz[:, 1:] - xyz[:, :1]
    inv = torch.linalg.inv(d)                       # inv[:, c, j]: d L_{j+1} / d x_c
    g = torch.cat([-inv.sum(2, keepdim=True), inv], dim=2).transpose(1, 2)   # [e, 4, 3]
    vol = torch.linalg.det(d).abs() / 6.0
    p, q = (5.0 + 3.0 * math.sqrt(5.0)) / 20.0, (5.0 - math.sqrt(5.0)) / 20.0
    pts = []
    for k in range(4):
        L = [p if j == k else q for j in range(4)]
        rows = [(4.0 * L[a] - 1.0) * g[:, a] for a in range(4)]
        rows += [4.0 * (L[a] * g[:, b] + L[b] * g[:, a]) for a, b in _EDGES]
        pts.append(torch.stack(rows, dim=1))
    E = torch.from_numpy(np.ascontiguousarray(m.young[el])).cuda()
    nu = torch.from_numpy(np.ascontiguousarray(m.poisson[el])).cuda()
    return conn, torch.stack(pts), vol / 4.0, E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))


def _stress(grad, lam, mu):
    """Stress [e, i, j, r] of displacement gradients [e, i, j, r]."""
    tr = torch.einsum("eiir->er", grad)
    s = mu[:, None, None, None] * (grad + grad.transpose(1, 2))
    s += torch.eye(3, device=grad.device, dtype=grad.dtype)[None, :, :, None] * (lam[:, None] * tr)[:, None, None, :]
    return s


def _chunks(m, R, elems):
    elems = np.arange(m.n_elem) if elems is None else elems
    step = max(1, 600000 // R)
    for k in range(0, len(elems), step):
        yield elems[k:k + step]


def _product(m, x, elems=None):
    """sum over elements of Q K_e Q^T x (no boundary conditions), x [N, R, 3] float64."""
    N, R, _ = x.shape
    y = torch.zeros_like(x)
    for el in _chunks(m, R, elems):
        conn, B, w, lam, mu = _gradients(m, el)
        u = x[conn].transpose(2, 3).reshape(len(el), 10, 3 * R)           # [e, a, (i, r)]
        f = torch.zeros_like(u)
        for k in range(4):
            grad = torch.bmm(B[k].transpose(1, 2), u).reshape(len(el), 3, 3, R).transpose(1, 2)   # [e, i, j, r]
            s = _stress(grad, lam, mu) * w[:, None, None, None]
            f += torch.bmm(B[k], s.transpose(1, 2).reshape(len(el), 3, 3 * R))
        y.index_add_(0, conn.reshape(-1), f.reshape(len(el) * 10, 3, R).transpose(1, 2).contiguous())
    return y


def _sensitivity(m, u, lam_u):
    out = torch.zeros(m.n_elem, dtype=torch.float64, device="cuda")
    R = u.shape[1]
    for el in _chunks(m, R, None):
        conn, B, w, lam, mu = _gradients(m, el)
        v = [t[conn].transpose(2, 3).reshape(len(el), 10, 3 * R) for t in (u, lam_u)]
        acc = 0.0
        for k in range(4):
            g = [torch.bmm(B[k].transpose(1, 2), t).reshape(len(el), 3, 3, R).transpose(1, 2) for t in v]
            acc = acc + w * (_stress(g[0], lam, mu) * g[1]).sum((1, 2, 3))
        out[torch.from_numpy(el).cuda()] = -acc
    return out


def _masked_product(m, x):
    P = torch.from_numpy(m.free).cuda().double()[:, None, :]
    return P * _product(m, P * x) + (1 - P) * x


def _level1(m):
    """The corner nodes of the mesh and, per node of the mesh, its two coarse ends."""
    vertex = np.unique(m.conn[:, :4])
    new = np.full(m.n_nodes, -1)
    new[vertex] = np.arange(len(vertex))
    ends = np.stack([new, new], axis=1)
    for q, (a, b) in enumerate(_EDGES):
        ends[m.conn[:, 4 + q]] = new[m.conn[:, [a, b]]]
    return torch.from_numpy(vertex).cuda(), torch.from_numpy(ends).cuda()


def _dense(m):
    n = 3 * m.n_nodes
    K = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    eye = torch.eye(3, device="cuda", dtype=torch.float64)
    for el in _chunks(m, 30, None):
        conn, B, w, lam, mu = _gradients(m, el)
        ke = 0.0
        for k in range(4):
            gg = torch.einsum("eai,ebj->eaibj", B[k], B[k])
            tr = torch.einsum("eai,ebi->eab", B[k], B[k])
            ke = ke + w[:, None, None, None, None] * (
                lam[:, None, None, None, None] * gg + mu[:, None, None, None, None] * gg.permute(0, 1, 4, 3, 2)
                + mu[:, None, None, None, None] * tr[:, :, None, :, None] * eye[None, None, :, None, :])
        dof = (3 * conn[:, :, None] + torch.arange(3, device="cuda")).reshape(len(el), 30)
        K.view(-1).index_add_(0, (dof[:, :, None] * n + dof[:, None, :]).reshape(-1), ke.reshape(-1))
    return K


def exact(case, seed):
    m, kind = _of(case).mesh, case["kind"]
    x = [v.double() for v in _vectors(case, seed)]
    if kind == "ebe":
        return _masked_product(m, x[0])
    if kind == "adjoint":
        P = torch.from_numpy(m.free).cuda().double()[:, None, :]
        return _sensitivity(m, P * x[0], P * x[1])
    if kind in ("coarse", "transfer"):
        vertex, ends = _level1(m)
        P = torch.from_numpy(m.free).cuda().double()[:, None, :]
        P4 = P[vertex]

        def up(v4):
            return P * 0.5 * (v4[ends[:, 0]] + v4[ends[:, 1]])

        def down(v):
            out = torch.zeros((len(vertex),) + v.shape[1:], dtype=torch.float64, device="cuda")
            out.index_add_(0, ends[:, 0], 0.5 * v)
            return P4 * out.index_add_(0, ends[:, 1], 0.5 * v)

        if kind == "transfer":
            r4 = down(x[0])
            return r4, up(r4)
        # the level-1 operator is P1^T K P1 on straight-sided elements (linear fields are in both spaces)
        v = 0.5 * ((P4 * x[0])[ends[:, 0]] + (P4 * x[0])[ends[:, 1]])
        return down(_product(m, v)) + (1 - P4) * x[0]
    if m.n_nodes > 5000:
        return None
    free = torch.from_numpy(m.free.reshape(-1)).cuda().bool()
    K = _dense(m)[free][:, free]
    f = x[0].transpose(1, 2).reshape(-1, case["R"])
    u = torch.zeros_like(f)
    u[free] = torch.cholesky_solve(f[free], torch.linalg.cholesky(K))
    return u.reshape(m.n_nodes, 3, case["R"]).transpose(1, 2).contiguous()
