"""Kernels chosen by size, at the sizes where they change shape, against the oracle.

* the residual's penalty with a velocity per surface point (a warp per host element): elements
  hosting fewer than 8, a few and several hundred points, slots and atomics.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.oracle import OracleMesh
from paper_2009_00706_gb300 import _lib, api
from paper_2009_00706_gb300 import inputs as I

C = (0.5, 0.5, 0.5)


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _lib.build()
    return torch.device("cuda:0")


def T(a, dev):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dev)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def pair(tri, level, radius=0.2, lmax=2):
    reg = [I.Region(I.REGION_SPHERE_BAND, level, (*C, radius, 0.05))]
    args = ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), 3, reg, tri, lmax)
    return api.Mesh(*args), OracleMesh(*args)


# float64 sums of at most a few hundred terms of one sign: well below 1e-12 of the result
TOL64 = 1e-12


@pytest.mark.parametrize("triangles,level", [(0, 5), (2, 4), (4, 4)])
@pytest.mark.parametrize("deterministic", [True, False])
def test_penalty_with_point_velocities(dev, triangles, level, deterministic):
    g, o = pair(I.icosphere(triangles, 0.2, C, 1e-3, 3), level)
    g.deterministic(deterministic)
    sq = g.surface_points()
    per = np.unique(sq[:, 8], return_counts=True)[1]
    assert {0: per.min() < 8, 2: per.max() > 8, 4: per.max() > 64}[triangles]
    vel = 0.3 * np.sin(7.0 * sq[:, :3] + np.array([0.0, 1.0, 2.0]))
    ph = I.Physics(mu=0.5, dt=1.0, scheme=I.SCHEME_CN, g=(0.1, -0.2, 0.05))   # the penalty dominates
    u, up, _ = I.state(g.n_nodes, 9)
    o.set_surface_velocity(0.3 * np.sin(7.0 * o.surface_points()[:, :3] + np.array([0.0, 1.0, 2.0])))
    try:
        want = o.residual_jvp(ph, u, up, v=up)[0]
    finally:
        o.set_surface_velocity(None)
    got = g.residual(ph, T(u, dev), T(up, dev), g_points=T(vel, dev)).cpu().numpy()
    assert rel(got, want) <= TOL64


# ---- the network: row counts around the tiles of 16, 32 and 64 rows and where the tile changes,
# odd output edges and inputs without 16-byte rows ----
def _mlp64(p, X):
    W1, b1, W2, b2, W3, b3 = p
    r = lambda a: a.to(torch.bfloat16).double()
    h1 = r((r(X) @ r(W1).T + b1).clamp_min(0))
    h2 = r((h1 @ r(W2).T + b2).clamp_min(0))
    return h1, h2, h2 @ r(W3).T + b3


def _params(net, dev):
    return [T(q, dev) for q in net.unpack(net.params())]


@pytest.mark.parametrize("rows", [1, 15, 17, 63, 64, 4863, 4864, 4865, 19455, 19457])
@pytest.mark.parametrize("shape", [(1027, 1024, 1040, 0), (45, 72, 45, 0), (64, 8, 67, 1)])
def test_mlp_forward_rows(dev, rows, shape):
    nin, nout, ldx, shift = shape
    net = api.Mlp(n_in=nin, n_out=nout, seed=5)
    torch.manual_seed(rows)
    X = torch.randn(rows * ldx + shift, device=dev)[shift:].view(rows, ldx)
    _, _, want = _mlp64(_params(net, dev), X[:, :nin].double())
    got = net.forward(X).double()
    # what is left is float32 sums and the activations they round to the other bf16 neighbour (2^-8)
    assert float((got - want).norm() / want.norm()) <= 2e-3


@pytest.mark.parametrize("rows,batch", [(130, 130), (257, 64), (2048, 1000)])
@pytest.mark.parametrize("nin,nout", [(1027, 1024), (45, 72)])
def test_mlp_gradient_rows(dev, rows, batch, nin, nout):
    net = api.Mlp(n_in=nin, n_out=nout, seed=6)
    torch.manual_seed(rows)
    X, Y = torch.randn(rows, nin, device=dev), torch.randn(rows, nout, device=dev)
    p = _params(net, dev)
    r = lambda a: a.to(torch.bfloat16).double()
    h1, h2, out = _mlp64(p, X.double())
    e = out - Y.double()
    dy = r(e / rows)
    d2 = r((dy @ r(p[4])) * (h2 > 0))
    d1 = r((d2 @ r(p[2])) * (h1 > 0))
    want = [d1.T @ r(X.double()), d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0)]
    loss, g = net.gradient(X, Y)
    # bf16 neighbours of the activations and errors, at most two roundings deep
    assert abs(loss - float((e * e).sum()) / (2 * rows)) <= 1e-3 * loss
    for k, (a, b) in enumerate(zip(net.unpack(g), want)):
        assert float((T(a, dev) - b).norm() / b.norm()) <= 1e-2, k
    first = net.train(X, Y, epochs=1, batch=batch, lr=1e-3)[0]
    assert net.train(X, Y, epochs=8, batch=batch, lr=1e-3)[-1] < first


# ---- float64 Intercepted elements: a block's four parts of 32 points at a time, from elements with a
# few points (less than one part) to several rounds, slots and atomics, all fields in use ----
@pytest.mark.parametrize("lmax", [0, 1, 3])
@pytest.mark.parametrize("scheme", [I.SCHEME_BE, I.SCHEME_CN, I.SCHEME_BDF2])
def test_float64_cut_elements(dev, lmax, scheme):
    g, o = pair(I.icosphere(2, 0.2, C, 1e-3, 5), 4, lmax=lmax)
    off, _ = g.cut_points()
    per = np.diff(off)[np.diff(off) > 0]
    assert {0: per.max() <= 8, 1: per.min() < 32 < per.max(), 3: per.max() > 256}[lmax]
    ph = I.Physics(mu=0.01, dt=0.02, scheme=scheme, g=(0.1, 0.0, -0.2))
    u, up, v = I.state(g.n_nodes, 3)
    up2, f = up + 0.01 * v, 0.3 * v[:, [1, 2, 3, 0]]
    Ro, Jo = o.residual_jvp(ph, u, up, up2, f, v)
    a = [T(x, dev) for x in (u, up, v, up2, f)]
    for det in (True, False):
        g.deterministic(det)
        R = g.residual(ph, a[0], a[1], a[3], f=a[4]).cpu().numpy()
        J = g.jvp(ph, a[0], a[1], a[2], a[3], f=a[4]).cpu().numpy()
        assert rel(R, Ro) <= TOL64 and rel(J, Jo) <= TOL64


# ---- float64 element Jacobians (a warp per element part, lane = column) ----
@pytest.mark.parametrize("scheme", [I.SCHEME_BE, I.SCHEME_CN, I.SCHEME_BDF2])
@pytest.mark.parametrize("lmax", [0, 2])
def test_float64_element_jacobians(dev, scheme, lmax):
    g, o = pair(I.icosphere(2, 0.2, C, 1e-3, 6), 4, lmax=lmax)
    ph = I.Physics(mu=0.02, dt=0.05, scheme=scheme, g=(0.2, -0.1, 0.0), drop_visc=int(lmax == 0))
    u, up, v = I.state(g.n_nodes, 4)
    u[:, 0] -= 1.5 * (np.arange(g.n_nodes) % 2)          # inflow and outflow at the surface
    up2, f = up + 0.01 * v, 0.2 * v[:, [2, 0, 1, 3]]
    a = [T(x, dev) for x in (u, up, up2, f)]
    mk, _ = g.markers()
    pick = np.concatenate([np.flatnonzero(mk == 0)[::37], np.flatnonzero(mk == 2)[::9], np.flatnonzero(mk == 1)[:2]])
    pick = np.random.RandomState(0).permutation(pick).astype(np.int32)[: 2 * (pick.size // 2) - 1]   # any order, odd count
    K = g.element_jacobians(ph, a[0], a[1], T(pick, dev), a[2], f=a[3]).cpu().numpy()
    for i, e in enumerate(pick):
        want = o.element_matrix(ph, u, up, int(e), up2, f)[0]
        # float64 throughout; the fine scale's direction u' / |u'| loses what it cancels
        assert np.linalg.norm(K[i] - want) <= 1e-11 * max(np.linalg.norm(want), 1e-300), (int(e), mk[e])
    # the assembled matrix (same columns through M_e) is the operator of J v
    Jv = g.jvp(ph, a[0], a[1], T(v, dev), a[2], f=a[3])
    Av = g.bsr_spmv(g.bsr_assemble(ph, a[0], a[1], a[2], f=a[3]), T(v, dev))
    assert float((Av - Jv).norm() / Jv.norm()) <= TOL64


def test_float64_block_jacobi_matches_mixed(dev):
    w = I.small_sphere(3)
    g = api.Mesh.from_workload(w)
    u, up, _ = I.state(g.n_nodes, 2)
    its = []
    for prec in (api.PRECISION_FP64, api.PRECISION_MIXED):
        st = g.newton_step(w.physics, T(u, dev), T(up, dev), precision=prec, precond=1, max_newton=2, raise_on_failure=False)
        its.append(st["krylov_per_newton"])
    # the same blocks to float32 rounding: the same iterations, give or take one
    assert np.abs(np.array(its[0]) - np.array(its[1])).max() <= 1


# ---- row products: a warp per row below 32,768 rows, eight lanes from there on ----
@pytest.mark.parametrize("level", [6, 7])
def test_row_products_and_vcycle(dev, level):
    reg = [I.Region(I.REGION_SPHERE_BAND, level, (*C, 0.1, 0.05))]
    g = api.Mesh((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), 3, reg, I.icosphere(2, 0.1, C, 1e-3, 6), 1)
    assert (g.n_nodes >= 32768) == (level == 7)
    ph = I.Physics(mu=0.02, dt=0.05)
    u, up, v = (T(a, dev) for a in I.state(g.n_nodes, 5))
    Av = g.bsr_spmv(g.bsr_assemble(ph, u, up, up), v)
    Jv = g.jvp(ph, u, up, v, up)
    assert float((Av - Jv).norm() / Jv.norm()) <= TOL64
    z = {}
    for prec in (api.PRECISION_FP64, api.PRECISION_MIXED):
        for sweeps in (1, 2):
            g.multilevel_setup(ph, u, up, up, precision=prec, sweeps=sweeps)
            z[prec, sweeps] = g.multilevel_apply(v).clone()
            out = torch.empty_like(v)
            graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.graph(graph, stream=side):
                g.multilevel_apply(v, out=out)
            for _ in range(20):   # launches that overlap, and captured ones that do not: the same bits every time
                graph.replay()
                assert torch.equal(out, z[prec, sweeps])
                assert torch.equal(g.multilevel_apply(v), z[prec, sweeps])
    for sweeps in (1, 2):
        # a float32 cycle: 6e-8 per operation, some hundred of them in a row and a few levels of block inverses
        # (entries up to ~1e2 times their blocks'); a row or an aggregate gone wrong would be of order one
        d = z[api.PRECISION_MIXED, sweeps] - z[api.PRECISION_FP64, sweeps]
        assert float(d.norm() / z[api.PRECISION_FP64, sweeps].norm()) <= 1e-2


# ---- in/out: the float32 filters leave every flag to float64 where they cannot decide ----
@pytest.mark.parametrize("lo", [(0.0, 0.0, 0.0), (1000.0, -2000.0, 500.0)])
@pytest.mark.parametrize("body", ["sphere", "box", "truck"])
def test_classify_near_the_surface(dev, body, lo):
    lo = np.array(lo)
    if body == "sphere":
        tri, edge, lev = I.icosphere(3, 0.2, C, 1e-4, 2), 1.0, 5
    elif body == "box":      # faces on element planes, edge-on to the rays
        tri, edge, lev = I.grid_box((0.25, 0.25, 0.375), (0.75, 0.5, 0.625), 1 / 16), 1.0, 4
    else:
        tri, edge, lev = I.truck(0.7, 3.2, 2.7, 8, 1e-5, 3), 6.4, 5
    tri = tri + lo
    args = (tuple(lo), tuple(lo + edge), lev, [], tri, 1)
    g, o = api.Mesh(*args), OracleMesh(*args)
    rs = np.random.RandomState(1)
    t = tri[rs.randint(0, tri.shape[0], 4000)]
    bary = rs.dirichlet((1, 1, 1), 4000)
    bary[:1000, 0] = 0                      # on edges, and at vertices
    bary[:500, 1] = 0
    bary /= bary.sum(1, keepdims=True)
    n = np.cross(t[:, 1] - t[:, 0], t[:, 2] - t[:, 0])
    n /= np.linalg.norm(n, axis=1, keepdims=True)
    off = np.concatenate([[0.0], 10.0 ** np.arange(-15, -1)])
    off = np.concatenate([off, -off])[rs.randint(0, 30, 4000)] * edge
    far = lo + edge * rs.rand(4000, 3)
    pts = np.concatenate([np.einsum("ni,nij->nj", bary, t) + off[:, None] * n, far, np.vstack([lo, lo + edge, lo - 1, np.full(3, np.nan)])])
    want = o.classify(np.nan_to_num(pts, nan=-1e9))
    assert np.array_equal(g.classify(T(pts, dev)).cpu().numpy(), want)
    # every ray by itself: +x rays through edge-on faces, grazes re-cast along +y and +z
    g.classify_rays_only(True)
    rays = g.classify(T(pts[4000:8000], dev)).cpu().numpy()
    assert np.array_equal(rays, want[4000:8000])


# ---- the caller's matrix and vectors as float64 views that start at an odd element (8-byte, not 16-byte
# addresses), on both sides of the size where the row products change shape ----
@pytest.mark.parametrize("level", [5, 7])
def test_matrix_in_views_at_odd_elements(dev, level):
    reg = [I.Region(I.REGION_SPHERE_BAND, level, (*C, 0.1, 0.05))]
    g = api.Mesh((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), 3, reg, I.icosphere(2, 0.1, C, 1e-3, 6), 1)
    assert (g.n_nodes >= 32768) == (level == 7)
    ph = I.Physics(mu=0.02, dt=0.05)
    u, up, v = (T(a, dev) for a in I.state(g.n_nodes, 5))
    ptr, idx = g.bsr_pattern()

    def odd(*shape):
        t = torch.empty(1 + int(np.prod(shape)), dtype=torch.float64, device=dev)[1:].view(*shape)
        assert t.data_ptr() % 16 == 8
        return t

    A = g.bsr_assemble(ph, u, up)
    B = g.bsr_assemble(ph, u, up, out=odd(idx.size, 4, 4))
    # float64 atomics add at most a few dozen terms per entry, in any order
    assert float((A - B).abs().max() / A.abs().max()) <= 1e-13
    rows = torch.from_numpy(np.repeat(np.arange(g.n_nodes), np.diff(ptr))).to(dev)
    on = rows == torch.from_numpy(idx.astype(np.int64)).to(dev)
    eye = torch.eye(4, dtype=torch.float64, device=dev)
    s = torch.zeros(g.n_nodes, 4, dtype=torch.float64, device=dev).index_add_(0, rows, B.abs().sum(2))
    flat = s == 1.0                                       # identity rows
    assert flat[:, :3].any() and torch.equal(B[on][flat], eye.expand(g.n_nodes, 4, 4)[flat])
    B.copy_(A)
    w = odd(g.n_nodes, 4).copy_(v)
    want = g.bsr_spmv(A, v)
    for vals, x in ((B, v), (A, w), (B, w)):
        assert torch.equal(g.bsr_spmv(vals, x, out=odd(g.n_nodes, 4)), want)


# ---- the training loss is a float64 sum of float64 squares ----
@pytest.mark.parametrize("rows", [16, 1000, 5000])
def test_mlp_loss_is_a_float64_sum(dev, rows):
    net = api.Mlp(seed=1)
    net.set_params(np.zeros(net.n_params, np.float32))    # y = 0: the errors are the targets
    X = torch.zeros(rows, 1027, device=dev)
    # at most 64 additions in a thread, 5 over its warp, then one of at most rows / 2 warps after another
    tol = (64 + 5 + rows / 2) * 2.0 ** -53
    for c in (1.9767611, 1.4614793, 3e-20, 1e20):         # squares below and above the float32 range among them
        t = torch.full((rows, 1024), c, device=dev)
        want = 0.5 * 1024 * float(t[0, 0].double()) ** 2
        assert abs(net.gradient(X, t)[0] / want - 1) <= tol, c
    t = torch.randn(rows, 1024, device=dev)
    t[rows // 2, 7] = float("inf")
    assert net.gradient(X, t)[0] == float("inf")
    t[0, 0] = float("nan")
    assert np.isnan(net.gradient(X, t)[0])


# ---- results written over the inputs: one thread block's results reach the rows that another reads ----
@pytest.mark.parametrize("rows", [17, 1000, 5000])
@pytest.mark.parametrize("nin,nout,ldx", [(1027, 1024, 1040), (45, 72, 72)])
def test_mlp_forward_in_place(dev, rows, nin, nout, ldx):
    net = api.Mlp(n_in=nin, n_out=nout, seed=3)
    torch.manual_seed(rows)
    X = torch.randn(rows, ldx, device=dev)
    want = net.forward(X.clone())
    api.check(_lib.load().imga_mlp_forward(net.h, api._ptr(X), ldx, rows, api._ptr(X), api._stream(None)))
    assert torch.equal(X.view(-1)[: rows * nout].view(rows, nout), want)   # the same sums in the same order


# ---- a mixed-precision solve's float64 evaluations take the fused launch too where it is switched on ----
@pytest.mark.parametrize("graphs", [False, True])
def test_fused_launch_in_mixed_solves(dev, graphs):
    w = I.small_sphere(4)
    g = api.Mesh.from_workload(w)
    u0, up, _ = I.state(g.n_nodes, 4)
    kw = dict(precision=api.PRECISION_MIXED, precond=1, max_newton=2, raise_on_failure=False)
    u = [T(u0, dev) for _ in range(2)]
    st = [None, None]
    for fused in (False, True):
        g.fused(fused)
        g.use_graphs(graphs)
        st[fused] = g.newton_step(w.physics, u[fused], T(up, dev), **kw)
    # the same sums but for the contraction of a last bit, which a solve to 1e-3 per linear step may amplify
    assert abs(st[0]["krylov_its"] - st[1]["krylov_its"]) <= 2
    assert float((u[0] - u[1]).norm() / u[0].norm()) <= 1e-5
    g.profile(True)                                        # (profiled solves are driven from the host)
    g.newton_step(w.physics, T(u0, dev), T(up, dev), **kw)
    n = {k: c for k, (_, c) in g.profile_read().items()}
    g.profile(False)
    assert n["fused"] > 0 and n["out_elements"] == 0 and n["cut_elements"] == 0


def test_tuning_reports_the_one_shape_of_few_cut_elements(dev):
    g, _ = pair(I.icosphere(2, 0.2, C, 1e-3, 5), 4, lmax=1)
    assert g.info["n_cut"] <= 16 * torch.cuda.get_device_properties(dev).multi_processor_count
    u, up, v = (T(a, dev) for a in I.state(g.n_nodes, 3))
    ph = I.Physics(mu=0.01, dt=0.02)
    want = g.jvp(ph, u, up, v, precision=api.PRECISION_MIXED)
    g.autotune(True)
    assert torch.equal(g.jvp(ph, u, up, v, precision=api.PRECISION_MIXED), want)
    wpb, lpt, ms = g.tuning()[(api.PRECISION_MIXED, "jvp")]
    assert wpb == 4 and lpt in (0, 1) and min(ms[2:4]) > 0 and ms[:2] + ms[4:] == [0.0] * 4


# ---- the V-cycle row by row against the oracle's on the exported matrix: rows on both sides of 32,768, and aggregates
# that fit the rows a block takes at a time (8 or 32), exceed them, and do not divide the row count ----
@pytest.mark.parametrize("level,aggs", [(6, (3, 9, 20)), (7, (6, 41))])
def test_vcycle_rows_against_oracle(dev, level, aggs):
    import scipy.sparse as sp
    from oracle import sparse as S
    reg = [I.Region(I.REGION_SPHERE_BAND, level, (*C, 0.1, 0.05))]
    # (without a body: nodes that only slivers reach have nearly singular blocks, and rows of z of 1e12 hide all others)
    g = api.Mesh((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), 3, reg, None, 1)
    n = g.n_nodes
    assert (n >= 32768) == (level == 7)
    ph = I.Physics(mu=0.02, dt=0.05)
    u, up, v = (T(a, dev) for a in I.state(n, 5))
    ptr, idx = g.bsr_pattern()
    A = sp.bsr_matrix((g.bsr_assemble(ph, u, up).cpu().numpy(), idx, ptr), shape=(4 * n, 4 * n)).tocsr()
    r = v.cpu().numpy().reshape(-1)
    for agg in aggs:
        levels = S.hierarchy(A, agg_size=agg, coarse_max=16)
        assert n % agg
        for prec, tol in ((api.PRECISION_FP64, 1e-9), (api.PRECISION_MIXED, 1e-2)):
            # float64: as the V-cycle's other test; float32: 6e-8 per operation, some hundred of them in a row, block inverses
            # of entries up to ~1e2.  Row by row: a row or an aggregate gone wrong is off by about the mean row
            for sweeps in (1, 2):
                want = S.vcycle(levels, r, nu=sweeps, omega=0.5)
                g.multilevel_setup(ph, u, up, precision=prec, agg=agg, coarse_max=16, sweeps=sweeps, omega=0.5)
                assert list(g.multilevel_info()[0]) == [L["n"] for L in levels]
                z = g.multilevel_apply(v).cpu().numpy().reshape(-1)
                assert np.abs(z - want).max() <= tol * np.linalg.norm(want) / np.sqrt(want.size), (agg, prec, sweeps)


# ---- targets at a 4-byte address take the general path, whose own buffers grow when it is first taken ----
def test_mlp_general_path_after_the_fused_one(dev):
    net = api.Mlp(seed=2)
    torch.manual_seed(0)
    X, Y = torch.randn(1500, 1040, device=dev), torch.randn(1500, 1024, device=dev)
    odd = torch.empty(1500 * 1024 + 1, device=dev)[1:].view(1500, 1024).copy_(Y)
    assert odd.data_ptr() % 8 == 4
    for rows in (100, 1500, 700):
        l1, g1 = net.gradient(X[:rows], Y[:rows])
        l2, g2 = net.gradient(X[:rows], odd[:rows])
        # the same products in the same order; a bf16 mask or a float32 sum may fall otherwise at most
        assert abs(l1 - l2) <= 1e-12 * l1 and np.linalg.norm(g1 - g2) <= 1e-5 * np.linalg.norm(g1)


# ---- the float64 Out elements' Gauss abscissa is the correctly rounded one.  At u = 0 on a uniform mesh the momentum rows
# of J v are c0 rho M + mu (K + K') + rho tau_C (grad div) in closed form; the abscissa enters through the 1D mass
# matrix h/4 [[1 + g^2, 1 - g^2], [1 - g^2, 1 + g^2]].  Its relative error is what the error of J v has along dJ/dg: a fit
# over 10^4 entries, whose own roundings (1e-16 each, of either sign) move it by about 1e-18 ----
def _uniform_momentum(v, h, c0, mu, tauC, g2):
    L = np.longdouble

    def st(x, ax, lo, mid, hi):
        return lo * x.take(range(0, x.shape[ax] - 2), ax) + mid * x.take(range(1, x.shape[ax] - 1), ax) + hi * x.take(range(2, x.shape[ax]), ax)
    M = lambda x, ax: st(x, ax, h / 4 * (1 - g2), h / 2 * (1 + g2), h / 4 * (1 - g2))
    K = lambda x, ax: st(x, ax, -1 / h, 2 / h, -1 / h)
    D = lambda x, ax: st(x, ax, L(-0.5), L(0), L(0.5))        # test value, trial derivative; the transpose is -D
    mass, visc, gd = [], [], []
    for i in range(3):
        m = v[..., i]
        for ax in range(3):
            m = M(m, ax)
        mass.append(c0 * m)
        vi, gi = 0, 0
        for j in range(3):
            k = v[..., i]
            for ax in range(3):
                k = K(k, ax) if ax == j else M(k, ax)
            vi = vi + k
            x = v[..., j]
            for ax in range(3):                                  # d_i w d_j v_j and d_j w d_i v_j: the same for i != j, both -D D
                x = K(x, ax) if i == j == ax else -D(x, ax) if ax == i else D(x, ax) if ax == j else M(x, ax)
            gi = gi + x
            vi = vi + x
        visc.append(mu * vi)
        gd.append(tauC * gi)
    return [np.stack(q, -1) for q in (mass, visc, gd)]


def test_float64_gauss_abscissa(dev):
    L, lev = np.longdouble, 4
    n, h, dt, mu = 2 ** lev + 1, 2.0 ** -lev, 2.0 ** -7, 2.0 ** -6
    g = api.Mesh((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), lev, [], None, 1)
    assert g.n_nodes == n ** 3
    at = tuple((g.export()["node_ijk"].astype(np.int64) >> (20 - lev)).T)
    v = I.state(g.n_nodes, 7)[2].copy()
    v[:, 3] = 0
    z = torch.zeros(g.n_nodes, 4, dtype=torch.float64, device=dev)
    ph = I.Physics(mu=mu, dt=dt)
    Jv = g.jvp(ph, z, z, T(v, dev)).cpu().numpy()
    grid = np.zeros((n, n, n, 3), L)
    got = np.zeros((n, n, n, 3), L)
    grid[at], got[at] = v[:, :3], Jv[:, :3]
    got = got[1:-1, 1:-1, 1:-1]
    g2 = L(2) / L(h)
    g2 = g2 * g2
    tauM = 1 / np.sqrt(4 / L(dt) ** 2 + 3 * L(ph.CI) * L(mu) ** 2 * g2 * g2)
    args = (grid, L(h), 1 / L(dt), L(mu), 1 / (3 * g2 * tauM))
    third, e = 1 / L(3), L(2) ** -20
    parts = _uniform_momentum(*args, third)
    b = (sum(_uniform_momentum(*args, third * (1 + e) ** 2)) - sum(_uniform_momentum(*args, third * (1 - e) ** 2))) / (2 * e)
    err = got - sum(parts)
    assert float(np.abs(err).max() / np.abs(sum(parts)).max()) < 1e-14           # the closed form is the operator
    # (the three parts may each have a constant of their own rounding: tau_C, and the scale of the stresses)
    fit = np.linalg.lstsq(np.stack([np.asarray(x, np.float64).ravel() for x in (b, *parts)], 1), np.asarray(err, np.float64).ravel(), rcond=None)[0]
    print("relative error of the abscissa", fit[0])
    assert abs(fit[0]) <= 2.0 ** -53                                              # correctly rounded


# ---- the block-Jacobi blocks themselves: the first Krylov vector of a solve from b is D^-1 b, so one Krylov iteration of
# one Newton step moves u along it.  Without hanging nodes D is the diagonal of the assembled matrix ----
@pytest.mark.parametrize("prec,tol", [(api.PRECISION_FP64, 1e-10), (api.PRECISION_MIXED, 1e-3)])
def test_block_jacobi_blocks(dev, prec, tol):
    g = api.Mesh((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), 4, [], I.icosphere(2, 0.2, C, 1e-3, 3), 2)
    assert g.n_hang == 0 and g.info["n_cut"] > 0 and g.info["n_surface_points"] > 0
    ph = I.Physics(mu=0.02, dt=0.05)
    u0, up = (T(a, dev) for a in I.state(g.n_nodes, 5)[:2])
    b = -g.residual(ph, u0, up)
    u = u0.clone()
    g.newton_step(ph, u, up, precision=prec, precond=1, max_newton=1, max_krylov=1, line_search=0, raise_on_failure=False)
    ptr, idx = g.bsr_pattern()
    rows = np.repeat(np.arange(g.n_nodes), np.diff(ptr))
    D = g.bsr_assemble(ph, u0, up)[torch.from_numpy(np.flatnonzero(rows == idx)).to(dev)]
    # D du = s b node by node, s the step along D^-1 b; a node of slivers alone may have no usable block (then the identity)
    x = torch.einsum("nij,nj->ni", D, u - u0)
    s = float((x * b).sum() / (b * b).sum())
    usable = torch.linalg.svdvals(D)[:, -1] > 1e-8 * D.abs().amax((1, 2))
    assert float(usable.double().mean()) > 0.95 and s != 0
    scale = torch.einsum("nij,nj->ni", D.abs(), (u - u0).abs()).amax(1) + abs(s) * b.abs().amax(1) + 1e-300
    off = (x - s * b).abs().amax(1) / scale
    # float64: an inverse and a product of 4 x 4 blocks; float32 element arithmetic: 6e-8 per operation, some hundred of them
    assert float(off[usable].max()) <= tol
