"""The scatter adjoint (csrc/scatter.cu): the shapes at which its dispatch
changes, against the FP64 oracle.

Tolerance: a coefficient is an FP32 sum of up to a few thousand terms in
arbitrary order; with random signs the running sum's rounding is about
sqrt(terms) * 2^-24 of a term's size against sqrt(terms) of the sum's, plus
about 20 roundings of a footprint: below 2e-6 in relative L2.
"""
import numpy as np
import pytest

from paper_2511_11078_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = 2e-6
DIMS = (13, 21, 18)


@pytest.fixture(scope="module")
def env():
    import torch

    from paper_2511_11078_gb300 import build as B
    from paper_2511_11078_gb300 import spl

    B.build()
    spl.lib()
    return torch, spl


def geom_of(orc, geo):
    if geo.kind == "rays":
        return orc.Geometry("rays", omega=geo.omega, s=geo.s)
    key = "direction" if geo.kind == "parallel" else "source"
    return orc.Geometry(geo.kind, det_center=geo.det_center, det_u=geo.det_u, det_v=geo.det_v, nu=geo.nu, nv=geo.nv,
                        **{key: geo.src})


def check(env, orc, geo, degrees, seed, dims=DIMS):
    """The degrees in turn on one geometry (they share the layouts), each
    twice: the layouts must be clear again after a call."""
    torch, spl = env
    rng = np.random.default_rng(seed)
    origin = I.centred_origin(dims)
    g = spl.Geometry(dims, origin, geo)
    y = rng.normal(size=geo.n_rays).astype(np.float32)
    yt = torch.tensor(y, device="cuda")
    for degree in degrees:
        ref = orc.adjoint(degree, dims, origin, y.astype(np.float64), geom_of(orc, geo))
        for _ in range(2):
            c = torch.full(g.coeff_shape, float("nan"), device="cuda")
            spl.adjoint(g, yt, c, spl.basis(degree))
            g.status()
            err = np.linalg.norm(c.cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err <= TOL, (degree, err)


@pytest.mark.parametrize("rays", [700, 25000, 90001])
def test_rays_per_split(env, orc, rays):
    """From too few rays to fill the GPU (8 threads a ray) to one thread a
    ray, with flat rays and short rays whose parts are empty.  The most rays
    at degree 3 (slow in the oracle) against the sum over two geometries with
    half of them each, which take two threads a ray."""
    rng = np.random.default_rng(rays)
    w = I.random_directions(rng, rays)
    w[::7, rng.integers(3)] = 0.0
    w /= np.linalg.norm(w, axis=1, keepdims=True)
    s = rng.uniform(-1.15, 1.15, size=(rays, 3)) * 0.5 * (np.asarray(DIMS) - 1.0)
    if rays < 10000:
        check(env, orc, I.RayGeometry(w, s), (3, 0, 2, 1, 3), 10)
        return
    check(env, orc, I.RayGeometry(w, s), (1,), 10)
    torch, spl = env
    y = torch.randn(rays, device="cuda")
    parts = []
    for sl in (slice(None), slice(0, rays // 2), slice(rays // 2, None)):
        g = spl.Geometry(DIMS, I.centred_origin(DIMS), I.RayGeometry(w[sl], s[sl]))
        c = torch.empty(g.coeff_shape, device="cuda")
        spl.adjoint(g, y[sl].contiguous(), c, spl.basis(3))
        g.status()
        parts.append(c.double())
    assert float((parts[0] - parts[1] - parts[2]).norm() / parts[0].norm()) <= 2 * TOL


@pytest.mark.parametrize("views", [1, 21, 60])
@pytest.mark.parametrize("turned", [False, True])
@pytest.mark.parametrize("kind", ["parallel", "cone"])
def test_views_per_split_lane_axis_and_batches(env, orc, kind, turned, views):
    """8 threads a ray to one, both lane directions of a warp, and (60 views)
    two batches through the FP64 total."""
    rng = np.random.default_rng(views)
    nu, nv = 37, 33
    if kind == "parallel":
        geo = I.parallel_views(I.random_directions(rng, views), nu, nv, 0.8, center=(0.3, -0.2, 0.1))
    else:
        geo = I.helical_cone(views, 50.0, 80.0, nu, nv, 0.9, turns=1.3, table_feed=6.0)
    if turned:
        geo = I.ViewGeometry(geo.kind, geo.src, geo.det_center, geo.det_v, -geo.det_u, nu, nv)
    check(env, orc, geo, (3, 1) if views < 60 else (1,), 20 + views)


@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 40, 3), (70, 61, 65)])
def test_thin_and_tiled_folds(env, orc, dims):
    """Grids thinner than a window, and one above the single-launch fold's
    size with partial tiles.  The sum of one coefficient's 3000 terms can
    come out near zero, so the error is taken against the sum of their
    magnitudes, A^T |y|: a running FP32 sum in any order is within a few
    roundings of 2^-24 of that."""
    rng = np.random.default_rng(5)
    w = I.random_directions(rng, 3000)
    s = rng.uniform(-0.6, 0.6, size=w.shape) * np.asarray(dims)
    torch, spl = env
    geo, origin = I.RayGeometry(w, s), I.centred_origin(dims)
    g = spl.Geometry(dims, origin, geo)
    y = rng.normal(size=geo.n_rays).astype(np.float32)
    for degree in (3, 2, 1, 0):
        ref = orc.adjoint(degree, dims, origin, y.astype(np.float64), geom_of(orc, geo))
        mag = orc.adjoint(degree, dims, origin, np.abs(y).astype(np.float64), geom_of(orc, geo))
        for _ in range(2):
            c = torch.full(g.coeff_shape, float("nan"), device="cuda")
            spl.adjoint(g, torch.tensor(y, device="cuda"), c, spl.basis(degree))
            g.status()
            assert np.linalg.norm(c.cpu().numpy() - ref) <= 8 * 2.0 ** -24 * np.linalg.norm(mag), degree


def test_flat_and_general_views_in_batches(env, orc):
    """Parallel views of all three classes (plane group, other flat views,
    general views), in and out of the plane path, with more than one batch."""
    torch, spl = env
    rng = np.random.default_rng(9)
    a = I.tilt_series(20, 25, 23, 0.9)
    b = I.parallel_views(np.array([[0.0, np.cos(t), np.sin(t)] for t in 0.2 + 0.1 * np.arange(15)]), 25, 23, 0.9)
    c = I.parallel_views(I.random_directions(rng, 70), 25, 23, 0.9)
    geo = I.ViewGeometry("parallel", *[np.concatenate([getattr(p, f) for p in (a, b, c)])
                                       for f in ("src", "det_center", "det_u", "det_v")], 25, 23)
    origin = I.centred_origin(DIMS)
    g = spl.Geometry(DIMS, origin, geo)
    y = rng.normal(size=geo.n_rays).astype(np.float32)
    ref = orc.adjoint(3, DIMS, origin, y.astype(np.float64), geom_of(orc, geo))
    for separable in (spl.SPL_SEP_AUTO, spl.SPL_SEP_OFF):
        out = torch.full(g.coeff_shape, float("nan"), device="cuda")
        spl.adjoint(g, torch.tensor(y, device="cuda"), out, spl.basis(3, separable=separable))
        g.status()
        err = np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= TOL, err


def test_first_adjoint_on_a_side_stream(env):
    """The first call of a fresh geometry on a stream that does not wait for
    the default one: the layouts (1.7 GB, in memory that held NaN) must be
    clear by then.  Against the same call later on the default stream; two
    runs differ by the order of the atomics only."""
    torch, spl = env
    rng = np.random.default_rng(11)
    dims = (320, 310, 300)
    w = I.random_directions(rng, 3000)
    s = rng.uniform(-0.4, 0.4, size=w.shape) * np.asarray(dims)
    poison = torch.full((3, 1 << 27), float("nan"), device="cuda")
    y = torch.randn(len(w), device="cuda")
    first, later = (torch.empty(dims[::-1], device="cuda") for _ in range(2))
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    del poison
    torch.cuda.empty_cache()
    g = spl.Geometry(dims, I.centred_origin(dims), I.RayGeometry(w, s))
    spl.adjoint(g, y, first, spl.basis(3), stream=side)
    torch.cuda.synchronize()
    spl.adjoint(g, y, later, spl.basis(3))
    g.status()
    assert float((first - later).norm() / later.norm()) <= TOL


def test_captured_call_after_a_failed_one(env):
    """A launch that fails (into a capture that a synchronisation made
    invalid) leaves the layouts to be cleared before the next use.  A captured
    call records that clear, which then runs with its graph only: the next
    capture, and the next eager call, must clear as well."""
    import ctypes as C

    torch, spl = env
    cu = C.CDLL("libcuda.so.1")
    rng = np.random.default_rng(13)
    w = I.random_directions(rng, 500)
    s = rng.uniform(-0.6, 0.6, size=w.shape) * np.asarray(DIMS)
    g = spl.Geometry(DIMS, I.centred_origin(DIMS), I.RayGeometry(w, s))
    y = torch.randn(500, device="cuda")
    ref, out = (torch.empty(g.coeff_shape, device="cuda") for _ in range(2))
    spl.adjoint(g, y, ref, spl.basis(3))
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    raw = C.c_void_p(st.cuda_stream)

    def capture(break_it=False):
        graph, n = C.c_void_p(), C.c_size_t(0)
        assert cu.cuStreamBeginCapture_v2(raw, 2) == 0  # relaxed
        if break_it:
            assert cu.cuStreamSynchronize(raw) != 0
            with pytest.raises(spl.SplError):
                spl.adjoint(g, y, out, spl.basis(3), stream=st)
            assert cu.cuStreamEndCapture(raw, C.byref(graph)) != 0
            return None
        spl.adjoint(g, y, out, spl.basis(3), stream=st)
        assert cu.cuStreamEndCapture(raw, C.byref(graph)) == 0
        assert cu.cuGraphGetNodes(graph, None, C.byref(n)) == 0
        assert cu.cuGraphDestroy(graph) == 0
        return n.value

    plain = capture()
    capture(break_it=True)
    assert [capture(), capture()] == [plain + 1, plain + 1]
    spl.adjoint(g, y, out, spl.basis(3), stream=st)
    torch.cuda.synchronize()
    g.status()
    assert float((out - ref).norm() / ref.norm()) <= TOL
    assert capture() == plain


@pytest.mark.parametrize("x_rays", [False, True])
@pytest.mark.parametrize("dims", [(150, 148, 146), (200, 190, 181), (262, 250, 241)])
def test_scattered_rays_form_per_target_size(env, orc, dims, x_rays):
    """Random rays whose target outgrows the L2: fewer shifted copies, then
    single values into one layout, per degree; and rays near the x direction,
    for which there is no x-fast layout.  400 rays meet a coefficient once or
    twice, so the error is the footprints' (about 20 roundings)."""
    rng = np.random.default_rng(14)
    w = I.random_directions(rng, 400)
    if x_rays:
        w *= (1.0, 0.3, 0.3)
        w[:, 0] = np.sign(w[:, 0]) * (np.abs(w[:, 0]) + 0.5)
        w /= np.linalg.norm(w, axis=1, keepdims=True)
    s = rng.uniform(-0.5, 0.5, size=w.shape) * np.asarray(dims)
    check(env, orc, I.RayGeometry(w, s), (3, 2, 1, 0), 15, dims)


@pytest.mark.parametrize("dims", [(150, 148, 146), (200, 190, 181)])
def test_scattered_rays_in_batches(env, dims):
    """More rays, which go in batches through the FP64 total: against the sum
    over geometries with a part of them each (fewer batches)."""
    torch, spl = env
    rng = np.random.default_rng(16)
    rays = 60001
    w = I.random_directions(rng, rays)
    s = rng.uniform(-0.5, 0.5, size=w.shape) * np.asarray(dims)
    y = torch.randn(rays, device="cuda")
    for degree in (3, 2, 1):
        parts = []
        for sl in (slice(None), slice(0, 20000), slice(20000, 30001), slice(30001, None)):
            g = spl.Geometry(dims, I.centred_origin(dims), I.RayGeometry(w[sl], s[sl]))
            c = torch.full(g.coeff_shape, float("nan"), device="cuda")
            for _ in range(2):
                spl.adjoint(g, y[sl].contiguous(), c, spl.basis(degree))
            g.status()
            parts.append(c.double())
            g.close()
        assert float((parts[0] - sum(parts[1:])).norm() / parts[0].norm()) <= TOL


def test_first_adjoint_captured(env):
    """A geometry's layouts are cleared by its first eager adjoint; a captured
    call before it records its own clear.  Layouts in memory that held NaN."""
    torch, spl = env
    rng = np.random.default_rng(17)
    dims = (120, 110, 100)
    w = I.random_directions(rng, 3000)
    s = rng.uniform(-0.4, 0.4, size=w.shape) * np.asarray(dims)
    y = torch.randn(len(w), device="cuda")
    poison = torch.full((1 << 27,), float("nan"), device="cuda")
    torch.cuda.synchronize()
    del poison
    torch.cuda.empty_cache()
    g = spl.Geometry(dims, I.centred_origin(dims), I.RayGeometry(w, s))
    replayed, eager = (torch.full(dims[::-1], float("nan"), device="cuda") for _ in range(2))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        spl.adjoint(g, y, replayed, spl.basis(3))
    spl.adjoint(g, y, eager, spl.basis(3))
    graph.replay()
    torch.cuda.synchronize()
    g.status()
    assert bool(torch.isfinite(eager).all())
    assert float((replayed - eager).norm() / eager.norm()) <= TOL
