"""The forward on resampled coefficients (csrc/line.cu): the shapes at which
its dispatch changes, against the FP64 oracle.

Tolerance: a ray is a Kahan sum of at most ~90 pieces here, each a chain of
about 4 + 4 + 4 + 5 roundings of 2^-24 on terms no larger than the window's
absolute sum; with random signs that is about 17 * 2^-24 = 1e-6 of a piece
and less of the sum, so the relative L2 error stays below 2e-6.
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


def check(env, orc, geo, degree, seed, dims=DIMS):
    torch, spl = env
    rng = np.random.default_rng(seed)
    origin = I.centred_origin(dims)
    c = rng.normal(size=dims[::-1]).astype(np.float32)
    g = spl.Geometry(dims, origin, geo)
    y = torch.full((g.n_rays,), float("nan"), device="cuda")
    spl.forward(g, torch.tensor(c, device="cuda"), y, spl.basis(degree))
    g.status()
    ref = orc.forward(degree, dims, origin, c.astype(np.float64), geom_of(orc, geo)).reshape(-1)
    err = np.linalg.norm(y.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err <= TOL, err


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("rays", [700, 25000, 50000, 90001])
def test_rays_per_split(env, orc, rays, degree):
    """Explicit rays from too few to fill the GPU (8 threads a ray) to one
    thread a ray, with short rays whose parts are empty."""
    rng = np.random.default_rng(rays + degree)
    w = I.random_directions(rng, rays)
    w[::7, rng.integers(3)] = 0.0
    w /= np.linalg.norm(w, axis=1, keepdims=True)
    half = 0.5 * (np.asarray(DIMS) - 1.0)
    s = rng.uniform(-1.15, 1.15, size=(rays, 3)) * half
    check(env, orc, I.RayGeometry(w, s), degree, 10 + degree)


@pytest.mark.parametrize("views", [1, 9, 21, 90])
@pytest.mark.parametrize("turned", [False, True])
@pytest.mark.parametrize("kind", ["parallel", "cone"])
def test_views_per_split_and_lane_axis(env, orc, kind, turned, views):
    """Views from 8 threads a ray to one, with detector columns along z and
    (turned) detector rows along z: both lane directions of a warp."""
    rng = np.random.default_rng(views)
    nu, nv = 37, 33
    if kind == "parallel":
        geo = I.parallel_views(I.random_directions(rng, views), nu, nv, 0.8, center=(0.3, -0.2, 0.1))
    else:
        geo = I.helical_cone(views, 50.0, 80.0, nu, nv, 0.9, turns=1.3, table_feed=6.0)
    if turned:
        geo = I.ViewGeometry(geo.kind, geo.src, geo.det_center, geo.det_v, -geo.det_u, nu, nv)
    check(env, orc, geo, 3, 20 + views)


@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 40, 3), (33, 2, 65)])
def test_thin_grids(env, orc, dims):
    """Grids thinner than a window and around the resampling's chunks."""
    rng = np.random.default_rng(5)
    w = I.random_directions(rng, 400)
    s = rng.uniform(-0.6, 0.6, size=(400, 3)) * np.asarray(dims)
    for degree in (1, 2, 3):
        check(env, orc, I.RayGeometry(w, s), degree, 30 + degree, dims)


def test_streams_take_turns(env):
    """Forwards of one geometry on two streams share the resampled arrays:
    each waits for the one before, and the results are those of calls in
    line, bit for bit (the sums have a fixed order)."""
    torch, spl = env
    rng = np.random.default_rng(6)
    g = spl.Geometry((64, 60, 56), I.centred_origin((64, 60, 56)),
                     I.circular_cone(40, 200.0, 300.0, 96, 88, 1.2))
    bas = spl.basis(3)
    cs = [torch.tensor(rng.normal(size=(56, 60, 64)).astype(np.float32), device="cuda") for _ in range(2)]
    ref = [torch.empty(g.n_rays, device="cuda") for _ in range(2)]
    for c, y in zip(cs, ref):
        spl.forward(g, c, y, bas)
    torch.cuda.synchronize()
    got = [[torch.empty(g.n_rays, device="cuda") for _ in range(4)] for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    for k in range(4):
        for i in range(2):
            spl.forward(g, cs[i], got[i][k], bas, stream=streams[i])
    torch.cuda.synchronize()
    g.status()
    for i in range(2):
        for y in got[i]:
            assert torch.equal(y, ref[i])


def test_captured_forward_matches(env):
    """A captured forward keeps the footprint form (no scratch to share);
    its replay agrees with the eager call to rounding."""
    torch, spl = env
    rng = np.random.default_rng(7)
    dims = (30, 28, 26)
    g = spl.Geometry(dims, I.centred_origin(dims), I.circular_cone(6, 100.0, 150.0, 40, 36, 1.2))
    bas = spl.basis(3)
    c = torch.tensor(rng.normal(size=dims[::-1]).astype(np.float32), device="cuda")
    eager, replayed = (torch.full((g.n_rays,), float("nan"), device="cuda") for _ in range(2))
    spl.forward(g, c, eager, bas)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        spl.forward(g, c, replayed, bas)
    graph.replay()
    torch.cuda.synchronize()
    g.status()
    assert float((eager - replayed).norm() / eager.norm()) <= TOL


@pytest.mark.parametrize("ra,rb", [(0.9, 0.04), (0.6, 0.066), (0.3, 0.11), (0.29, 0.29), (0.95, 0.2), (1.0, 1.0)])
def test_four_node_pieces_single_footprint(env, orc, ra, rb):
    """One coefficient, so a ray's value is one footprint, for ray slopes on
    both sides of the 4-node rule's bound (line_short: 5.67e-6 (ra rb + ra +
    rb) ra^2 rb^2 against 2^-28).  Allowed: at most 12 pieces of 2^-28 each
    and 20 roundings of 2^-25 at the peak (about 0.45 |w| / |w_d|)."""
    torch, spl = env
    rng = np.random.default_rng(8)
    dims = (9, 9, 9)
    w = np.tile([ra, 1.0, rb], (2000, 1))
    s = rng.uniform(-1.5, 1.5, size=w.shape)
    geo = I.RayGeometry(w / np.linalg.norm(w, axis=1, keepdims=True), s)
    c = np.zeros(dims, dtype=np.float32)
    c[4, 4, 4] = 1.0
    g = spl.Geometry(dims, I.centred_origin(dims), geo)
    y = torch.empty(g.n_rays, device="cuda")
    spl.forward(g, torch.tensor(c, device="cuda"), y, spl.basis(3))
    g.status()
    ref = orc.forward(3, dims, I.centred_origin(dims), c.astype(np.float64), geom_of(orc, geo)).reshape(-1)
    scale = np.sqrt(1.0 + ra * ra + rb * rb)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= scale * (12 * 2.0 ** -28 + 20 * 2.0 ** -25)


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("threads", [False, True])
def test_streams_take_turns_on_the_plane_path(env, mixed, threads):
    """Forwards of a tilt series (and of one with other views, whose plane
    path runs on the geometry's own stream) on two streams, from one thread
    and from two: the results are those of calls in line, bit for bit."""
    import threading

    torch, spl = env
    rng = np.random.default_rng(12)
    dims = (70, 66, 60)
    geo = I.tilt_series(60, 96, 88, 1.0)
    if mixed:
        other = I.parallel_views(I.random_directions(rng, 30), 96, 88, 1.0)
        geo = I.ViewGeometry("parallel", *[np.concatenate([getattr(geo, f), getattr(other, f)])
                                           for f in ("src", "det_center", "det_u", "det_v")], 96, 88)
    g = spl.Geometry(dims, I.centred_origin(dims), geo)
    bas = spl.basis(3)
    spl.prepare(g, bas)
    cs = [torch.tensor(rng.normal(size=dims[::-1]).astype(np.float32), device="cuda") for _ in range(2)]
    ref = [torch.empty(g.n_rays, device="cuda") for _ in range(2)]
    for c, y in zip(cs, ref):
        spl.forward(g, c, y, bas)
    torch.cuda.synchronize()
    got = [[torch.empty(g.n_rays, device="cuda") for _ in range(6)] for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]

    def calls(i, ks):
        for k in ks:
            spl.forward(g, cs[i], got[i][k], bas, stream=streams[i])

    if threads:
        both = [threading.Thread(target=calls, args=(i, range(6))) for i in range(2)]
        for t in both:
            t.start()
        for t in both:
            t.join()
    else:
        for k in range(6):
            calls(0, [k])
            calls(1, [k])
    torch.cuda.synchronize()
    g.status()
    for i in range(2):
        for y in got[i]:
            assert torch.equal(y, ref[i])


def project(env, dims, geo, c, degree, kahan=True):
    torch, spl = env
    g = spl.Geometry(dims, I.centred_origin(dims), geo)
    y = torch.empty(g.n_rays, device="cuda")
    spl.forward(g, torch.tensor(c, device="cuda"), y, spl.basis(degree, kahan=kahan))
    g.status()
    return y.cpu().numpy()


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("d,a", [(0, 1), (1, 2), (2, 0), (2, 1)])
def test_support_corner_is_accurate_by_itself(env, orc, degree, d, a):
    """One coefficient and rays that clip the corner of its support within
    t = 1e-3 .. 0.3 cells, where two weights are t^n and (ra (tau - t))^n: the
    projection is positive, and accurate relative to itself.  Allowed: the
    clipped argument's rounding at the outermost node (0.047 of the piece),
    n 2^-25 / 0.047, the 2^-32 of the position, n 2^-32 / (ra t) = 5e-7, and 20
    roundings of 2^-24: below 6e-6."""
    rng = np.random.default_rng(20)
    dims, W = (9, 9, 9), 0.5 * (degree + 1)
    b = 3 - d - a
    ra, tau = 0.7, 10.0 ** rng.uniform(-3.0, -0.5, 2000)
    w, s = np.zeros((2000, 3)), np.zeros((2000, 3))
    w[:, d], w[:, a], w[:, b] = 1.0, -ra, 0.02
    # at the low d face of the support, ra tau inside its low a face
    s[:, d], s[:, a], s[:, b] = -W, -W + ra * tau, rng.uniform(-0.4, 0.4, 2000)
    s += 3.0 * w  # elsewhere on the line
    geo = I.RayGeometry(w / np.linalg.norm(w, axis=1, keepdims=True), s)
    c = np.zeros(dims, dtype=np.float32)
    c[4, 4, 4] = 1.0
    y = project(env, dims, geo, c, degree)
    ref = orc.forward(degree, dims, I.centred_origin(dims), c.astype(np.float64), geom_of(orc, geo)).reshape(-1)
    assert np.all(ref > 0.0)
    assert np.all(y > 0.0)
    assert np.max(np.abs(y - ref) / ref) <= 6e-6


@pytest.mark.parametrize("degree", [1, 2, 3])
def test_nonnegative_coefficients_project_nonnegative(env, degree):
    """c >= 0 with many zeros: no ray comes out below zero."""
    rng = np.random.default_rng(21)
    dims = (13, 12, 11)
    c = rng.uniform(0.0, 1.0, dims[::-1]) * (rng.uniform(size=dims[::-1]) < 0.02)
    w = I.random_directions(rng, 200000)
    s = rng.uniform(-0.75, 0.75, size=w.shape) * np.asarray(dims)
    y = project(env, dims, I.RayGeometry(w, s), c.astype(np.float32), degree)
    assert np.all(y >= 0.0) and np.any(y > 0.0)


@pytest.mark.parametrize("degree", [1, 2, 3])
def test_large_and_infinite_coefficients(env, orc, degree):
    """Neighbours of 2e37 (a ray's integral stays below the largest float) and
    one infinite coefficient (in plain sums: a compensation of an infinite sum is
    NaN by itself)."""
    rng = np.random.default_rng(22)
    dims = (9, 9, 9)
    w = I.random_directions(rng, 2000)
    s = rng.uniform(-0.5, 0.5, size=w.shape) * 9.0
    geo = I.RayGeometry(w, s)
    c = rng.uniform(0.9, 1.0, dims).astype(np.float32)
    one, big = project(env, dims, geo, c, degree), project(env, dims, geo, c * np.float32(2.0 ** 124), degree)
    assert np.array_equal(big, one * np.float32(2.0 ** 124))
    hot = np.zeros(dims, dtype=np.float32)
    hot[4, 4, 4] = 1.0
    ref = orc.forward(degree, dims, I.centred_origin(dims), hot.astype(np.float64), geom_of(orc, geo)).reshape(-1)
    c[4, 4, 4] = np.inf
    y = project(env, dims, geo, c, degree, kahan=False)
    assert np.all(np.isposinf(y[ref > 1e-3])) and np.all(np.isfinite(y[ref == 0.0]))


def test_scratch_comes_with_prepare(env):
    """The resampled arrays are allocated by spl_prepare for the degree asked
    for: a geometry that is only made, or used for A^T, holds none, degree 1 takes
    half of a cubic array's bytes, and a first call that is captured takes none
    and leaves them to the next eager one.  Degrees in turn on one geometry share
    the block: the values are those of a fresh geometry, bit for bit."""
    torch, spl = env
    rng = np.random.default_rng(25)
    dims = (256, 250, 240)
    geo = I.circular_cone(12, 700.0, 1000.0, 260, 250, 1.4)
    cubic = sum((dims[d] + 3) * (dims[p] + 6) * ((dims[q] + 6 + 7) // 8 * 8 + 3) * 16 for d, p, q in
                ((0, 1, 2), (1, 0, 2)))  # no ray has z as its dominant axis

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    c = torch.tensor(rng.normal(size=dims[::-1]).astype(np.float32), device="cuda")
    y, b = torch.zeros(geo.n_rays, device="cuda"), torch.empty(dims[::-1], device="cuda")

    def captured(g):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            spl.forward(g, c, y, spl.basis(1))
        graph.replay()
        torch.cuda.synchronize()

    fresh = {}
    for degree in (1, 2, 3):
        g = spl.Geometry(dims, I.centred_origin(dims), geo)
        spl.forward(g, c, y, spl.basis(degree))
        fresh[degree] = y.clone()
        spl.adjoint(g, y, b, spl.basis(3))
        captured(g)  # (loads its kernels, which takes memory too)
        g.close()
    g = spl.Geometry(dims, I.centred_origin(dims), geo)
    made = free()
    spl.adjoint(g, y, b, spl.basis(3))
    assert made - free() < 16 << 20
    captured(g)
    assert made - free() < 32 << 20
    assert float((y - fresh[1]).norm() / y.norm()) <= TOL
    used = {}
    for degree in (1, 3, 2, 1, 3):
        spl.forward(g, c, y, spl.basis(degree))
        g.status()
        assert torch.equal(y, fresh[degree]), degree
        used.setdefault(degree, made - free())
    assert 0.4 * cubic < used[1] < 0.6 * cubic + (32 << 20)
    assert 0.95 * cubic < used[3] < 1.05 * cubic + (32 << 20) and abs(used[2] - used[3]) < 16 << 20


def test_warp_mates_in_any_order(env):
    """The Gauss rule of a cubic ray depends on which rays share its warp and on
    nothing else: rays put in another order within each group of 32 keep their
    values bit for bit."""
    torch, spl = env
    rng = np.random.default_rng(23)
    rays = 90016  # one thread a ray
    w = I.random_directions(rng, rays)
    w[::3] = np.array([1.0, 0.3, 0.01]) * rng.uniform(0.5, 1.0, size=(len(w[::3]), 1)) + 0.02 * w[::3]
    w[rays // 2:] = w[0] + 0.01 * w[rays // 2:]  # whole groups that take four nodes
    w /= np.linalg.norm(w, axis=1, keepdims=True)
    s = rng.uniform(-1.15, 1.15, size=(rays, 3)) * 0.5 * (np.asarray(DIMS) - 1.0)
    perm = np.concatenate([32 * k + rng.permutation(32) for k in range(rays // 32)])
    c = rng.normal(size=DIMS[::-1]).astype(np.float32)
    y = project(env, DIMS, I.RayGeometry(w, s), c, 3)
    assert np.array_equal(y[perm], project(env, DIMS, I.RayGeometry(w[perm], s[perm]), c, 3))


def test_position_at_the_end_of_a_long_ray(env, orc):
    """Rays along 2040 cells whose step is no multiple of 2^-40 (2^-48 exactly),
    to a coefficient whose support they enter g = 1e-4 .. 2e-4 inside one face and
    leave through it: the projection goes with g^7, so a drift of half a
    2^-40 per cell, 9e-10, would show as 3e-5 to 6e-5.  Allowed: the 2^-32 to
    which a cell takes its fraction, 7 * 2^-32 / g = 1.6e-5, and 6e-6 as for the
    other clipped corners."""
    rng = np.random.default_rng(24)
    dims, k = (2048, 9, 9), 2040
    ra = (np.floor(0.003 * 2.0 ** 40) + 126.0 / 256.0) / 2.0 ** 40
    g = rng.uniform(1e-4, 2e-4, 500)
    x0 = -0.5 * (dims[0] - 1)  # the grid's first coefficient
    w = np.tile([1.0, -ra, 0.0003], (500, 1))
    s = np.zeros((500, 3))
    # the low face of the support along x is at k - 2; there y is g above the low face
    s[:, 0], s[:, 1], s[:, 2] = x0, -2.0 + g + ra * (k - 2), rng.uniform(-0.9, -0.7, 500)
    geo = I.RayGeometry(w / np.linalg.norm(w, axis=1, keepdims=True), s)
    c = np.zeros(dims[::-1], dtype=np.float32)
    c[4, 4, k] = 1.0
    ref = orc.forward(3, dims, I.centred_origin(dims), c.astype(np.float64), geom_of(orc, geo)).reshape(-1)
    assert np.all(ref > 0.0)
    y = project(env, dims, geo, c, 3)
    assert np.max(np.abs(y - ref) / ref) <= 2.2e-5


def check_forms(env, orc, geo, degree, dims, modes, line):
    """A geometry that spl_prepare has not seen takes the forms without
    scratch (SPL_FP_QUAD: footprints, SPL_FP_DIRECT: the direct march), also in a
    captured call; a prepared one the resampled arrays, whose sums round
    otherwise (`line`: some bit differs).  All against the oracle."""
    import ctypes as C

    torch, spl = env
    rng = np.random.default_rng(31)
    origin = I.centred_origin(dims)
    c = rng.normal(size=dims[::-1]).astype(np.float32)
    ct = torch.tensor(c, device="cuda")
    ref = orc.forward(degree, dims, origin, c.astype(np.float64), geom_of(orc, geo)).reshape(-1)
    out = {}
    for mode in modes:
        g, b = spl.Geometry(dims, origin, geo), spl.basis(degree, mode)
        out[mode], captured, prepared = (torch.full((g.n_rays,), float("nan"), device="cuda") for _ in range(3))
        st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        spl.check(spl.lib().spl_forward(g.handle, C.byref(b), spl._ptr(ct), spl._ptr(out[mode]), st))
        spl.forward(g, ct, prepared, b)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            spl.forward(g, ct, captured, b)
        graph.replay()
        torch.cuda.synchronize()
        g.status()
        for y in (out[mode], prepared):
            err = np.linalg.norm(y.cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err <= TOL, (mode, err)
        assert torch.equal(captured, out[mode])
        assert torch.equal(prepared, out[mode]) != line
    if len(modes) == 2 and degree > 0:
        assert not torch.equal(*out.values())  # two forms


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("kind", ["parallel", "cone", "rays"])
def test_forms_with_and_without_scratch(env, orc, kind, degree):
    torch, spl = env
    rng = np.random.default_rng(32)
    if kind == "parallel":
        geo = I.parallel_views(I.random_directions(rng, 9), 23, 21, 1.1, center=(0.3, -0.2, 0.1))
    elif kind == "cone":
        geo = I.helical_cone(9, 50.0, 80.0, 23, 21, 1.4, turns=1.3, table_feed=6.0)
    else:
        w = I.random_directions(rng, 3000)
        geo = I.RayGeometry(w, rng.uniform(-0.6, 0.6, size=w.shape) * np.asarray(DIMS))
    check_forms(env, orc, geo, degree, DIMS, (spl.SPL_FP_QUAD, spl.SPL_FP_DIRECT), True)


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("rays", [2000, 9000])
def test_eight_threads_a_ray_on_resampled_arrays(env, orc, rays, degree):
    """Few rays, yet enough for the resampled form: 8 threads a ray at every
    degree, with flat rays and short ones whose parts are empty."""
    torch, spl = env
    rng = np.random.default_rng(rays + degree)
    w = I.random_directions(rng, rays)
    w[::7, rng.integers(3)] = 0.0
    w /= np.linalg.norm(w, axis=1, keepdims=True)
    s = rng.uniform(-1.15, 1.15, size=(rays, 3)) * 0.5 * (np.asarray(DIMS) - 1.0)
    check_forms(env, orc, I.RayGeometry(w, s), degree, DIMS, (spl.SPL_FP_QUAD,), True)


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("dims", [(33, 2, 65), (2, 64, 33), (70, 31, 3)])
def test_chunks_of_the_resampling(env, orc, dims, degree):
    """Axes just beyond one and two chunks of 32 cells, with enough rays for the
    resampled form; and too few, which keep the other."""
    torch, spl = env
    rng = np.random.default_rng(33)
    w = I.random_directions(rng, 1500)
    s = rng.uniform(-0.6, 0.6, size=w.shape) * np.asarray(dims)
    check_forms(env, orc, I.RayGeometry(w, s), degree, dims, (spl.SPL_FP_QUAD,), True)
    check_forms(env, orc, I.RayGeometry(w[:60], s[:60]), degree, dims, (spl.SPL_FP_QUAD,), False)
