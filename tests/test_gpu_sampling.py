"""CUDA sampling through the C ABI against the FP64 oracle (Definitions 1-4,
Remark 1, Section 3).  Counts and triangle ids bit-exact, depths within
1e-5 of the cube diagonal, normals within 1e-5."""
import ctypes

import numpy as np
import pytest

import meshgen as M
import oracle
from ldni_compare import compare_ldni

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

O3 = (-0.5, -0.5, -0.5)
DIAG = 3 ** 0.5


@pytest.fixture(scope="module")
def ldni():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1009_0794_gb300 as pkg
    pkg._lib.load()
    return pkg


def _check_all_axes(ldni, mesh, res, origin=O3, width=1.0):
    v, t = mesh
    grid = ldni.Grid.cube(origin, width, res)
    got = ldni.sample(v, t, grid, "all", check_odd=True)
    stats = []
    for a in range(3):
        ref = oracle.sample(v, t, grid.origin, grid.width, res, a, "scan")
        stats.append(compare_ldni(got[a].numpy(), ref, DIAG * grid.width))
    return got, stats


@pytest.mark.parametrize("res", [128, 100, 37])
def test_pr1_parity(ldni, res):
    A, B = M.pr1_pair()
    for mesh in (A, B):
        _check_all_axes(ldni, mesh, res)


def test_single_axis_calls_match_fused(ldni):
    A, _ = M.pr1_pair()
    grid = ldni.Grid.cube(O3, 1.0, 96)
    fused = ldni.sample(*A, grid, "all")
    for a in range(3):
        one = ldni.sample(*A, grid, a).numpy()
        ref = oracle.sample(*A, grid.origin, 1.0, 96, a, "scan")
        compare_ldni(one, ref, DIAG)
        assert np.array_equal(one["offsets"], fused[a].numpy()["offsets"])


def test_octahedron_on_pixel_centres(ldni):
    """Edges and vertices exactly on ray lattice points (Remark 1)."""
    res = 64
    h = 1.0 / res
    cc = -0.5 + 32.5 * h
    mesh = M.octahedron([cc, cc, cc], 11 * h)
    got, _ = _check_all_axes(ldni, mesh, res)
    for a in range(3):
        assert set(np.unique(got[a].counts().cpu().numpy())) <= {0, 2}


def test_big_triangles_and_partial_cover(ldni):
    """Faces spanning thousands of pixels (CTA-per-triangle path), a mesh
    sticking out of the cube (clamped boxes), a ragged resolution."""
    _check_all_axes(ldni, M.box([-0.45, -0.3, -0.41], [0.37, 0.44, 0.33]), 201)
    _check_all_axes(ldni, M.box([-0.7, -0.2, -0.1], [0.3, 0.9, 0.2]), 130)
    _check_all_axes(ldni, M.icosphere(3, r=0.6, noise=0.05, seed=3), 150)


def test_flower_and_knot_multilayer(ldni):
    """Multi-layer rays (petals, knot strands) at a moderate resolution."""
    _check_all_axes(ldni, M.flower(96, 96), 160)
    _check_all_axes(ldni, M.torus_knot(n_ring=128, n_side=16), 160)


@pytest.mark.parametrize("k", [3, 40, 100, 450])
def test_deep_rays_ordered(ldni, k):
    """Stacked boxes give rays of up to 2k samples, so every way of ordering
    a ray is taken: by its lane (up to 4), by a warp from shared memory (up to
    128), by ranks in place (up to 768) and by insertion beyond."""
    mesh = M.slab_stack(k, axis=k % 3, seed=k)
    got, _ = _check_all_axes(ldni, mesh, 48)
    assert int(got[k % 3].counts().max()) > {3: 4, 40: 64, 100: 128, 450: 768}[k]


def test_grid_offset_and_scale(ldni):
    """A non-unit cube with a non-trivial origin."""
    v, t = M.icosphere(6, r=0.3, noise=0.02, seed=8)
    v2 = (v.astype(np.float64) * 3.0 + np.array([10.0, -4.0, 2.5])).astype(np.float32)
    _check_all_axes(ldni, (v2, t), 90, origin=(8.7, -5.3, 1.2), width=2.6)


def test_empty_mesh_and_outside_mesh(ldni):
    grid = ldni.Grid.cube(O3, 1.0, 32)
    v = np.zeros((3, 3), np.float32)
    t = np.zeros((0, 3), np.int32)
    out = ldni.sample(v, t, grid, "all")
    for L in out:
        assert L.n == 0 and int(L.offsets[-1]) == 0 and int(L.counts().abs().sum()) == 0
    far = M.translate(M.icosphere(2, r=0.2), (3.0, 0.0, 0.0))
    out = ldni.sample(*far, grid, "all")
    assert out[0].n > 0 and out[1].n == 0 and out[2].n == 0


def test_open_mesh_reports_odd_rays(ldni):
    """Definition 4 violated on purpose (a face removed): the odd rays are
    reported, and the count map still equals the oracle's."""
    v, t = M.icosphere(4, r=0.35)
    t_open = t[1:]
    grid = ldni.Grid.cube(O3, 1.0, 64)
    got = ldni.sample(v, t_open, grid, 2)
    ref = oracle.sample(v, t_open, grid.origin, 1.0, 64, 2, "scan")
    assert np.array_equal(got.numpy()["offsets"], ref["offsets"])
    assert np.any(np.diff(ref["offsets"]) % 2 == 1)
    with pytest.raises(ldni.LDNIError):
        ldni.sample(v, t_open, grid, 2, check_odd=True)


def _guarded_layers(ldni, grid, axis, cap, guard, fill):
    """Output arrays of one image carved from a single allocation, with
    `guard` words of `fill` before, between and after them."""
    N = grid.res * grid.res
    sizes = [N + 1, cap, cap, cap, cap, cap]  # offsets, depth, nx, ny, nz, tri
    backing = torch.full((sum(sizes) + guard * (len(sizes) + 1),), fill, dtype=torch.int32, device="cuda")
    views, guards, at = [], [backing[:guard]], guard
    for k in sizes:
        views.append(backing[at:at + k])
        guards.append(backing[at + k:at + k + guard])
        at += k + guard
    f = lambda t: t.view(torch.float32)
    L = ldni.LDNI(grid, axis, views[0], f(views[1]), f(views[2]), f(views[3]), f(views[4]), views[5], 0)
    return L, guards


def test_capacity_overflow_flagged_not_written(ldni):
    """Outputs of half the needed size, each array fenced by guard words in
    the same allocation: the overflow is reported and no write lands outside
    the arrays."""
    A, _ = M.pr1_pair()
    grid = ldni.Grid.cube(O3, 1.0, 64)
    exact = ldni.sample(*A, grid, "all")
    caps = [L.n for L in exact]
    lib = ldni._lib.load()
    vt = torch.from_numpy(A[0]).cuda()
    tt = torch.from_numpy(A[1]).cuda()
    fill = 0x7F5A5A5A
    outs, guards = zip(*[_guarded_layers(ldni, grid, a, caps[a] // 2, 1024, fill) for a in range(3)])
    arr = (ldni._CLayers * 3)(*[o.c() for o in outs])
    ws = torch.empty(ldni.sample_workspace_size(len(A[0]), len(A[1]), 64), dtype=torch.uint8, device="cuda")
    info = ldni.new_info()
    g = grid.c()
    rc = lib.ldni_sample(vt.data_ptr(), vt.shape[0], tt.data_ptr(), tt.shape[0], ctypes.byref(g), 3, 0, arr,
                         info.data_ptr(), ws.data_ptr(), ws.numel(), None)
    assert rc == 0
    meta = ldni.info_decode(info)
    assert meta["status"] & ldni._lib.ST_CAPACITY
    assert [meta["n"][a] for a in range(3)] == caps  # the sizes needed
    for gs in guards:
        for gd in gs:
            assert bool((gd == fill).all())
    plan2 = ldni.SamplePlan(len(A[0]), len(A[1]), grid, caps)
    plan2.run(vt, tt)
    outs = plan2.finish()
    for a in range(3):
        ref = oracle.sample(*A, grid.origin, 1.0, 64, a, "scan")
        compare_ldni(outs[a].numpy(), ref, DIAG)


def test_repeatable_bitwise(ldni):
    """Two calls give bit-identical LDNIs (slot order is atomic, but the
    per-ray sort fixes the final order)."""
    A, _ = M.pr1_pair()
    grid = ldni.Grid.cube(O3, 1.0, 128)
    x = [L.numpy() for L in ldni.sample(*A, grid, "all")]
    y = [L.numpy() for L in ldni.sample(*A, grid, "all")]
    for a in range(3):
        for k in ("offsets", "depth", "nrm", "tri"):
            assert np.array_equal(x[a][k], y[a][k])


@pytest.mark.parametrize("res", [1024, 2048])
def test_scale_sphere_full_size(ldni, res):
    """The 1,310,720-triangle noisy icosphere at both resolutions of the
    sampling-throughput workload, every ray compared with the oracle; the
    one-pass form with fixed two-layer capacity gives the same bits."""
    got, _ = _check_all_axes(ldni, M.scale_sphere(), res)
    grid = ldni.Grid.cube(O3, 1.0, res)
    one = ldni.sample_learned(*M.scale_sphere(), grid, "all", net=None, layers=2)
    assert all(ldni.identical(x, y) for x, y in zip(one, got))


def test_max_resolution_sampled_rays(ldni):
    """res 8192, the largest grid the library accepts: every ray's count."""
    v, t = M.icosphere(16, r=0.4, noise=0.03, seed=2)
    res = 8192
    grid = ldni.Grid.cube(O3, 1.0, res)
    L = ldni.sample(v, t, grid, 1)
    off = L.offsets.cpu().numpy().astype(np.int64)
    assert np.all(np.diff(off) % 2 == 0)
    ref = oracle.sample(v, t, grid.origin, 1.0, res, 1, "scan")
    assert np.array_equal(off, ref["offsets"])


def _count_then_fill(ldni, binned, first, second, grid, fills, fresh=False):
    """ldni_sample_count of mesh `first`, then `fills` times ldni_sample_fill of
    mesh `second` on the same workspace and offsets (fresh: the last one into
    arrays of its own).  Returns the images and each fill's status; the bytes
    around the workspace and past the arrays are checked."""
    import ctypes
    from paper_1009_0794_gb300 import _lib
    lib = _lib.load()
    count = lib.ldni_sample_binned_count if binned else lib.ldni_sample_count
    fill = lib.ldni_sample_binned_fill if binned else lib.ldni_sample_fill
    size = ldni.sample_binned_workspace_size if binned else ldni.sample_workspace_size
    up = lambda m: (torch.from_numpy(m[0]).cuda(), torch.from_numpy(m[1]).cuda())
    (v, t), (v2, t2) = up(first), up(second)
    assert t.shape == t2.shape
    need = size(len(v), len(t), grid.res, "all")
    buf = torch.full((need + (1 << 20),), 0x5A, dtype=torch.uint8, device="cuda")
    ws, past = buf[:need], buf[need:]
    info, g = ldni.new_info(), grid.c()
    offsets = [torch.zeros(grid.res ** 2 + 1, dtype=torch.int32, device="cuda") for _ in range(3)]
    arr = (_lib.Layers * 3)(*[_lib.Layers(o.data_ptr()) for o in offsets])
    args = lambda v, t, arr: (v.data_ptr(), len(v), t.data_ptr(), len(t), ctypes.byref(g), 3, arr, info.data_ptr(),
                              ws.data_ptr(), need, None)
    torch.cuda.synchronize()
    assert count(*args(v, t, arr)) == 0
    n = [int(x) for x in info[:3].tolist()]
    slack = 1000  # never written: the arrays end at the count

    def arrays(a):
        f = lambda x: torch.full((n[a] + slack,), x, dtype=torch.float32, device="cuda")
        return ldni.LDNI(grid, a, offsets[a], f(-7.0), f(-7.0), f(-7.0), f(-7.0),
                         torch.full((n[a] + slack,), -1, dtype=torch.int32, device="cuda"), n[a])

    outs, status = [arrays(a) for a in range(3)], []
    for k in range(fills):
        if fresh and k == fills - 1:
            outs = [arrays(a) for a in range(3)]
        info.zero_()
        arr = (_lib.Layers * 3)(*[o.c() for o in outs])
        torch.cuda.synchronize()
        assert fill(*args(v2, t2, arr)) == 0
        torch.cuda.synchronize()
        status.append(int(info[3].item()) & 0xFFFFFFFF)
    assert bool((past == 0x5A).all())
    for L in outs:
        for x in (L.depth, L.nx, L.ny, L.nz):
            assert bool((x[L.n:] == -7.0).all())
        assert bool((L.tri[L.n:] == -1).all())
    return outs, status


@pytest.mark.parametrize("binned", [False, True])
@pytest.mark.parametrize("mesh,res", [("box", 700), ("ball", 96), ("slabs", 65), ("flower", 200)])
def test_a_second_fill_is_reported_and_stays_in_place(ldni, binned, mesh, res):
    """The cursors of a count serve one fill: further ones report
    LDNI_ST_CAPACITY, leave the first one's samples as they are, and write
    nothing past the workspace (few triangles, many rays: the list of runs is
    its largest part) or outside a ray of the arrays."""
    from paper_1009_0794_gb300 import _lib
    m = {"box": M.box([-0.4, -0.3, -0.2], [0.3, 0.35, 0.4]), "ball": M.icosphere(8, r=0.4, noise=0.05, seed=1),
         "slabs": M.slab_stack(9, axis=1, seed=2), "flower": M.flower(60, 60)}[mesh]
    grid = ldni.Grid.cube((-0.5, -0.5, -0.5), 1.0, res)
    ref = ldni.sample(*m, grid, "all")
    outs, status = _count_then_fill(ldni, binned, m, m, grid, 4)
    assert not status[0] & _lib.ST_CAPACITY and all(s & _lib.ST_CAPACITY for s in status[1:])
    assert all(ldni.identical(x, y) for x, y in zip(outs, ref))
    outs, status = _count_then_fill(ldni, binned, m, m, grid, 3, fresh=True)
    assert status[2] & _lib.ST_CAPACITY
    _check_rays(outs, ref)


def _check_rays(outs, ref):
    """Every slot holds a sample of its own ray, or none (id -1)."""
    for L, R in zip(outs, ref):
        ray = np.repeat(np.arange(L.grid.res ** 2), np.diff(L.offsets.cpu().numpy()))
        rray = np.repeat(np.arange(L.grid.res ** 2), np.diff(R.offsets.cpu().numpy()))
        key = lambda r, t: r.astype(np.int64) << 32 | t.astype(np.int64)
        tri = L.tri[:L.n].cpu().numpy()
        have = key(ray, tri)[tri >= 0]
        assert np.isin(have, key(rray, R.tri[:R.n].cpu().numpy())).all(), L.axis


@pytest.mark.parametrize("binned", [False, True])
@pytest.mark.parametrize("change", ["wider", "twice", "fewer", "deeper"])
def test_a_fill_of_another_mesh_is_reported(ldni, binned, change):
    """More crossings than were counted (new rays, more per ray, on rays that
    were pairs and on others) or fewer: reported, and no slot of another ray
    is written."""
    from paper_1009_0794_gb300 import _lib
    def join(*ms):
        at = np.cumsum([0] + [len(m[0]) for m in ms[:-1]])
        return (np.concatenate([m[0] for m in ms]).astype(np.float32),
                np.concatenate([m[1] + k for m, k in zip(ms, at)]).astype(np.int32))
    A, T = M.box([-0.4, -0.3, -0.2], [0.3, 0.35, 0.4]), M.box([0.41, 0.41, 0.41], [0.42, 0.42, 0.42])
    one, two = join(A, T), join(A, A)
    S = M.slab_stack(7, axis=0, seed=5)
    W = ((S[0] * np.float32([1, 1.15, 0.9])).astype(np.float32), S[1])
    first, second = {"wider": (one, (one[0] * np.float32(1.1), one[1])), "twice": (one, two), "fewer": (two, one),
                     "deeper": (S, W)}[change]
    grid = ldni.Grid.cube((-0.5, -0.5, -0.5), 1.0, 90)
    ref = ldni.sample(*second, grid, "all")
    outs, status = _count_then_fill(ldni, binned, first, second, grid, 1)
    assert status[0] & _lib.ST_CAPACITY
    _check_rays(outs, ref)


def _sheets(k, seed, lo, hi, u0, u1):
    """k open sheets across the x-axis at random depths in [lo, hi], listed in
    random order: every x-ray through [u0, u1]^2 has exactly k samples."""
    rng = np.random.default_rng(seed)
    d = rng.permutation(np.linspace(lo, hi, k)).astype(np.float32)
    v = np.array([[x, y, z] for x in d for y, z in ((u0, u0), (u1, u0), (u1, u1), (u0, u1))], np.float32)
    t = np.array([[4 * i + a, 4 * i + b, 4 * i + c] for i in range(k) for a, b, c in ((0, 1, 2), (0, 2, 3))], np.int32)
    return v, t


@pytest.mark.parametrize("packed", [False, True])
@pytest.mark.parametrize("res", [64, 820])
def test_rays_of_any_count_in_either_ordering(ldni, packed, res):
    """Rays of 0 to 9, 40 and 300 samples side by side, odd counts among them,
    in images small enough to be ordered in one kernel and in three large ones
    that take two (820^2: 2.02 M rays): ids by ascending depth, the same in the
    call for all images, the one for one image and the binned form."""
    parts, at, base = [], [], 0
    for j, k in enumerate([1, 2, 3, 4, 5, 6, 7, 8, 9, 40, 300]):
        u0 = -0.48 + 0.085 * j
        m = _sheets(k, j, -0.45, 0.45, u0, u0 + (0.07 if k < 40 else 3.0 / res))
        parts.append((m[0], m[1] + base))
        base += len(m[0])
    v, t = np.concatenate([m[0] for m in parts]), np.concatenate([m[1] for m in parts])
    order = np.random.default_rng(res).permutation(len(t))
    t = t[order]
    grid = ldni.Grid.cube(O3, 1.0, res)
    got = ldni.sample(v, t, grid, "all", packed=packed)
    one = ldni.sample(v, t, grid, 0, packed=packed)
    binned = ldni.sample(v, t, grid, "all", mode="binned2", packed=packed)
    assert ldni.identical(got[0], one)
    assert all(ldni.identical(x, y) for x, y in zip(got, binned))
    g = got[0].numpy()
    counts = np.diff(g["offsets"])
    assert set(np.unique(counts)) >= {0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 40, 300}
    ray = np.repeat(np.arange(res * res), counts)
    x = v[t[g["tri"]][:, 0], 0]  # a sheet's depth
    assert np.all(np.abs(g["depth"] - x) <= 1e-5 * DIAG)  # the sampling bound
    assert np.array_equal(np.lexsort((g["tri"], g["depth"], ray)), np.arange(len(ray)))
    same = ray[1:] == ray[:-1]
    assert np.all(x[1:][same] > x[:-1][same])  # one sample of every sheet
    e1, e2 = v[t[:, 1]] - v[t[:, 0]], v[t[:, 2]] - v[t[:, 0]]
    nrm = np.cross(e1.astype(np.float64), e2.astype(np.float64))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    if packed:
        code = np.rint((nrm[g["tri"]] + 1) * 127.5).astype(np.uint32)
        assert np.array_equal(g["nrm8"], code[:, 0] | (code[:, 1] << 8) | (code[:, 2] << 16))
    else:
        assert np.all(np.abs(g["nrm"] - nrm[g["tri"]]) <= 1e-5)  # the sampling bound


@pytest.mark.parametrize("res", [40, 400, 816, 817])
def test_big_pairs_beside_and_after_the_triangles(ldni, res):
    """Twelve faces in images small and large enough for the fill to take their
    pairs beside the triangles and in a launch of their own (from 2 M rays)."""
    m = M.box([-0.41, -0.33, -0.27], [0.35, 0.39, 0.44])
    grid = ldni.Grid.cube(O3, 1.0, res)
    assert (3 * res * res > 2000000) == (res >= 817)
    _check_all_axes(ldni, m, res)
    assert all(ldni.identical(x, y) for x, y in zip(ldni.sample(*m, grid, "all"),
                                                    ldni.sample(*m, grid, "all", mode="binned2")))
