"""Chains of unions in one call (ldni_union_chain, Sections 4.1.1 and 4.2)
and the bounded device waits, through the C ABI.

The chain's result must equal the step-by-step chain of ldni_boolean calls
and the oracle's step-by-step unions bit for bit (counts, depths, normals,
ids), with and without small-interval removal at every step, for one or
three images per call and for packed normals.  A ray whose accumulated
result outgrows the per-ray limit is reported, not answered wrongly.  The
timeout path of a bounded wait is made to run out on purpose (a word that
nothing sets) and must report LDNI_ST_TIMEOUT with the device still usable.
"""
import ctypes

import numpy as np
import pytest

import meshgen as M
import oracle
from ldni_compare import bit_equal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

O3 = (-0.5, -0.5, -0.5)


@pytest.fixture(scope="module")
def ldni():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1009_0794_gb300 as pkg
    pkg._lib.load()
    return pkg


def _sweep_parts(ldni, steps, res, packed=False):
    base = M.torus(R=0.16, r=0.06, nu=48, nv=24)
    offs = M.helix_offsets(steps, seed=11, radius=0.12, pitch=0.4, turns=1.5)
    grid = ldni.Grid.cube(O3, 1.0, res)
    return [ldni.sample(*M.translate(base, d), grid, "all", packed=packed) for d in offs]


def _stepwise(ldni, P, eps):
    acc = P[0]
    for k in range(1, len(P)):
        acc = ldni.boolean(acc, P[k], "union", eps=eps)
    return acc


@pytest.mark.parametrize("eps", [0.0, 1e-2])
def test_chain_equals_stepwise_and_oracle(ldni, eps):
    steps, res = 24, 80
    parts = _sweep_parts(ldni, steps, res)
    for a in range(3):
        P = [parts[k][a] for k in range(steps)]
        run, finish = ldni.union_chain(P, eps=eps)
        run()
        got = finish()
        want = _stepwise(ldni, P, eps)
        assert ldni.identical(got, want), a
        acc = P[0].numpy()
        for k in range(1, steps):
            acc = oracle.boolean(acc, P[k].numpy(), "union", eps=eps)
        assert bit_equal(got.numpy(), acc), a


def test_three_images_in_one_call_and_graph(ldni):
    steps, res = 16, 96
    parts = _sweep_parts(ldni, steps, res)
    per_image = [[parts[k][a] for k in range(steps)] for a in range(3)]
    run, finish = ldni.union_chain_many(per_image)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        run(stream=s)  # warm-up outside capture
    torch.cuda.current_stream().wait_stream(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        run(stream=s)
    g.replay()
    torch.cuda.synchronize()
    outs = finish()
    for a in range(3):
        r1, f1 = ldni.union_chain(per_image[a])
        r1()
        assert ldni.identical(outs[a], f1()), a
        assert ldni.identical(outs[a], _stepwise(ldni, per_image[a], 0.0)), a


def test_packed_normals_chain(ldni):
    steps, res = 12, 64
    parts = _sweep_parts(ldni, steps, res, packed=True)
    for a in range(3):
        P = [parts[k][a] for k in range(steps)]
        run, finish = ldni.union_chain(P)
        run()
        assert ldni.identical(finish(), _stepwise(ldni, P, 0.0)), a


def test_short_chains_and_empty_parts(ldni):
    grid = ldni.Grid.cube(O3, 1.0, 48)
    A, B = M.pr1_pair()
    LA, LB = ldni.sample(*A, grid, 2), ldni.sample(*B, grid, 2)
    E = ldni.sample(np.zeros((3, 3), np.float32), np.zeros((0, 3), np.int32), grid, 2)
    run, finish = ldni.union_chain([LA])  # one part: the part itself
    run()
    assert ldni.identical(finish(), LA)
    for P in ([LA, LB], [LA, E, LB, E], [E, LA, E], [E, E]):
        run, finish = ldni.union_chain(P, eps=1e-5)
        run()
        assert ldni.identical(finish(), _stepwise(ldni, P, 1e-5))


def test_deep_rays_are_reported(ldni):
    """A stack of 40 slabs gives rays of 80 samples, more than a ray's
    accumulated result may hold: the call reports it instead of answering."""
    grid = ldni.Grid.cube(O3, 1.0, 16)
    L = ldni.sample(*M.slab_stack(40, axis=0, seed=1), grid, 0)
    assert int(L.counts().max()) > 64
    run, finish = ldni.union_chain([L, L])
    run()
    with pytest.raises(ldni.LDNIError):
        finish()


def test_bounded_wait_runs_out(ldni):
    """The bounded wait on a word that nothing sets gives up after the set
    number of polls and reports LDNI_ST_TIMEOUT; the device keeps working."""
    lib = ldni._lib.load()
    assert lib.ldni_set_wait_limit(-1) == -1
    assert lib.ldni_set_wait_limit(2000) == 0
    try:
        assert lib.ldni_get_wait_limit() == 2000
        info = ldni.new_info()
        assert lib.ldni_wait_selftest(info.data_ptr(), None) == 0
        torch.cuda.synchronize()
        assert ldni.info_decode(info)["status"] & ldni._lib.ST_TIMEOUT
    finally:
        assert lib.ldni_set_wait_limit(0) == 0
    assert lib.ldni_get_wait_limit() == 1 << 22
    # the device still answers: a Boolean through the one-launch look-back form
    A, B = M.pr1_pair()
    grid = ldni.Grid.cube(O3, 1.0, 128)
    LA, LB = ldni.sample(*A, grid, 0), ldni.sample(*B, grid, 0)
    got = ldni.boolean(LA, LB, "union").numpy()
    assert bit_equal(got, oracle.boolean(LA.numpy(), LB.numpy(), "union"))


def test_tiny_wait_limit_terminates(ldni):
    """With one poll per wait the look-back of a one-launch Boolean over many
    tiles may give up; the call still ends, and either its result is right
    or the timeout is reported."""
    from paper_1009_0794_gb300 import tune
    lib = ldni._lib.load()
    grid = ldni.Grid.cube(O3, 1.0, 512)
    (va, ta), (vb, tb) = M.pr1_pair()
    LA, LB = ldni.sample(va, ta, grid, 0), ldni.sample(vb, tb, grid, 0)
    ref = oracle.boolean(LA.numpy(), LB.numpy(), "union")
    prev = tune.set(bool_split=0, bool_tile_rays=256)
    assert lib.ldni_set_wait_limit(1) == 0
    try:
        info = ldni.new_info()
        out = ldni.boolean(LA, LB, "union", info=info, sync=False)
        torch.cuda.synchronize()
        st = ldni.info_decode(info)["status"]
        if not st & ldni._lib.ST_TIMEOUT:
            out.n = ldni.info_decode(info)["n"][0]
            assert bit_equal(out.numpy(), ref)
    finally:
        lib.ldni_set_wait_limit(0)
        tune.set(**prev)


def _random_part(ldni, grid, rng, most, levels):
    """An image of random intervals whose ends are multiples of 1 / levels:
    shared depths, touching and empty intervals across and within parts."""
    N = grid.res * grid.res
    depth, off = [], [0]
    for _ in range(N):
        k = 2 * int(rng.integers(0, most + 1)) if rng.random() < 0.6 else 0
        depth += sorted(rng.integers(0, levels, size=k).tolist())
        off.append(off[-1] + k)
    n = off[-1]
    t = lambda x, dt: torch.from_numpy(np.asarray(x, dt)).cuda()
    nrm = rng.standard_normal((3, n)).astype(np.float32)
    return ldni.LDNI(grid, 0, t(off, np.int32), t(np.asarray(depth) / levels, np.float32), *[t(x, np.float32) for x in nrm],
                     t(rng.integers(0, 1000, size=n), np.int32), n)


@pytest.mark.parametrize("count,most,levels,res", [(2, 1, 8, 9), (5, 3, 4096, 13), (12, 2, 64, 16), (64, 1, 5000, 7),
                                                   (70, 1, 300, 7), (66, 1, 40, 5), (3, 14, 100000, 11)])
def test_random_intervals(ldni, count, most, levels, res):
    """Every form a ray's result takes, against the step-by-step unions: ties
    and touching intervals, a few or many disjoint ones, results longer than
    the sources kept between the passes, more than 64 parts."""
    rng = np.random.default_rng(count * 100 + most)
    grid = ldni.Grid.cube(O3, 1.0, res)
    P = [_random_part(ldni, grid, rng, most, levels) for _ in range(count)]
    for eps in (0.0, 0.01):
        run, finish = ldni.union_chain(P, eps=eps)
        run()
        try:
            got = finish()
        except ldni.LDNIError as e:
            assert e.code == -4 and count >= 64  # a ray of more than 64 samples at some step
            continue
        assert ldni.identical(got, _stepwise(ldni, P, eps)), eps


def _intervals(ldni, grid, counts, lo, hi, shift, seed):
    """An image with counts[p] disjoint intervals on ray p, evenly spaced in
    [lo, hi] and moved by `shift` of their spacing."""
    rng = np.random.default_rng(seed)
    counts = np.asarray(counts)
    off = np.concatenate([[0], np.cumsum(2 * counts)])
    n = int(off[-1])
    j = np.arange(n) - np.repeat(off[:-1], 2 * counts)
    k = np.repeat(np.maximum(counts, 1), 2 * counts)
    depth = lo + (hi - lo) * (j // 2 + shift + 0.4 * (j & 1)) / (k + 1)
    t = lambda x, dt: torch.from_numpy(np.ascontiguousarray(x, dt)).cuda()
    nrm = rng.standard_normal((3, n))
    return ldni.LDNI(grid, 0, t(off, np.int32), t(depth, np.float32), *[t(x, np.float32) for x in nrm],
                     t(rng.integers(0, 1000, size=n), np.int32), n)


def _layers_needed(ldni, P, eps):
    """Most samples on a ray at any step, the first part alone included."""
    acc, most = P[0], int(P[0].counts().max())
    for k in range(1, len(P)):
        acc = ldni.boolean(acc, P[k], "union", eps=eps)
        most = max(most, int(acc.counts().max()))
    return most


@pytest.mark.parametrize("first,second,count", [(32, 0, 2), (32, 1, 2), (33, 0, 2), (33, 0, 1), (16, 16, 3), (20, 13, 2),
                                                (31, 1, 70)])
@pytest.mark.parametrize("eps", [0.0, 1e-6])
def test_limit_of_layers_exactly(ldni, first, second, count, eps):
    """A chain is reported (a ray of more than 64 samples) exactly when a step
    of the step-by-step unions has such a ray, a last part over everything
    notwithstanding."""
    res = 6
    grid = ldni.Grid.cube(O3, 1.0, res)
    at = np.zeros(res * res, np.int64)
    at[[3, 17, 35]] = 1
    P = [_intervals(ldni, grid, first * at, -0.4, 0.4, 0.0, 1)]
    if count > 1:
        P.append(_intervals(ldni, grid, second * at, -0.4, 0.4, 0.5, 2))  # in the gaps of equally many, else across
    P += [_intervals(ldni, grid, at, -0.45, 2.0, 0.0, 3) for _ in range(count - len(P))]
    most = _layers_needed(ldni, P, eps)
    run, finish = ldni.union_chain(P, eps=eps)
    run()
    if most > 64:
        with pytest.raises(ldni.LDNIError) as e:
            finish()
        assert e.value.code == -4
    else:
        assert ldni.identical(finish(), _stepwise(ldni, P, eps))


@pytest.mark.parametrize("eps", [0.0, 1e-7])
def test_more_intervals_than_records(ldni, eps):
    """An image whose result has more intervals than the workspace has records
    (2 M for 160,000 rays): rays of one to four, of more, and empty ones, with
    and without records, equal the step-by-step unions; so does one part
    alone."""
    res = 400
    grid = ldni.Grid.cube(O3, 1.0, res)
    rng = np.random.default_rng(9)
    c = np.where(rng.random(res * res) < 0.75, rng.integers(16, 31, size=res * res), rng.integers(0, 4, size=res * res))
    A = _intervals(ldni, grid, c, -0.45, 0.45, 0.0, 4)
    B = _intervals(ldni, grid, rng.integers(0, 2, size=res * res), -0.3, 0.3, 0.2, 5)
    for P in ([A, B, A], [A]):
        run, finish = ldni.union_chain(P, eps=eps)
        run()
        got = finish()
        assert got.n > 2 * (2 << 20)
        assert ldni.identical(got, _stepwise(ldni, P, eps))


def test_workspace_stays_small(ldni):
    """About 16 bytes a ray for large images."""
    for res in (2048, 4096, 8192):
        assert ldni.union_chain_workspace_size(res, 3) <= 17 * 3 * res * res
