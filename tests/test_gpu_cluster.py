"""One-cluster CG (csrc/cluster.cu) against the two-kernel engine (csrc/pcg.cu).

Both engines do the same arithmetic, so a solve must give the same bits, CG
iterations and sweeps with either.  A profiled batch runs the two-kernel
engine; sizes lie at the edges of tiles (30 nodes), of cluster sizes and of
reduction chunks (256 tiles), and beyond what a cluster keeps on chip.  No
tolerance: equality."""
import numpy as np
import pytest

import meshgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sso():
    import paper_2407_20026_gb300 as pkg
    from paper_2407_20026_gb300 import _build
    _build.build()
    return pkg


def _run(sso, meshes, profiled, g=None, **kw):
    models = [sso.Model(m) for m in meshes]
    batch = sso.Batch(models)
    batch.set_profiling(profiled)
    stats = batch.solve(sso.options(**kw), raise_on_error=False)
    batch.gradient(g=g, raise_on_error=False)
    batch.set_profiling(False)
    return stats, [m.result() for m in models]


def _same(sso, meshes, g=None, **kw):
    a, ra = _run(sso, meshes, False, g, **kw)
    b, rb = _run(sso, meshes, True, g, **kw)
    for x, y, p, q in zip(a, b, ra, rb):
        for k in ("status", "iterations", "sweeps", "rel_residual"):
            assert x[k] == y[k], (k, x, y)
        for k in ("u", "C", "dz", "dt", "lam"):
            assert np.array_equal(p[k], q[k]), k
    return a


def _strip(n):
    """A clamped-free beam line of n nodes, numbered along it (n = 30 k + r)."""
    m = meshgen.arch2d(n_el=n - 1, E=2e11)
    m["xyz"][:, 1] = 0.1 * np.sin(np.arange(n))
    return m


@pytest.mark.parametrize("precond", ["jacobi", "block_jacobi", "two_level"])
@pytest.mark.parametrize("n", [2, 29, 30, 31, 61])
def test_tile_edges(sso, n, precond):
    _same(sso, [_strip(n)], precond=precond, rtol=1e-6, max_iter=400)


@pytest.mark.parametrize("precond", ["jacobi", "block_jacobi", "two_level"])
@pytest.mark.parametrize("size", [3, 8, 19, 33, 64])
def test_shells(sso, size, precond):
    # 16 to 4,225 nodes: one to sixteen CTAs, K resident or through L2
    _same(sso, [meshgen.shell(size, seed=size)], precond=precond, rtol=1e-6, max_iter=3000)


@pytest.mark.parametrize("precond", ["block_jacobi", "two_level"])
@pytest.mark.parametrize("side", [87, 88, 100])
def test_reduction_chunks(sso, side, precond):
    # 7,569, 7,744 and 10,000 nodes: 253, 259 and 334 tiles, one and two chunks
    _same(sso, [meshgen.gridshell(side, seed=side)], precond=precond, rtol=1e-6, max_iter=700)


def test_scattered_numbering_and_hub(sso):
    # windows as wide as the system; one row of as many blocks as it has nodes
    m = meshgen.gridshell(17, seed=4)
    rng = np.random.default_rng(5)
    perm = rng.permutation(m["xyz"].shape[0])
    inv = np.argsort(perm)
    m["beam_conn"] = inv[m["beam_conn"]].astype(np.int32)
    for k in ("xyz", "fixed", "nodal_load"):
        m[k] = m[k][perm]
    _same(sso, [m], rtol=1e-6)
    h = meshgen.gridshell(9, seed=6)
    hub = 40
    far = np.array([j for j in range(81) if j not in (hub,) and (j // 9 + j) % 3 == 0], np.int32)
    have = {tuple(sorted(c)) for c in h["beam_conn"].tolist()}
    new = np.array([(hub, j) for j in far if tuple(sorted((hub, int(j)))) not in have], np.int32)
    h["beam_conn"] = np.concatenate([h["beam_conn"], new])
    h["beam_props"] = np.tile(h["beam_props"][0], (h["beam_conn"].shape[0], 1))
    _same(sso, [h], rtol=1e-6)


def test_mixed_batch_more_systems_than_clusters_and_adjoint(sso):
    meshes = [meshgen.shell(20, seed=1), meshgen.gridshell(10), meshgen.gridshell(50, seed=2),
              meshgen.shell(7)] + [meshgen.shell(33, seed=s) for s in range(20)]
    rng = np.random.default_rng(9)
    g = [rng.standard_normal(6 * m["xyz"].shape[0]) * (k % 2) for k, m in enumerate(meshes)]
    _same(sso, meshes, g=g, rtol=1e-6, max_iter=4000)


@pytest.mark.parametrize("precond", ["jacobi", "block_jacobi", "two_level"])
def test_launches_of_systems_with_different_warps(sso, precond):
    # one launch's CTAs have the warps of its largest system
    meshes = [meshgen.gridshell(side, seed=side) for side in range(31, 101, 3)]
    _same(sso, meshes, precond=precond, rtol=1e-6, max_iter=300)


def test_many_launches_and_caps(sso):
    # a wall-clock cap launches iters_per_launch steps at a time: the state
    # passes through memory between launches, also in the middle of a sweep
    m = meshgen.shell(12, seed=3)
    whole = _run(sso, [m], False, rtol=1e-8)
    for n in (1, 7, 64):
        cut = _run(sso, [m], False, rtol=1e-8, timeout_ms=6e4, iters_per_launch=n)
        assert cut[0][0]["iterations"] == whole[0][0]["iterations"]
        assert np.array_equal(cut[1][0]["u"], whole[1][0]["u"])
    two = [_run(sso, [m], False, rtol=1e-8, precond="two_level", **kw)
           for kw in ({}, {"timeout_ms": 6e4, "iters_per_launch": 5})]
    assert np.array_equal(two[0][1][0]["u"], two[1][1][0]["u"])
    _same(sso, [m], rtol=1e-8, max_iter=50)
    _same(sso, [m], rtol=1e-8, max_sweeps=1)


def test_zero_load_mechanism_and_warm_start(sso):
    m = meshgen.gridshell(10)
    z = dict(m, nodal_load=np.zeros_like(m["nodal_load"]))
    assert _same(sso, [z], rtol=1e-8)[0]["iterations"] == 0
    free = dict(m, fixed=np.zeros_like(m["fixed"]))
    assert _same(sso, [free], rtol=1e-8, max_iter=2000)[0]["status"] != 0
    mdl = sso.Model(m)
    mdl.solve(rtol=1e-4)
    assert mdl.solve(rtol=1e-8, warm_start=1)["status"] == 0


def test_server_switches_engines(sso):
    # a system beyond the engine's size joins and leaves while others run: the
    # server's running systems change engines in the middle of their sweeps
    from paper_2407_20026_gb300.serve import Server
    opts = sso.options(rtol=1e-4)
    small = [meshgen.gridshell(side, seed=side) for side in (60, 30, 90, 45, 20, 100)]
    large = meshgen.gridshell(176, seed=1)  # 30,976 nodes: five reduction chunks
    srv = Server(opts, max_systems=8)
    tickets = [srv.submit(m) for m in small[:3]]
    for _ in range(3):
        srv.step()
    tickets.append(srv.submit(large))
    tickets += [srv.submit(m) for m in small[3:]]
    while any(srv.step()):
        pass
    for m, t in zip(small[:3] + [large] + small[3:], tickets):
        mdl = sso.Model(m)
        mdl.solve(opts)
        mdl.gradient()
        want, got = mdl.result(), srv.poll(t)
        assert got["stats"]["status"] == 0
        assert np.array_equal(got["u"], want["u"]) and got["C"] == want["C"]
    srv.close()


@pytest.mark.parametrize("precond", ["jacobi", "block_jacobi"])
@pytest.mark.parametrize("nodes", [30690, 30720, 30721, 92160, 92161])
def test_teams_of_all_sms(sso, nodes, precond):
    # systems beyond a cluster: 1,023 to 1,025 tiles (four and five reduction
    # chunks), twelve chunks, and one node more, which takes the two kernels
    _same(sso, [_strip(nodes)], precond=precond, rtol=1e-6, max_iter=200)


@pytest.mark.parametrize("count", [2, 3, 5])
def test_batches_of_teams(sso, count):
    # several teams in a launch, several launches, and a cluster beside them
    meshes = [meshgen.gridshell(110 + 9 * k, seed=k) for k in range(count)]
    _same(sso, meshes + [meshgen.shell(9)], rtol=1e-6, max_iter=300)


def test_teams_many_launches_and_adjoint(sso):
    m = meshgen.shell(90, seed=2)
    whole = _run(sso, [m], False, rtol=1e-6, max_iter=600)
    cut = _run(sso, [m], False, rtol=1e-6, max_iter=600, timeout_ms=6e4, iters_per_launch=7)
    assert cut[0][0]["iterations"] == whole[0][0]["iterations"]
    assert np.array_equal(cut[1][0]["u"], whole[1][0]["u"])
    g = np.random.default_rng(3).standard_normal(6 * m["xyz"].shape[0])
    _same(sso, [m], g=[g], rtol=1e-6, max_iter=600)


@pytest.mark.parametrize("precond", ["jacobi", "block_jacobi"])
@pytest.mark.parametrize("n", [2, 29, 30, 31, 61, 4591])
def test_fp64_tile_edges(sso, n, precond):
    # 4,591 nodes: 154 tiles, more than one on some CTAs
    _same(sso, [_strip(n)], precision="fp64", precond=precond, rtol=1e-10, max_iter=400)


@pytest.mark.parametrize("precond", ["jacobi", "block_jacobi"])
def test_fp64_batches_launches_and_adjoint(sso, precond):
    kw = dict(precision="fp64", precond=precond, rtol=1e-10, max_iter=500)
    one = meshgen.shell(24, seed=2)  # K beyond a CTA's shared memory where CTAs are few
    g = np.random.default_rng(3).standard_normal(6 * one["xyz"].shape[0])
    _same(sso, [one], g=[g], **kw)
    _same(sso, [meshgen.gridshell(41, seed=1)] * 3 + [meshgen.shell(9), meshgen.gridshell(75)], **kw)
    _same(sso, [meshgen.shell(16, seed=s) for s in range(24)], **kw)
    whole = _run(sso, [one], False, **kw)
    cut = _run(sso, [one], False, timeout_ms=6e4, iters_per_launch=7, **kw)
    assert cut[0][0]["iterations"] == whole[0][0]["iterations"]
    assert np.array_equal(cut[1][0]["u"], whole[1][0]["u"])
    warm = sso.Model(meshgen.gridshell(20))
    warm.solve(precision="fp64", precond=precond, rtol=1e-6)
    assert warm.solve(precision="fp64", precond=precond, rtol=1e-10, warm_start=1)["status"] == 0


@pytest.mark.parametrize("steps", [1, 4, 5, 6, 7])
def test_team_launches_begin_in_every_state(sso, steps):
    # a team per launch of a few steps, over several sweeps to convergence:
    # launches begin in the first residual, the iteration, the fold and the
    # residual after it (1 step: two kernels)
    m = meshgen.gridshell(110, seed=5)
    kw = dict(rtol=1e-6, inner_rtol=0.1, max_iter=20000)
    want = _same(sso, [m], **kw)
    whole = _run(sso, [m], False, **kw)
    cut = _run(sso, [m], False, timeout_ms=1e5, iters_per_launch=steps, **kw)
    assert want[0]["status"] == 0 and want[0]["sweeps"] > 2
    for k in ("status", "iterations", "sweeps", "rel_residual"):
        assert cut[0][0][k] == whole[0][0][k] == want[0][k], k
    for k in ("u", "C", "dz", "dt", "lam"):
        assert np.array_equal(cut[1][0][k], whole[1][0][k]), k


def test_team_launch_that_begins_in_the_fold_at_the_cap(sso):
    # the first launch's 1,024 steps end with the last iteration of the cap
    m = meshgen.shell(90, seed=2)
    st = _same(sso, [m], rtol=1e-6, max_iter=1023)
    assert st[0]["iterations"] == 1023 and st[0]["sweeps"] == 1


@pytest.mark.parametrize("size,precond,steps", [
    (90, "jacobi", 4), (90, "block_jacobi", 4), (20, "jacobi", 4), (20, "block_jacobi", 5),
    (20, "two_level", 10), (33, "two_level", 13)])
def test_launches_that_begin_in_the_fold_and_after_it(sso, size, precond, steps):
    # teams (90 x 90) and clusters; the residual, a sweep of max_iter iterations,
    # the fold and the second residual: launch 11 begins in the sweep's last
    # iteration, in the fold, in the residual after it
    m = meshgen.shell(size, seed=2)
    for max_iter in (10 * steps, 10 * steps - 1, 10 * steps - 2):
        kw = dict(rtol=1e-8, precond=precond, inner_rtol=1e-7, max_iter=max_iter)
        st = _same(sso, [m], **kw)
        assert st[0]["iterations"] == max_iter and st[0]["sweeps"] == 1
        whole = _run(sso, [m], False, **kw)
        cut = _run(sso, [m], False, timeout_ms=1e5, iters_per_launch=steps, **kw)
        for k in ("status", "iterations", "sweeps", "rel_residual"):
            assert cut[0][0][k] == whole[0][0][k], k
        for k in ("u", "C", "dz", "dt", "lam"):
            assert np.array_equal(cut[1][0][k], whole[1][0][k]), k


def test_teams_of_several_threads_and_parts(sso):
    # solves with teams at the same time (each plans for its share of the SMs)
    # give the bits of each solve alone
    import threading
    cases = [(meshgen.gridshell(10, seed=1), dict(precision="fp64", rtol=1e-10)),
             (meshgen.gridshell(41, seed=2), dict(precision="fp64", rtol=1e-10)),
             (meshgen.gridshell(100, seed=3), dict(precision="fp64", rtol=1e-10, max_iter=400)),
             (meshgen.shell(90, seed=4), dict(rtol=1e-6, max_iter=600)),
             (meshgen.gridshell(110, seed=5), dict(rtol=1e-6, max_iter=600)),
             (meshgen.shell(30, seed=6), dict(rtol=1e-6, max_iter=600))] * 2
    want = [_run(sso, [m], True, **kw) for m, kw in cases]
    models = [sso.Model(m) for m, _ in cases]
    got = [None] * len(cases)

    def work(i):
        for _ in range(3):
            st = models[i].solve(sso.options(**cases[i][1]), raise_on_error=False)
            got[i] = (st, models[i].result())
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(cases))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for (st, res), (wst, wres) in zip(got, want):
        assert (st["status"], st["iterations"]) == (wst[0]["status"], wst[0]["iterations"])
        assert np.array_equal(res["u"], wres[0]["u"])
    # 32 models and more run as parts on threads of their own
    _same(sso, [meshgen.gridshell(9 + k % 3, seed=k) for k in range(34)], precision="fp64",
          rtol=1e-10)
    _same(sso, [meshgen.gridshell(110, seed=k) for k in range(32)], rtol=1e-6, max_iter=60)


@pytest.mark.parametrize("precond", ["jacobi", "block_jacobi"])
def test_fp64_batches_of_unequal_and_many_systems(sso, precond):
    # teams of different sizes in a launch, of one CTA, more systems than a
    # launch takes, launches planned again as systems finish, a split batch
    kw = dict(precision="fp64", precond=precond, rtol=1e-10, max_iter=1500)
    sides = [8, 13, 19, 24, 30, 41, 52, 60]
    _same(sso, [meshgen.gridshell(s, seed=s) for s in sides] + [_strip(2), meshgen.shell(24)], **kw)
    many = [meshgen.gridshell(6 + k % 5, seed=k) for k in range(170)]
    _same(sso, many + [meshgen.gridshell(41, seed=1)], **kw)
    g = np.random.default_rng(4)
    meshes = [meshgen.gridshell(7 + 2 * k, seed=k) for k in range(12)]
    _same(sso, meshes, g=[g.standard_normal(6 * m["xyz"].shape[0]) * (k % 3 == 0)
                          for k, m in enumerate(meshes)], **kw)


@pytest.mark.parametrize("side", [191, 233, 234])
def test_fp64_largest_teams(sso, side):
    # 1,217 and 1,810 tiles on CTAs of 9 and 12 tiles; 1,826, which takes two kernels
    _same(sso, [meshgen.gridshell(side, seed=side)], precision="fp64", rtol=1e-10, max_iter=60)


def test_teams_beside_a_server(sso):
    # a server's clusters and set-up kernels between the teams of two batches
    import threading
    from paper_2407_20026_gb300.serve import Server
    opts = sso.options(rtol=1e-4)
    meshes = [meshgen.gridshell(side, seed=side) for side in (60, 30, 90, 45, 20, 100)] * 2
    team = [meshgen.shell(90, seed=3), meshgen.gridshell(110, seed=4)]
    want = _run(sso, team, True, rtol=1e-6, max_iter=900)
    kw64 = dict(precision="fp64", rtol=1e-10, max_iter=400)
    small = [meshgen.gridshell(9 + 8 * k, seed=k) for k in range(6)]
    want64 = _run(sso, small, True, **kw64)
    got = {}

    def solve(key, ms, kw):
        got[key] = [_run(sso, ms, False, **kw) for _ in range(3)]
    threads = [threading.Thread(target=solve, args=a) for a in
               (("team", team, dict(rtol=1e-6, max_iter=900)), ("fp64", small, kw64))]
    srv = Server(opts, max_systems=6)
    tickets = [srv.submit(m) for m in meshes]
    for t in threads:
        t.start()
    while any(srv.step()):
        pass
    for t in threads:
        t.join()
    for key, ref in (("team", want), ("fp64", want64)):
        for stats, results in got[key]:
            for a, b, x, y in zip(stats, ref[0], results, ref[1]):
                assert (a["status"], a["iterations"]) == (b["status"], b["iterations"])
                assert np.array_equal(x["u"], y["u"]) and np.array_equal(x["dz"], y["dz"])
    for m, t in zip(meshes, tickets):
        mdl = sso.Model(m)
        mdl.solve(opts)
        res = srv.poll(t)
        assert res["stats"]["status"] == 0 and np.array_equal(res["u"], mdl.result()["u"])
    srv.close()


def _shuffled(m, seed):
    n = m["xyz"].shape[0]
    perm = np.random.default_rng(seed).permutation(n)
    inv = np.argsort(perm)
    m = dict(m)
    for k in ("beam_conn", "quad_conn"):
        if len(m[k]):
            m[k] = inv[m[k]].astype(np.int32)
    for k in ("xyz", "fixed", "nodal_load"):
        m[k] = m[k][perm]
    return m


@pytest.mark.parametrize("side,count", [(50, 1), (75, 1), (90, 1), (70, 24)])
def test_wide_windows(sso, side, count):
    # shuffled numbering: windows as wide as the system, on clusters, teams and,
    # where it is faster (24 systems), two kernels an iteration
    meshes = [_shuffled(meshgen.gridshell(side, seed=k), k) for k in range(count)]
    kw = dict(rtol=1e-10, max_iter=120)
    _same(sso, meshes, **kw)
    before = sso.kernel_launches()
    sso.Batch([sso.Model(m) for m in meshes]).solve(sso.options(**kw), raise_on_error=False)
    two_kernels = sso.kernel_launches() - before >= 2 * 120
    assert two_kernels == (count == 24)
