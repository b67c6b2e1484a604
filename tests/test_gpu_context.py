"""Contexts: what creating one costs, the scratch it holds, and the launch configuration it
reports, takes and runs."""
import math
import time

import pytest

from oracle.oracle import Oracle
from paper_2202_07989_gb300 import workloads as W

from .helpers import TOL_FP64, case, masked_fieldwise, need_gpu, rel_max_err, to_dev

pytestmark = pytest.mark.gpu


def _ctx(pb, precision=0):
    from paper_2202_07989_gb300 import es
    return es.Context(pb, precision)


def _create_ms(pb, form, torch):
    best = float("inf")
    for _ in range(5):
        t = time.perf_counter()
        ctx = _ctx(pb, form)
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
        del ctx
    return 1e3 * best


def test_fp64_context_creation_time():
    """An FP64 3D context, which picks its flux tiles among all extents, is created in at most
    twice the time of a mixed one (about 2.5 ms each at 256^3, nearly all of it allocations)."""
    torch = need_gpu()
    pb = W.random_problem(3, 2, (256, 256, 256))
    fp64, mixed = _create_ms(pb, 0, torch), _create_ms(pb, 1, torch)
    assert fp64 <= 2.0 * mixed, (fp64, mixed)


@pytest.mark.parametrize("N", [1, 2])
def test_mixed_3d_scratch(N):
    """A mixed 3D context holds no more than the FP64 one and its nine binary32 edge spacings a node
    (36 bytes, and those of one more layer of nodes)."""
    need_gpu()
    pb = W.random_problem(3, N, (64, 64, 64))
    fp64, mixed = _ctx(pb, 0).scratch_bytes, _ctx(pb, 1).scratch_bytes
    assert mixed - fp64 <= 36 * 65 ** 3, (mixed - fp64) / pb.ncell


@pytest.mark.parametrize("form", [0, 1])
def test_profile_counts_one_launch_per_direction(form):
    """Every flux class counts one launch per residual (in the 3D mixed form too, where the
    node-field pass precedes direction 1), so that time / launches is a launch's time."""
    torch = need_gpu()
    pb, JU, J, x, xdot = case(3, 2, (20, 12, 11), "periodic", seed=5)
    ctx = _ctx(pb, form)
    G = [to_dev(t, torch) for t in (JU, J, x, xdot)]
    ctx.es_profile(True)
    ctx.es_rhs(*G)
    prof = ctx.es_profile_read()
    ctx.es_profile(False)
    assert [prof["flux_k%d" % k][1] for k in (1, 2, 3)] == [1, 1, 1]


@pytest.mark.parametrize("n0", [124, 100])
def test_caller_fixed_grid_runs(n0):
    """A CTA count fixed by es_set_tuning is the one launched, also where it shares a factor with
    the segments per line (two here): two CTAs take 1/2 or, with a partial segment, 62/100 of the
    time of one (node counts), not the same."""
    torch = need_gpu()
    pb, JU, J, x, xdot = case(3, 1, (n0, 16, 16), "periodic", seed=6)
    ctx = _ctx(pb, 1)
    G = [to_dev(t, torch) for t in (JU, J, x, xdot)]
    ms = []
    for grid in (1, 2):
        ctx.es_set_tuning(0, 0, grid)
        assert ctx.es_get_tuning()[0][:4] == (0, 62, 4, grid)
        ctx.es_rhs(*G)
        ctx.es_profile(True)
        ctx.es_rhs(*G)
        ms.append(ctx.es_profile_read()["flux_k1"][0])
        ctx.es_profile(False)
    assert ms[0] >= 1.3 * ms[1], ms


@pytest.mark.parametrize("form", [0, 1])
def test_library_grid_is_reported(form):
    """The CTA count that the library chooses, lowered where lines end in a partial segment until it
    shares no factor with the segments per line, is the one es_get_tuning reports."""
    need_gpu()
    for n in ((150, 40, 33), (156, 52, 64), (40, 64, 150)):
        ctx = _ctx(W.random_problem(3, 1, n), form)
        for shape in (None, 0, 3, 4, 5):
            for k in range(3):
                if shape is not None:
                    ctx.es_set_tuning(k, shape)
                _, S, WT, grid, _ = ctx.es_get_tuning()[k]
                ns, lines = -(-n[k] // S), -(-n[1 if k == 0 else 0] // WT) * n[1 if k == 2 else 2]
                spread = n[k] % S != 0 and ns * lines > grid
                assert not spread or math.gcd(grid, ns) == 1, (n, shape, k, S, WT, grid)


# every tile the library has: stage tiles (both forms, FP64 only) and mesh tiles
STAGE_TILES = ((16, 12), (12, 16), (14, 14), (24, 8), (20, 10), (8, 8), (12, 8), (16, 8))
STAGE_TILES_FP64 = ((16, 14), (24, 15))
MESH_TILES = ((32, 8), (32, 16), (24, 16), (24, 12), (16, 8), (8, 8))


def _same(a, b):
    return all(bool((u == v).all()) for u, v in zip(a, b))


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("d,N,n", [(2, 1, (64, 64, 1)), (2, 2, (150, 75, 1)), (3, 1, (63, 17, 10))])
def test_tuning_round_trip(d, N, n, form):
    """The tiles that an autotuned context runs, read with es_get_tiles and set on a new context,
    are the tiles that one runs, with the same results; and the table's calls stay consistent: the
    shape, extent and grid of es_get_tuning, es_get_fusion and es_get_mesh_tiles, set on another
    context, are reported there again."""
    torch = need_gpu()
    pb, JU, J, x, xdot = case(d, N, n[:d], "mixed", es=True, seed=81 + N, jump=True)
    pb = pb.with_(mu=5, nf=3, sigma=(W.SIG_RHO1, W.SIG_P), alpha=(60.0, 25.0))
    G = [to_dev(t, torch) for t in (JU, J, x)]
    a, b, t = _ctx(pb, form), _ctx(pb, form), _ctx(pb, form)
    untuned = a.es_step(*[g.clone() for g in G])
    a.es_autotune(*G, None, reps=2)
    for launch in b.TILES:
        TX, TY, grid, ms = a.es_get_tiles(launch)
        runs = (launch != "flux_k3" or d == 3) and (launch != "stage" or d == 2) and (launch != "mesh" or (d == 2 and form == 1))
        assert (TX > 0 and ms > 0) == (runs and (launch != "stage" or a.es_get_fusion()[0] >= 0)), launch
        if TX or (launch == "stage" and d == 2):
            b.es_set_tiles(launch, TX, TY, grid)
        assert b.es_get_tiles(launch)[:3] == (TX, TY, grid), launch
    assert _same(a.es_step(*[g.clone() for g in G]), untuned) and _same(b.es_step(*[g.clone() for g in G]), untuned)
    for k, (sh, S, WT, grid, ms) in enumerate(a.es_get_tuning()):
        t.es_set_tuning(k, sh, grid)
        assert t.es_get_tuning()[k][:4] == (sh, S, WT, grid) and t.es_get_tiles("flux_k%d" % (k + 1))[:3] == (S, WT, grid) and ms > 0
        if a.es_get_tiles("flux_k%d" % (k + 1))[:2] != (S, WT):
            assert a.es_get_tiles("flux_k%d" % (k + 1))[3] < ms
    if d == 2:
        sh, TX, TY, grid, ms = a.es_get_fusion()
        t.es_set_fusion(sh, grid)
        assert t.es_get_fusion()[:4] == (sh, TX, TY, grid) == (sh,) + t.es_get_tiles("stage")[:3] and ms > 0
        if a.es_get_tiles("stage")[:2] != (TX, TY):
            assert a.es_get_tiles("stage")[3] < ms
    if d == 2 and form == 1:
        sh, TX, TY, thr, ms = a.es_get_mesh_tiles()
        t.es_set_mesh_tiles(sh)
        assert t.es_get_mesh_tiles()[:4] == (sh, TX, TY, thr) and t.es_get_tiles("mesh")[:2] == (TX, TY) and ms > 0


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("N", [1, 2])
@pytest.mark.parametrize("weno,es_", [(0, True), (1, True), (0, False)])
def test_every_stage_tile_bitwise(form, N, weno, es_):
    """Every stage tile, 24 x 15 with its 375 interfaces a direction among them, gives the residual
    of the per-direction launches bit for bit on ragged, sub-tile and several-wave grids."""
    torch = need_gpu()
    for n, bc, seed in (((70, 37), "mixed", 91), ((10, 11), "reflect", 92), ((349, 151), "mixed", 93), ((33, 300), "periodic", 94)):
        pb, JU, J, x, xdot = case(2, N, n, bc, es=es_, seed=seed + N, jump=True)
        ctx = _ctx(pb.with_(weno=weno), form)
        G = [to_dev(t, torch) for t in (JU, J, x, xdot)]
        ctx.es_set_tiles("stage", 0, 0)
        assert ctx.es_get_fusion()[0] == -1
        ref = ctx.es_rhs(*G)
        for tile in STAGE_TILES + (STAGE_TILES_FP64 if form == 0 else ()):
            for grid in (0, 152):
                ctx.es_set_tiles("stage", *tile, grid)
                assert ctx.es_get_tiles("stage")[:2] == tile and grid in (0, ctx.es_get_tiles("stage")[2])
                assert _same(ctx.es_rhs(*G), ref), (n, tile, grid)


@pytest.mark.parametrize("bc", ["periodic", "mixed", "reflect"])
@pytest.mark.parametrize("mu,nf", [(1, 0), (5, 3), (8, 4), (9, 3), (16, 4), (3, 6)])
def test_every_mesh_tile_bitwise(bc, mu, nf):
    """Every mesh tile gives the mesh velocity and Delta t / Delta tau of the 32 x 8 tiles bit for bit."""
    torch = need_gpu()
    for n, seed in (((70, 37), 95), ((10, 11), 96), ((200, 199), 97)):
        pb, JU, J, x, _ = case(2, 2, n, bc, es=True, seed=seed, jump=True)
        ctx = _ctx(pb.with_(mu=mu, nf=nf, sigma=(W.SIG_RHO1, W.SIG_P), alpha=(60.0, 25.0)), 1)
        G = [to_dev(t, torch) for t in (JU, J, x)]
        ref = None
        for tile in MESH_TILES:
            ctx.es_set_tiles("mesh", *tile)
            assert ctx.es_get_tiles("mesh")[:2] == tile
            out = ctx.mesh_redistribute(*G)
            ref = ref or out
            assert _same(out, ref), (n, tile)


@pytest.mark.parametrize("N", [1, 2])
def test_fp64_3d_extents_bitwise(N):
    """FP64 3D flux tiles of any extent, the longest segment (255 x 1) and the most lines (15 x 16)
    among them, give the residual of the table's shape bit for bit."""
    torch = need_gpu()
    for n, seed in (((260, 10, 11), 98), ((10, 33, 130), 99)):
        pb, JU, J, x, xdot = case(3, N, n, "mixed", es=True, seed=seed, jump=True)
        ctx = _ctx(pb, 0)
        G = [to_dev(t, torch) for t in (JU, J, x, xdot)]
        for k in range(3):
            ctx.es_set_tuning(k, 0)
        ref = ctx.es_rhs(*G)
        for tile in ((255, 1), (15, 16), (1, 16), (1, 1), (127, 2), (50, 5), (7, 13), (255, 1)):
            for k in range(3):
                ctx.es_set_tiles("flux_k%d" % (k + 1), *tile)
                assert ctx.es_get_tiles("flux_k%d" % (k + 1))[:2] == tile
            assert _same(ctx.es_rhs(*G), ref), (n, tile)


def test_tiles_refused():
    """Extents without a tile, launches that do not exist and forms without the launch are refused."""
    need_gpu()
    from paper_2202_07989_gb300 import es
    c2, f2 = _ctx(W.random_problem(2, 1, (20, 20)), 1), _ctx(W.random_problem(2, 1, (20, 20)), 0)
    c3, f3 = _ctx(W.random_problem(3, 1, (20, 20, 20)), 1), _ctx(W.random_problem(3, 1, (20, 20, 20)), 0)
    for ctx, launch, a, b in ((c2, "stage", 16, 14), (c2, "stage", 9, 9), (c2, "stage", 8, 0), (c3, "stage", 16, 12), (c2, "flux_k3", 62, 4),
                              (c2, "flux_k1", 61, 4), (f2, "flux_k1", 61, 4), (c3, "flux_k1", 61, 4), (f3, "flux_k1", 256, 1),
                              (f3, "flux_k2", 0, 4), (f3, "flux_k2", 4, 0), (f3, "flux_k2", 14, 17), (f3, "flux_k3", 16, 16),
                              (f3, "flux_k1", 2 ** 31 - 1, 2), (f2, "mesh", 32, 8), (c3, "mesh", 32, 8), (c2, "mesh", 9, 9)):
        with pytest.raises(es.EsError):
            ctx.es_set_tiles(launch, a, b)
    with pytest.raises(es.EsError):
        c2.es_set_tiles("stage", 8, 8, -1)
    assert c2.L.es_set_tiles(c2.h, 5, 8, 8, 0) == 1 and c2.L.es_set_tiles(None, 3, 8, 8, 0) == 1


@pytest.mark.parametrize("n,mu,nf", [((64, 64), 1, 0), ((64, 64), 8, 4), ((200, 100), 3, 0), ((400, 200), 8, 0), ((400, 200), 8, 4),
                                     ((1200, 480), 1, 4), ((1200, 480), 3, 3), ((1200, 480), 8, 0), ((1200, 480), 8, 4),
                                     ((1200, 480), 16, 4)])
def test_untuned_mesh_tiles_speed(n, mu, nf):
    """The mesh tiles that an untuned context picks for its grid, sweeps and filter passes take no
    more than 8% longer than the best tiles (a mesh step's time comes in steps of about 2 us, up to
    7% of the smallest ones here)."""
    torch = need_gpu()
    pb, U, x = W.shock_bubble_2d(*n)
    ctx = _ctx(pb.with_(mu=mu, nf=nf), 1)
    xg = to_dev(x, torch)
    J = ctx.es_init_mesh(xg)
    JU = to_dev(U, torch) * J
    xd, dd = torch.empty_like(xg), torch.empty(2, dtype=torch.float64, device="cuda")

    def us():
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            ctx.mesh_redistribute(JU, J, xg, xdot=xd, dt_dtau=dd)
            st.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st):
                ctx.mesh_redistribute(JU, J, xg, xdot=xd, dt_dtau=dd)
            best = float("inf")
            for _ in range(6):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                g.replay()
                e[0].record(st)
                for _ in range(10):
                    g.replay()
                e[1].record(st)
                e[1].synchronize()
                best = min(best, 100 * e[0].elapsed_time(e[1]))
        return best

    picked, t = ctx.es_get_tiles("mesh")[:2], us()
    all_ = {}
    for tile in MESH_TILES:
        ctx.es_set_tiles("mesh", *tile)
        all_[tile] = us()
    assert t <= 1.08 * min(all_.values()) + 3.0, (picked, t, all_)


@pytest.mark.parametrize("bc", ["periodic", "mixed", "reflect"])
@pytest.mark.parametrize("mu,nf", [(9, 3), (10, 0), (17, 4), (3, 6)])
def test_per_sweep_launches_bitwise(bc, mu, nf):
    """One launch per filter pass and sweep (1 x 1), offered beyond 8 sweeps or 4 filter passes, gives
    the mesh velocity and Delta t / Delta tau of the fused launches bit for bit; with fewer of both it
    is refused."""
    torch = need_gpu()
    from paper_2202_07989_gb300 import es
    for n, seed in (((70, 37), 101), ((10, 11), 102), ((200, 199), 103)):
        pb, JU, J, x, _ = case(2, 2, n, bc, es=True, seed=seed, jump=True)
        pb = pb.with_(sigma=(W.SIG_RHO1, W.SIG_P), alpha=(60.0, 25.0))
        ctx = _ctx(pb.with_(mu=mu, nf=nf), 1)
        G = [to_dev(t, torch) for t in (JU, J, x)]
        ctx.es_set_mesh_tiles(0)
        ref = ctx.mesh_redistribute(*G)
        ctx.es_set_tiles("mesh", 1, 1)
        assert ctx.es_get_tiles("mesh")[:2] == (1, 1)
        assert _same(ctx.mesh_redistribute(*G), ref), n
        with pytest.raises(es.EsError):
            _ctx(pb.with_(mu=8, nf=4), 1).es_set_tiles("mesh", 1, 1)


def test_large_grid_sweeps_run_per_sweep():
    """On grids where it is the faster by far (2000 x 400 with 16 sweeps: 380 us a mesh step against
    480), an untuned context runs one launch per sweep; on small ones (64 x 64) the fused launches."""
    need_gpu()
    for n, per_sweep in (((2000, 400), True), ((64, 64), False)):
        ctx = _ctx(W.shock_bubble_2d(*n)[0].with_(mu=16, nf=4), 1)
        assert (ctx.es_get_tiles("mesh")[:2] == (1, 1)) == per_sweep, n


@pytest.mark.parametrize("form", [0, 1])
def test_library_grid_shares_no_factor_with_segments(form):
    """Also where every segment is full, so that no CTA stays in one part of the lines: what an
    interface costs depends on the flow there."""
    need_gpu()
    for n in ((128, 128, 128), (112, 60, 56), (208, 40, 40)):
        ctx = _ctx(W.random_problem(3, 1, n), form)
        for shape in (None, 0, 4, 5):
            for k in range(3):
                if shape is not None:
                    ctx.es_set_tuning(k, shape)
                S, WT, grid, _ = ctx.es_get_tiles("flux_k%d" % (k + 1))
                ns, lines = -(-n[k] // S), -(-n[1 if k == 0 else 0] // WT) * n[1 if k == 2 else 2]
                assert ns * lines <= grid or math.gcd(grid, ns) == 1, (n, shape, k, S, WT, grid)


@pytest.mark.parametrize("chi", [(0.009, 0.09, 0.9), (0.5, 0.4, 0.3)])
@pytest.mark.parametrize("d,N", [(2, 1), (2, 2), (3, 1), (3, 2)])
def test_weights_that_do_not_sum_to_one(d, N, chi):
    """FP64 WENO-MR with linear weights that do not sum to one, which then weigh W itself instead of its
    differences: the oracle's residual in 2D, and the same bits in every tile.  (In 3D such weights
    make the dissipation depend on the shear directions, which rounding picks where the normal is x_3.)"""
    torch = need_gpu()
    n = (41, 29) if d == 2 else (40, 11, 10)
    pb, JU, J, x, xdot = case(d, N, n, "mixed", es=True, seed=121 + N, jump=True)
    pb = pb.with_(chi=chi)
    ctx = _ctx(pb, 0)
    G = [to_dev(t, torch) for t in (JU, J, x, xdot)]
    ref = ctx.es_rhs(*G)
    if d == 2:
        want, wantJ, mg = Oracle(pb).rhs_margins(JU, J, x, xdot)
        e, skipped = masked_fieldwise(ref[0].cpu().numpy(), want, mg, N, d)
        assert max(e + [rel_max_err(ref[1].cpu().numpy(), wantJ)]) <= TOL_FP64 and skipped <= 0.01 * pb.ncell, (e, skipped)
    if d == 2:
        tiles = [[("stage", t)] for t in ((0, 0),) + STAGE_TILES + STAGE_TILES_FP64]
    else:
        tiles = [[("flux_k%d" % (k + 1), t) for k in range(3)] for t in ((62, 4), (30, 8), (15, 16), (255, 1), (7, 13))]
    for t in tiles:
        for launch, extent in t:
            ctx.es_set_tiles(launch, *extent)
        assert _same(ctx.es_rhs(*G), ref), t
