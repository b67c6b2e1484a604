"""Contexts: what creating one costs, the scratch it holds, and the launch configuration it
reports, takes and runs."""
import math
import time

import pytest

from paper_2202_07989_gb300 import workloads as W

from .helpers import case, need_gpu, to_dev

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
