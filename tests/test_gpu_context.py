"""Contexts: what creating one costs, the scratch it holds, and the launch configuration it
reports, takes and runs."""
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
