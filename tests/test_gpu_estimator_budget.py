"""estimator_reduce within the context's memory budget: the grid's 8 KB of scratch is
charged to it, gives way to the buffers that a call needs, and without it the estimate
comes from one CTA, bit for bit the sums of a plan's batched estimator."""
import numpy as np
import pytest

import oracle.estimator as oest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

import paper_2304_03311_gb300 as jz  # noqa: E402
from paper_2304_03311_gb300 import build as jzbuild  # noqa: E402

N, BETA, STEPS = 9000, 0.44, 8


@pytest.fixture(scope="module")
def batched():
    """Work values of a plan's job and its batched estimate (one CTA per job)."""
    jzbuild.build()
    ctx = jz.ising_replica_init(0, 0, None)
    w = torch.empty(N, dtype=torch.int64, device="cuda")
    est = torch.empty(1, 3, dtype=torch.float64, device="cuda")
    plan = jz.jz_plan_create(ctx, [jz.make_params(2, 8, 8, BETA, 3, STEPS, 1, N, 7, n_therm=10)],
                             [w], est, 256)
    jz.jz_plan_launch(plan)
    jz.ising_sync(ctx)
    jz.jz_plan_free(plan)
    jz.ising_replica_free(ctx)
    return w, est.cpu().numpy()[0]


def _estimate(ctx, w):
    return np.array(jz.estimator_reduce(ctx, w, N, BETA, STEPS, 1, 32))


def test_budget_below_the_scratch_takes_one_cta(batched):
    w, est = batched
    free = jz.ising_replica_init(0, 0, None)
    tight = jz.ising_replica_init(0, 4096, None)
    grid, one = _estimate(free, w), _estimate(tight, w)
    assert np.array_equal(_estimate(tight, w), one) and np.array_equal(_estimate(free, w), grid)
    jz.ising_replica_free(free)
    jz.ising_replica_free(tight)
    assert not np.array_equal(grid, est)   # the two orders of summation can be told apart here
    assert np.array_equal(one, est)
    ds, err = oest.delta_s2_with_error(w.cpu().numpy(), BETA, STEPS, 1, 32)
    for e in (grid, one):
        assert abs(e[1] - ds) <= 1e-12 * abs(ds) + 1e-13


def test_scratch_gives_way_to_a_calls_own_buffers(batched):
    w, est = batched
    # room for the scratch, but not for it and the host work values' copy together
    ctx = jz.ising_replica_init(0, 8 * N + 4096, None)
    assert not np.array_equal(_estimate(ctx, w), est)            # by the grid
    host = w.cpu().numpy()
    assert np.array_equal(_estimate(ctx, host), est)             # the copy needs its room
    assert np.array_equal(_estimate(ctx, w), est)
    jz.ising_replica_free(ctx)


def test_too_small_a_budget_is_still_refused(batched):
    w, _ = batched
    ctx = jz.ising_replica_init(0, 16, None)
    with pytest.raises(jz.IsingError):
        _estimate(ctx, w)
    jz.ising_replica_free(ctx)
