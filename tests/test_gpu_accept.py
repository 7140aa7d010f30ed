"""GPU parity of the acceptance forms and row streams against the oracle: jobs
whose couplings the pair table cannot hold (a threshold of zero) or whose
switched thresholds round up to 2^32 - 1, lattices that leave no shared memory
for the table, and slice steps and row counts around the bulk loop's pass of
four rows.  W_int and final spins are whole numbers: every job must give the
oracle's bits."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

import paper_2304_03311_gb300 as jz  # noqa: E402
from paper_2304_03311_gb300 import build as jzbuild  # noqa: E402

# (d, L, L_t, beta, l, n_step, n_therm, n_traj, options)
CASES = {
    "never_2d": (2, 64, 64, 4.0, 20, 3, 2, 3, {}),
    "never_2d_ragged_reverse": (2, 10, 12, 3.0, 4, 5, 3, 17, dict(direction=-1)),
    "never_3d": (3, 16, 8, 2.5, 5, 3, 2, 3, {}),
    "never_one_row_teams": (2, 16, 16, 4.0, 4, 6, 4, 40, {}),
    "last_threshold_above_zero": (2, 16, 32, 2.77, 4, 6, 4, 9, {}),   # 2^32 e^(-8 beta) = 1.02
    "weak": (2, 32, 32, 1e-10, 9, 4, 2, 9, {}),
    "weak_3d_whole": (3, 6, 6, 1e-10, 3, 4, 2, 9, dict(whole=True)),
    "zero": (2, 16, 16, 0.0, 4, 6, 4, 40, dict(n_replica=4)),
    "no_room_for_the_table": (2, 240, 240, 0.44, 100, 2, 1, 2, {}),
}


def _check(ctx, d, L, L_t, beta, l, n_step, n_therm, n_traj, opt, seed=77):
    p = jz.make_params(d, L, L_t, beta, l, n_step, 1, n_traj, seed, n_therm=n_therm, **opt)
    V = opt.get("n_replica", 2) * L_t * L ** (d - 1)
    w = torch.empty(n_traj, dtype=torch.int64, device="cuda")
    s = torch.empty(n_traj, V, dtype=torch.int8, device="cuda")
    jz.jarzynski_run_ex(ctx, p, w, s)
    jz.ising_sync(ctx)
    Wo, So = oracle.run(d, L, L_t, beta, l, n_step, 1, n_traj, seed, n_therm=n_therm,
                        want_spins=True, **opt)
    np.testing.assert_array_equal(w.cpu().numpy(), Wo)
    np.testing.assert_array_equal(s.cpu().numpy(), So.reshape(n_traj, -1))


@pytest.fixture(scope="module")
def ctx():
    jzbuild.build()
    c = jz.ising_replica_init(0, 0, None)
    yield c
    jz.ising_replica_free(c)


@pytest.mark.parametrize("name", CASES)
def test_acceptance_forms(ctx, name):
    _check(ctx, *CASES[name])


# CTA teams of 36 TS threads (3D L = 18): TS = 1, 2 without and 3, 4 with the
# rotated first rows; L_t / TS from 1 to 10 rows per thread
@pytest.mark.parametrize("ts,L_t", [(1, 2), (1, 8), (2, 2), (2, 4), (2, 14), (3, 4), (3, 14),
                                    (4, 4), (4, 10), (4, 40)])
def test_slice_steps_and_row_counts(ts, L_t):
    c = jz.ising_replica_init(0, 0, None)
    try:
        jz.ising_set_threads(c, 3, 18, L_t, 36 * ts)
        _check(c, 3, 18, L_t, 0.22, 7, 3, 2, 3, {})
    finally:
        jz.ising_replica_free(c)


def test_plan_with_a_never_flipping_job():
    """A persistent plan takes the counts as soon as one of its jobs needs them."""
    c = jz.ising_replica_init(0, 0, None)
    jobs = [(2, 32, 32, 4.0, 5), (2, 20, 20, 0.44, 5), (3, 8, 8, 0.22, 2)]
    outs = [torch.empty(9, dtype=torch.int64, device="cuda") for _ in jobs]
    plan = jz.jz_plan_create(c, [jz.make_params(d, L, Lt, b, l, 4, 1, 9, 3, n_therm=3)
                                 for d, L, Lt, b, l in jobs], outs, None, 256)
    jz.jz_plan_launch(plan)
    jz.ising_sync(c)
    for (d, L, Lt, b, l), w in zip(jobs, outs):
        Wo, _ = oracle.run(d, L, Lt, b, l, 4, 1, 9, 3, n_therm=3)
        np.testing.assert_array_equal(w.cpu().numpy(), Wo)
    jz.jz_plan_free(plan)
    jz.ising_replica_free(c)
