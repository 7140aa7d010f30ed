"""What a persistent plan's CTA size and layouts are chosen by: the schedule of the
sweeps its kernel runs."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

import paper_2304_03311_gb300 as jz  # noqa: E402
from paper_2304_03311_gb300 import build as jzbuild  # noqa: E402


def _info(jobs):
    """(CTA size, grid, items) of a plan that is created and not run."""
    jzbuild.build()
    ctx = jz.ising_replica_init(0, 0, None)
    try:
        outs = [torch.empty(p.n_traj, dtype=torch.int64, device="cuda") for p in jobs]
        plan = jz.jz_plan_create(ctx, jobs, outs, None, 0)
        try:
            return tuple(jz.jz_plan_info(plan))
        finally:
            jz.jz_plan_free(plan)
    finally:
        jz.ising_replica_free(ctx)


def _job(i, d, L, L_t, n_traj, n_step, n_therm, therm_update=0, beta=None):
    return jz.make_params(d, L, L_t, beta or (0.44 if d == 2 else 0.22), 1, n_step, 1, n_traj, 5,
                          n_therm=n_therm, therm_update=therm_update, traj0=i << 20)


# (d, L, L_t, trajectories) of a job from a cluster start and of one from a Metropolis
# start: the cluster sweeps run in launches of their own, so their number does not count
@pytest.mark.parametrize("a,b", [
    ((3, 24, 24, 200), (2, 64, 64, 3000)), ((2, 96, 96, 300), (3, 8, 8, 4000)),
    ((3, 20, 20, 100), (2, 32, 32, 9000)), ((2, 64, 64, 2000), (3, 24, 24, 500)),
    ((2, 128, 128, 200), (3, 12, 12, 5000)), ((3, 16, 16, 1000), (2, 128, 128, 400)),
])
def test_cluster_starts_weigh_what_the_kernel_runs(a, b):
    few, many = (_info([_job(0, *a, 10, n, 1), _job(1, *b, 200, 200)]) for n in (1, 1000000))
    assert few == many


def test_strong_couplings_have_no_table():
    """2D L = 128, L_t = 892: one 114,176 byte lattice per CTA.  Two such CTAs share an
    SM's 233,472 bytes, with the acceptance table (2 KB each) they do not; jobs whose
    couplings the table cannot hold run without it, two CTAs of 256 threads per SM."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    job = (2, 128, 892, 4 * n_sm, 100, 100)
    assert _info([_job(0, *job, beta=4.0)])[:2] == (256, 2 * n_sm)
    assert _info([_job(0, *job)])[1] == n_sm


def test_one_long_trajectory_among_many_short_ones():
    """30,000 short items, which one team per CTA makes of 30,000 trajectories, do not
    hide the long one: its team of 512 threads is done first, whatever the others take."""
    assert _info([_job(0, 2, 128, 128, 1, 100000, 100), _job(1, 2, 20, 20, 30000, 100, 100)])[0] == 512
