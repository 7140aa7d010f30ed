"""Which launch shape the library chooses at the ends of the trajectory count's
range, where the shape decides the time by factors."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

import paper_2304_03311_gb300 as jz  # noqa: E402
from paper_2304_03311_gb300 import build as jzbuild  # noqa: E402


def _shape(d, L, L_t, n_replica, n_traj):
    jzbuild.build()
    ctx = jz.ising_replica_init(0, 0, None)
    try:
        return jz.ising_launch_shape(ctx, jz.make_params(d, L, L_t, 0.3, 1, 4, 1, n_traj, 1,
                                                         n_therm=2, n_replica=n_replica))
    finally:
        jz.ising_replica_free(ctx)


# four warp teams to a CTA by default: with one trajectory three of them are idle
# and must not count as work done
@pytest.mark.parametrize("L,L_t,n", [(80, 320, 2), (96, 96, 4), (128, 128, 3), (160, 160, 2)])
def test_a_lone_trajectory_gets_a_wide_team(L, L_t, n):
    sh = _shape(2, L, L_t, n, 1)
    assert sh["teams"] == 1 and sh["team_threads"] >= 256, sh


# one CTA per SM: a slice per slot, six or more warps, beats a third of them with
# three times the rows each
@pytest.mark.parametrize("L", [28, 32])
@pytest.mark.parametrize("n_traj", [1, 152])
def test_few_trajectories_get_a_team_of_every_slice(L, n_traj):
    sh = _shape(3, L, 6, 2, n_traj)
    assert sh["team_threads"] == -(-L // 16) * L * 6, sh
