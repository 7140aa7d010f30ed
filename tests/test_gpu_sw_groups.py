"""GPU parity of the Swendsen-Wang kernel's grouped bond phase against the
oracle at the shapes where its word arithmetic can go wrong: rows shorter than a
word, rows and replicas that straddle words, a partial last word, uneven groups
of words per warp, the sizes on both sides of the switch from the plain form,
the cut's slice across a replica boundary, and states beyond shared memory at
both register variants.  W_int and final spins are whole numbers: exact."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

import paper_2304_03311_gb300 as jz  # noqa: E402
from paper_2304_03311_gb300 import build as jzbuild  # noqa: E402

# (d, L, L_t, beta, l, n_traj, options): 2D words per CTA warp = V / 256, 3D V / 512
CASES = {
    "2d_below_the_switch": (2, 20, 32, 0.44, 7, 5, {}),              # V = 1280: 5 words
    "2d_at_the_switch": (2, 22, 30, 0.44, 7, 5, {}),                 # V = 1320: 6 words
    "2d_two_columns": (2, 2, 400, 0.44, 1, 4, {}),
    "2d_short_rows_reverse": (2, 6, 128, 0.5, 3, 4, dict(direction=-1)),
    "2d_straddling_rows": (2, 50, 34, 0.42, 20, 4, {}),
    "2d_eight_replicas": (2, 10, 24, 0.44, 4, 4, dict(n_replica=8)),
    "2d_partial_last_word": (2, 26, 54, 0.44, 25, 4, dict(n_replica=3, whole=True)),
    "2d_two_rounds_of_groups": (2, 70, 70, 0.44, 33, 3, {}),         # 307 words, 8 warps
    "2d_L_t_2": (2, 1024, 2, 0.44, 500, 3, {}),
    "3d_below_the_switch": (3, 6, 34, 0.22, 3, 4, {}),               # V = 2448: 5 words
    "3d_at_the_switch": (3, 6, 36, 0.22, 3, 4, dict(direction=-1)),  # V = 2592: 6 words
    "3d_protocol_2": (3, 10, 16, 0.22, 4, 3, dict(protocol=2)),
    "3d_whole_three_replicas": (3, 14, 6, 0.25, 9, 3, dict(n_replica=3, whole=True)),
    "3d_strong": (3, 12, 12, 1.5, 11, 3, {}),
}


def _check(d, L, L_t, beta, l, n_traj, opt, n_step=None, n_therm=3, update=1):
    jzbuild.build()
    n_step = n_step or (2 * L if opt.get("protocol") == 2 else 4)
    ctx = jz.ising_replica_init(0, 0, None)
    p = jz.make_params(d, L, L_t, beta, l, n_step, 1, n_traj, 5, n_therm=n_therm, update=update,
                       **opt)
    V = opt.get("n_replica", 2) * L_t * L ** (d - 1)
    w = torch.empty(n_traj, dtype=torch.int64, device="cuda")
    s = torch.empty(n_traj, V, dtype=torch.int8, device="cuda")
    jz.jarzynski_run_ex(ctx, p, w, s)
    jz.ising_sync(ctx)
    jz.ising_replica_free(ctx)
    some = sorted({0, n_traj // 2, n_traj - 1}) if n_traj > 8 else range(n_traj)
    for i in some:
        o = dict(opt, traj0=i)
        Wo, So = oracle.run(d, L, L_t, beta, l, n_step, 1, 1, 5, n_therm=n_therm, update=update,
                            want_spins=True, **o)
        assert int(w[i]) == int(Wo[0])
        np.testing.assert_array_equal(s[i].cpu().numpy(), So.reshape(-1))


@pytest.mark.parametrize("name", CASES)
def test_grouped_bond_phase(name):
    _check(*CASES[name])


# 3D states beyond shared memory: 4 trajectories fit two CTAs per SM, 320 do not
@pytest.mark.parametrize("n_traj", [4, 320])
def test_hbm_register_variants(n_traj):
    _check(3, 32, 26, 0.2216, 9, n_traj, {}, n_step=1, n_therm=2)
