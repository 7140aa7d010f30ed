"""GPU parity of how a team shares out its rows, against the oracle: rows whose
last word holds one to four sites (those half words on threads of their own) or
five to seven, lattices of half words only, replicas on slots of their own, and
row counts around the bulk loop's pass of four with slots that lack the last row.
W_int and final spins are whole numbers: every job must give the oracle's bits."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

import paper_2304_03311_gb300 as jz  # noqa: E402
from paper_2304_03311_gb300 import build as jzbuild  # noqa: E402

# (d, L, L_t, l, threads, options); threads = 0: the default shape
CASES = [
    (2, 2, 2, 1, 0, {}), (2, 8, 8, 3, 0, {}), (2, 4, 40, 2, 0, dict(n_replica=3)),
    (2, 18, 6, 9, 32, {}), (2, 40, 40, 12, 32, {}), (2, 34, 34, 5, 32, dict(n_replica=3)),
    (2, 46, 46, 20, 32, {}), (2, 20, 200, 7, 0, dict(direction=-1)),
    (2, 64, 64, 21, 32, dict(n_replica=4)), (2, 64, 64, 32, 32, dict(n_replica=3)),
    (3, 2, 6, 1, 0, {}), (3, 4, 4, 2, 0, dict(protocol=2)), (3, 8, 8, 3, 0, {}),
    (3, 18, 14, 7, 36 * 7, {}), (3, 18, 40, 9, 36 * 13, dict(n_replica=3)),
    (3, 20, 10, 11, 40 * 6, dict(protocol=2, direction=-1)), (3, 24, 18, 23, 48 * 5, {}),
    (3, 22, 12, 2, 44 * 11, dict(whole=True)),
    (3, 16, 2, 5, 32, {}), (3, 16, 4, 8, 32, dict(n_replica=3)), (3, 16, 14, 9, 32, {}),
    (3, 32, 4, 20, 64 * 2, {}), (3, 32, 10, 31, 64 * 2, dict(direction=-1)),
]


@pytest.fixture(scope="module")
def lib():
    jzbuild.build()


@pytest.mark.parametrize("case", CASES, ids=lambda c: "d%dL%dLt%dl%dthr%d" % c[:5])
def test_shared_out_rows_are_bit_exact(lib, case):
    d, L, L_t, l, threads, opt = case
    n_traj, n_step, n_therm, seed = 7, 2 * L if opt.get("protocol") == 2 else 4, 3, 1234
    beta = 0.44 if d == 2 else 0.22
    c = jz.ising_replica_init(0, 0, None)
    try:
        if threads:
            jz.ising_set_threads(c, d, L, L_t, threads)
        p = jz.make_params(d, L, L_t, beta, l, n_step, 1, n_traj, seed, n_therm=n_therm, **opt)
        V = opt.get("n_replica", 2) * L_t * L ** (d - 1)
        w = torch.empty(n_traj, dtype=torch.int64, device="cuda")
        s = torch.empty(n_traj, V, dtype=torch.int8, device="cuda")
        jz.jarzynski_run_ex(c, p, w, s)
        jz.ising_sync(c)
        Wo, So = oracle.run(d, L, L_t, beta, l, n_step, 1, n_traj, seed, n_therm=n_therm,
                            want_spins=True, **opt)
        np.testing.assert_array_equal(w.cpu().numpy(), Wo)
        np.testing.assert_array_equal(s.cpu().numpy(), So.reshape(n_traj, -1))
    finally:
        jz.ising_replica_free(c)


def test_half_words_in_a_persistent_plan(lib):
    c = jz.ising_replica_init(0, 0, None)
    shapes = [(2, 8, 8), (2, 40, 40), (2, 46, 46), (3, 8, 8), (3, 18, 18), (3, 20, 20)]
    jobs = [jz.make_params(d, L, L_t, 0.3, 3, 5, 1, 5, 99, n_therm=2)
            for d, L, L_t in shapes]
    ws = [torch.empty(5, dtype=torch.int64, device="cuda") for _ in jobs]
    try:
        plan = jz.jz_plan_create(c, jobs, ws)
        jz.jz_plan_launch(plan)
        jz.ising_sync(c)
        jz.jz_plan_free(plan)
        for i, (d, L, L_t) in enumerate(shapes):
            Wo, _ = oracle.run(d, L, L_t, 0.3, 3, 5, 1, 5, 99, n_therm=2, want_spins=True)
            np.testing.assert_array_equal(ws[i].cpu().numpy(), Wo)
    finally:
        jz.ising_replica_free(c)


# warp teams whose lattices take more than the CTA's share of shared memory, and
# few trajectories: one team per CTA; many: warp teams
@pytest.mark.parametrize("cta", [0, 256, 512])
@pytest.mark.parametrize("n_traj", [3, 80])
def test_plan_layouts(lib, cta, n_traj):
    c = jz.ising_replica_init(0, 0, None)
    shapes = [(2, 128, 128), (2, 96, 96), (2, 32, 32), (3, 12, 12)]
    jobs = [jz.make_params(d, L, L_t, 0.3, 3, 2, 1, n_traj, 99, n_therm=1)
            for d, L, L_t in shapes]
    ws = [torch.empty(n_traj, dtype=torch.int64, device="cuda") for _ in jobs]
    try:
        plan = jz.jz_plan_create(c, jobs, ws, None, cta)
        jz.jz_plan_launch(plan)
        jz.ising_sync(c)
        jz.jz_plan_free(plan)
        for w, (d, L, L_t) in zip(ws, shapes):
            Wo, _ = oracle.run(d, L, L_t, 0.3, 3, 2, 1, n_traj, 99, n_therm=1)
            np.testing.assert_array_equal(w.cpu().numpy(), Wo)
    finally:
        jz.ising_replica_free(c)
