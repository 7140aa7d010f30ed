"""The estimator's grid of CTAs against the NumPy oracle at the sizes where its
split changes: fewer values than jackknife blocks, one chunk per block, several
chunks, the most CTAs, one and 64 blocks, equal work values (every block ties
for the maximum), one dominant block, and beta = 0."""
import numpy as np
import pytest

import oracle.estimator as oest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

import paper_2304_03311_gb300 as jz  # noqa: E402
from paper_2304_03311_gb300 import build as jzbuild  # noqa: E402

BETA, N = 0.44, 500
CASES = [(n, b, kind) for n, b in ((1, 1), (2, 64), (5, 32), (33, 32), (64, 64), (65, 64),
                                   (5119, 32), (5121, 32), (10240, 1), (10241, 64), (90001, 33))
         for kind in ("normal", "equal", "dominant")] + [(4096, 32, "beta0")]


@pytest.mark.parametrize("n,bins,kind", CASES)
def test_grid_estimate_matches_numpy(n, bins, kind):
    jzbuild.build()
    rng = np.random.default_rng(n * 64 + bins)
    w = 2 * np.rint(rng.normal(2.0, 1.5, n) * N / BETA / 2).astype(np.int64)
    if kind == "equal":
        w[:] = 1234
    elif kind == "dominant":
        w[n // 2] -= 40 * N
    beta = 0.0 if kind == "beta0" else BETA
    ctx = jz.ising_replica_init(0, 0, None)
    got = [jz.estimator_reduce(ctx, torch.from_numpy(w).cuda(), n, beta, N, 1, bins)
           for _ in range(2)]
    jz.ising_replica_free(ctx)
    assert got[0] == got[1]   # the counter of finished CTAs is back at zero
    ds, err = oest.delta_s2_with_error(w, beta, N, 1, bins)
    assert abs(got[0][1] - ds) <= 1e-12 * abs(ds) + 1e-13
    assert got[0][0] == -got[0][1]
    if min(n, bins) < 2:   # one block has no jackknife error: reported as 0
        assert got[0][2] == 0.0
        return
    # a difference of nearly equal estimates: relative to them, not to itself
    assert abs(got[0][2] - err) <= 1e-10 * abs(err) + 1e-12 * max(abs(ds), 1.0)
