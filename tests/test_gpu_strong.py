"""Strong couplings (a threshold of zero, which the acceptance table cannot hold)
keep the one-row teams of 2D L = 16: the same shape at the critical coupling runs the
same path, so the two times are nearly alike (2.9 against 1.7 ms where they are
not).  Kernel times of the library's own launch events."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

import paper_2304_03311_gb300 as jz  # noqa: E402
from paper_2304_03311_gb300 import build as jzbuild  # noqa: E402


@pytest.mark.parametrize("beta", [2.8, 4.0])
def test_one_row_teams_at_strong_couplings(beta):
    jzbuild.build()
    ctx = jz.ising_replica_init(0, 0, None)
    n = 20000
    w = torch.empty(n, dtype=torch.int64, device="cuda")

    def best(b):
        p = jz.make_params(2, 16, 16, b, 5, 100, 1, n, 3, n_therm=100)
        t = []
        for _ in range(6):
            jz.jarzynski_run_ex(ctx, p, w)
            jz.ising_sync(ctx)
            t.append(jz.ising_last_launch_ms(ctx))
        return min(t[1:])

    try:
        assert best(beta) <= 1.25 * best(0.44)
    finally:
        jz.ising_replica_free(ctx)
