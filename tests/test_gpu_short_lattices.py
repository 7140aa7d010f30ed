"""Short lattices with ragged rows (L_t = 2, teams of two slices) take about as long
as those with whole rows of as many words: an edge row's geometry is computed once
per trajectory in both.  Two edge rows per thread and half-sweep, so the 25 % that
recomputing them cost shows in full; the ragged rows' two more instructions per word
are within the 12 % allowed.  Kernel times of the library's own launch events."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

import paper_2304_03311_gb300 as jz  # noqa: E402
from paper_2304_03311_gb300 import build as jzbuild  # noqa: E402


def test_ragged_rows_of_short_lattices():
    jzbuild.build()
    ctx = jz.ising_replica_init(0, 0, None)
    w = torch.empty(100, dtype=torch.int64, device="cuda")

    def best(L):
        p = jz.make_params(2, L, 2, 0.44, 60, 100, 1, 100, 3, n_therm=100)
        t = []
        for _ in range(6):
            jz.jarzynski_run_ex(ctx, p, w)
            jz.ising_sync(ctx)
            t.append(jz.ising_last_launch_ms(ctx))
        return min(t[1:])

    try:
        ragged, whole = best(200), best(208)   # 13 words per row
        assert ragged <= 1.12 * whole, (ragged, whole)
    finally:
        jz.ising_replica_free(ctx)
