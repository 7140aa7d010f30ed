"""The bounds-checked debug build on the Swendsen-Wang kernel's grouped bond
phase: states in shared memory whose rows and replicas straddle words and whose
last word is partial, and states beyond shared memory in 2D and 3D (there a
cluster start before the Metropolis protocol as well).  A clean run leaves the
status word at zero and gives the oracle's bits.  The binding binds one library
per process, so the debug run happens in a child process."""
import json
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

from conftest import ROOT  # noqa: E402

CHILD = r'''
import json, sys
import numpy as np
import torch
sys.path.insert(0, sys.argv[1])
import oracle
from paper_2304_03311_gb300 import build as jzbuild
import paper_2304_03311_gb300 as jz
jzbuild.build(debug=True)
jz.use_debug_library()
jz.ising_bounds_status(clear=True)
ctx = jz.ising_replica_init(0, 0, None)
bad = []
# (d, L, L_t, beta, l, options)
jobs = [(2, 50, 34, 0.42, 20, {}), (2, 26, 54, 0.44, 25, dict(n_replica=3, whole=True)),
        (2, 6, 128, 0.5, 3, dict(direction=-1)), (3, 10, 16, 0.22, 4, dict(protocol=2)),
        (3, 14, 6, 0.25, 9, dict(n_replica=3, whole=True)),
        (2, 170, 170, 0.44, 60, {}), (3, 30, 30, 0.22, 9, dict(therm_update=1))]
for d, L, L_t, beta, l, opt in jobs:
    n_step = 2 * L if opt.get("protocol") == 2 else 2
    opt = dict(dict(update=0 if opt.get("therm_update") else 1), **opt)
    n = 2
    w = torch.empty(n, dtype=torch.int64, device="cuda")
    s = torch.empty(n * opt.get("n_replica", 2) * L_t * L ** (d - 1), dtype=torch.int8,
                    device="cuda")
    jz.jarzynski_run_ex(ctx, jz.make_params(d, L, L_t, beta, l, n_step, 1, n, 5, n_therm=2, **opt),
                        w, s)
    jz.ising_sync(ctx)
    W, S = oracle.run(d, L, L_t, beta, l, n_step, 1, n, 5, n_therm=2, want_spins=True, **opt)
    if not (np.array_equal(w.cpu().numpy(), W) and np.array_equal(s.cpu().numpy(), S.reshape(-1))):
        bad.append(str((d, L, L_t, opt)))
jz.ising_replica_free(ctx)
sites, index = jz.ising_bounds_status()
print(json.dumps({"lib": jz.lib_path(), "sites": sites, "index": index, "mismatch": bad}))
'''


def test_grouped_bond_phase_runs_clean_and_bit_exact():
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True,
                       timeout=1800)
    assert r.returncode == 0, r.stderr[-3000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["lib"].endswith("libisingjz_debug.so")
    assert out["mismatch"] == []
    assert out["sites"] == 0, out
