"""The on-chip key step at the edges of its split: ranks without columns, 64 columns a
rank, each cluster size (few, some, many units), ragged shares, window rows short of 128,
both dtypes, and one retained token more than it takes.  Bounds as in test_key_step."""
import numpy as np
import pytest

import grkv_inputs as gi
import oracle as O
from paper_2605_31105_gb300 import binding as b
from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g,w,n,B,units,dtype", [
    (1, 1, 300, 17, 2, "bf16"), (2, 8, 400, 64, 2, "f32"), (4, 32, 1500, 511, 2, "bf16"),
    (4, 32, 1500, 512, 2, "f32"), (4, 32, 1500, 513, 2, "bf16"), (1, 127, 900, 300, 2, "bf16"),
    (4, 16, 900, 200, 39, "bf16"), (4, 16, 900, 130, 39, "f32"), (4, 16, 900, 100, 77, "bf16"),
    (2, 33, 700, 128, 77, "f32"), (4, 32, 1200, 257, 20, "bf16"),
])
@pytest.mark.parametrize("causal", [True, False])
def test_key_split_edges(grkv_lib, g, w, n, B, units, dtype, causal):
    wl = gi.Workload(f"key_{g}_{w}_{B}", 2, g, n, 128, w, B, 7, 1e-2, dtype, "lowrank", 9000 + B)
    c = G.Case(wl)
    op = G.oracle_params(wl, update_k=True, lambda_k=0.1, cg_iters=4000, cg_tol=1e-12, causal=causal)
    ora = [O.compress_unit(c.q[i], c.k[i], c.v[i], op) for i in range(2)]
    pick = np.arange(units) % 2
    c.units = list(pick)
    c.dq, c.dk, c.dv = (t[pick].contiguous() for t in (c.dq, c.dk, c.dv))
    args = [np.stack([o[k].astype(t) for o in ora])[pick]
            for k, t in (("scores32", np.float32), ("y", np.float32), ("idx", np.int32))]
    p = G.lib_params(wl, units, causal=causal)
    ko0, vo0 = G.run_merge(c, p, *args)
    p.flags, p.lambda_k, p.cg_iters, p.cg_tol = b.GRKV_UPDATE_K, 0.1, 4000, 1e-6
    ko, vo = G.run_merge(c, p, *args)
    np.testing.assert_array_equal(vo, vo0)
    rnd = 2.0 ** -8 if dtype == "bf16" else 2.0 ** -23
    for i in range(units):
        o = ora[i % 2]
        K0 = c.k[i % 2][o["idx"]].astype(np.float64)
        np.testing.assert_array_equal(ko[i][o["fixed"]], ko0[i][o["fixed"]])
        G.assert_values(ko[i], o["k_out"], dtype, what="k_out")
        err = np.linalg.norm(ko[i].astype(np.float64) - o["k_out"])
        lim = 2e-3 * np.linalg.norm(o["k_out"] - K0) + rnd * np.linalg.norm(o["k_out"])
        assert err <= lim, f"unit {i}: {err:.3e} > {lim:.3e}"
