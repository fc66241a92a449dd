"""The regression solve at the edges of its 8 x 8 tiles and 128-row blocks, for each
split of the right-hand side (few, some, many units), against the oracle's merge."""
import numpy as np
import pytest

import grkv_inputs as gi
import oracle as O
from paper_2605_31105_gb300 import binding as b
from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


def _prepare(g, w, units):
    """`units` copies of two units in turn: the sizes of the launch, two oracle runs."""
    wl = gi.Workload(f"solve_{g}_{w}", 2, g, 400, 128, w, max(200, w + 40), 7, 1e-2, "bf16",
                     "lowrank", 5000 + g * w)
    c, op = G.Case(wl), G.oracle_params(wl)
    ora = [O.compress_unit(c.q[i], c.k[i], c.v[i], op) for i in range(2)]
    s32 = np.stack([o["scores32"] for o in ora])
    y32 = np.stack([o["y"].astype(np.float32) for o in ora])
    idx = np.stack([o["idx"] for o in ora])
    ref = [O.merge_unit(c.q[i], c.k[i], c.v[i], s32[i], y32[i], idx[i], op) for i in range(2)]
    pick = np.arange(units) % 2
    c.units = list(pick)
    c.dq, c.dk, c.dv = (t[pick].contiguous() for t in (c.dq, c.dk, c.dv))
    return wl, c, s32[pick], y32[pick], idx[pick], ref


@pytest.mark.parametrize("flags", [0, b.GRKV_FORCE_SIMT], ids=["default", "portable"])
@pytest.mark.parametrize("units", [2, 39, 77])
@pytest.mark.parametrize("g,w", [(1, 1), (1, 8), (3, 3), (1, 127), (4, 32), (3, 43), (8, 17),
                                 (1, 255), (4, 64)])
def test_solve_edges(grkv_lib, g, w, units, flags):
    wl, c, s32, y32, idx, ref = _prepare(g, w, units)
    p = G.lib_params(wl, units)
    p.flags = flags
    _, vo = G.run_merge(c, p, s32, y32, idx)
    for i in range(units):
        G.assert_values(vo[i], ref[i % 2]["v_out"], "bf16")


@pytest.mark.parametrize("flags", [0, b.GRKV_FORCE_SIMT], ids=["default", "portable"])
def test_singular_two_block_system(grkv_lib, flags):
    """m = 256, lambda = 0 and every retained token fixed: the first pivot is 0."""
    wl, c, s32, y32, _, _ = _prepare(4, 64, 2)
    wl = wl.replace(budget=wl.window)
    idx = np.tile(np.arange(wl.n - wl.window, wl.n, dtype=np.int32), (2, 1))
    p = G.lib_params(wl, 2, lambda_v=0.0)
    p.flags = flags
    _, vo = G.run_merge(c, p, s32, y32, idx, expect_status=b.GRKV_ERR_NUMERIC)
    np.testing.assert_array_equal(vo, np.stack([c.v[i][idx[i]] for i in range(2)]))
