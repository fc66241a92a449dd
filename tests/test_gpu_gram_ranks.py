"""The merge's Gram kernel at the edges of its split over a cluster: 1, 2, 4 and 8 ranks,
ranks without tiles or without non-fixed positions, ragged last tiles, one and two row
blocks, with and without the full-cache statistics, and units that start over because
their retained keys lie far below the full row maximum."""
import numpy as np
import pytest

import grkv_inputs as gi
import oracle as O
from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


def _case(g, w, n, B, units, far=False):
    """`units` copies of two units in turn; far: the retained set leaves out every row's best keys."""
    wl = gi.Workload(f"gram_{g}_{w}_{B}", 2, g, n, 128, w, B, 7, 1e-2, "bf16", "lowrank", 4000 + B)
    c = G.Case(wl)
    if far:
        # one prefix key far along every window query's direction, not retained
        c.q[:] = np.abs(c.q) + 1
        c.k[:, 5] = 8.0
        c.dq, c.dk = G.to_device(c.q, "bf16"), G.to_device(c.k, "bf16")
        c.q, c.k = G.to_host(c.dq), G.to_host(c.dk)
    op = G.oracle_params(wl)
    ora = [O.compress_unit(c.q[i], c.k[i], c.v[i], op) for i in range(2)]
    idx = np.stack([o["idx"] for o in ora])
    if far:
        rest = np.concatenate([np.arange(6, 6 + B - w), np.arange(n - w, n)])
        idx = np.stack([rest, rest]).astype(np.int32)
    s32 = np.stack([o["scores32"] for o in ora])
    y32 = np.stack([o["y"].astype(np.float32) for o in ora])
    rs = np.stack([np.stack([o["row_max"], o["row_sum"]], axis=1).astype(np.float32) for o in ora])
    ref = [O.merge_unit(c.q[i], c.k[i], c.v[i], s32[i], y32[i], idx[i], op) for i in range(2)]
    pick = np.arange(units) % 2
    c.units = list(pick)
    c.dq, c.dk, c.dv = (t[pick].contiguous() for t in (c.dq, c.dk, c.dv))
    return wl, c, s32[pick], y32[pick], idx[pick], rs[pick], ref


@pytest.mark.parametrize("stats", [True, False], ids=["one_phase", "two_phases"])
@pytest.mark.parametrize("g,w,n,B,units", [
    (4, 32, 600, 40, 2), (4, 32, 600, 129, 2), (2, 16, 900, 500, 3), (4, 32, 1500, 1100, 2),
    (4, 32, 1500, 1024, 16), (4, 32, 900, 520, 33), (4, 32, 700, 300, 65), (4, 64, 1500, 1100, 2),
    (3, 50, 900, 400, 20), (4, 64, 700, 300, 66), (1, 256, 700, 300, 2),
])
def test_gram_ranks(grkv_lib, g, w, n, B, units, stats):
    wl, c, s32, y32, idx, rs, ref = _case(g, w, n, B, units)
    _, vo = G.run_merge(c, G.lib_params(wl, units), s32, y32, idx, row_stats=rs if stats else None)
    for i in range(units):
        G.assert_values(vo[i], ref[i % 2]["v_out"], "bf16")


@pytest.mark.parametrize("B,units", [(100, 2), (1100, 2), (300, 130)])
def test_gram_starts_over(grkv_lib, B, units):
    """Every row's full maximum (key 5) is more than 2^64 above its retained maximum."""
    wl, c, s32, y32, idx, rs, ref = _case(4, 32, 1500, B, units, far=True)
    op = G.oracle_params(wl)
    for u in range(2):
        logits = c.q[u].reshape(-1, 128).astype(np.float64) @ c.k[u].T.astype(np.float64) / np.sqrt(128)
        kept = logits[:, idx[u]].max(axis=1)
        assert ((rs[u][:, 0] - kept) * np.log2(np.e) > 64).any(), op
    _, vo = G.run_merge(c, G.lib_params(wl, units), s32, y32, idx, row_stats=rs)
    for i in range(units):
        G.assert_values(vo[i], ref[i % 2]["v_out"], "bf16")
