"""Tensor-core scoring at the edges of its partition and row blocks: fewer tiles than
SMs, one tile, several segments per CTA, ragged last tiles, one and two blocks of window
rows with a short second block, and the deterministic mode's slots."""
import numpy as np
import pytest

import grkv_inputs as gi
import oracle as O
from paper_2605_31105_gb300 import binding as b
from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, b.GRKV_DETERMINISTIC], ids=["default", "deterministic"])
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("g,w,n,units", [
    (1, 1, 1, 1), (1, 1, 129, 3), (4, 32, 128, 2), (1, 129, 140, 2), (4, 64, 1000, 5),
    (2, 100, 300, 40), (7, 19, 260, 160), (4, 32, 700, 61), (8, 32, 400, 97),
])
def test_score_partition_edges(grkv_lib, g, w, n, units, causal, flags):
    """`units` copies of two units in turn; bounds as in the score stage test."""
    wl = gi.Workload(f"score_{g}_{w}_{n}", 2, g, n, 128, w, w, 7, 1e-2, "bf16", "lowrank", 700 + n)
    c, op = G.Case(wl), G.oracle_params(wl, causal=causal)
    pick = np.arange(units) % 2
    c.units = list(pick)
    c.dq, c.dk, c.dv = (t[pick].contiguous() for t in (c.dq, c.dk, c.dv))
    p = G.lib_params(wl, units, causal=causal)
    p.flags = flags
    scores, y, rs = G.run_score(c, p)
    ora = [O.compress_unit(c.q[i], c.k[i], c.v[i], op) for i in range(2)]
    for i in range(units):
        u, o = i % 2, ora[i % 2]
        tol = G.score_rel_tol(c.q[u], c.k[u], op)
        G.assert_scores(scores[i], o["scores"], tol)
        # probabilities enter Y as bf16 (relative 2^-9 each)
        lim = (tol + n * G.U + 2.0 ** -8) * (o["attn"] @ np.abs(c.v[u].astype(np.float64)))
        assert (np.abs(y[i] - o["y"]) <= lim).all()
        lb = G.logit_bound(c.q[u], c.k[u], op)
        assert np.abs(rs[i][:, 0] - o["row_max"]).max() <= lb + 1e-6 * np.abs(o["row_max"]).max()
        assert (np.abs(rs[i][:, 1] / o["row_sum"] - 1) <= tol + n * G.U).all()
