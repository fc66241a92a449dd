"""The CUDA-core scoring and value step at the edges of their tiles: 16 / 32 / 64 /
128 window rows, 64 keys per scoring tile, 32 retained slots, 8 x 32 regression
tiles, 32-column solve blocks, the fp64 solve of m > 128 and of ill-conditioned
units.  Same bounds as the stage tests of test_gpu_parity.py."""
import numpy as np
import pytest

import grkv_inputs as gi
import oracle as O
from paper_2605_31105_gb300 import binding as b
from tests import gpu_cases as G

pytestmark = pytest.mark.gpu

SHAPES = [  # g, w, n, B
    (1, 1, 64, 2), (1, 31, 65, 32), (1, 32, 127, 64), (1, 33, 128, 65), (2, 32, 129, 96),
    (5, 13, 1000, 97), (1, 127, 700, 160), (4, 32, 1025, 255), (3, 43, 500, 129),
    (4, 64, 900, 300),
]


def _case(g, w, n, B, dtype):
    return gi.Workload(f"tiles_{g}_{w}_{n}_{B}", 2, g, n, 128, w, B, 7, 1e-2, dtype, "lowrank",
                       1000 + n)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("g,w,n,B", SHAPES)
def test_tile_edges(grkv_lib, g, w, n, B, dtype):
    wl = _case(g, w, n, B, dtype)
    c, op = G.Case(wl), G.oracle_params(wl)
    p = G.lib_params(wl, c.U)
    p.flags = b.GRKV_FORCE_SIMT
    scores, y, rs = G.run_score(c, p)
    ora = [O.compress_unit(c.q[i], c.k[i], c.v[i], op) for i in range(c.U)]
    for i, o in enumerate(ora):
        tol = G.score_rel_tol(c.q[i], c.k[i], op)
        G.assert_scores(scores[i], o["scores"], tol)
        lim = (tol + n * G.U) * (o["attn"] @ np.abs(c.v[i].astype(np.float64)))
        assert (np.abs(y[i] - o["y"]) <= lim).all()
        # the row maximum is one logit, the row sum a sum of n exponentials
        lb = G.logit_bound(c.q[i], c.k[i], op)
        assert np.abs(rs[i][:, 0] - o["row_max"]).max() <= lb + 1e-6 * np.abs(o["row_max"]).max()
        assert (np.abs(rs[i][:, 1] / o["row_sum"] - 1) <= tol + n * G.U).all()
    s32 = np.stack([o["scores32"] for o in ora])
    y32 = np.stack([o["y"].astype(np.float32) for o in ora])
    idx = np.stack([o["idx"] for o in ora])
    ko, vo = G.run_merge(c, p, s32, y32, idx)
    for i in range(c.U):
        ref = O.merge_unit(c.q[i], c.k[i], c.v[i], s32[i], y32[i], idx[i], op)
        np.testing.assert_array_equal(ko[i], c.k[i][idx[i]])
        np.testing.assert_array_equal(vo[i][ref["fixed"]], c.v[i][idx[i]][ref["fixed"]])
        G.assert_values(vo[i], ref["v_out"], dtype)


def _merge_inputs(c, op):
    ora = [O.compress_unit(c.q[i], c.k[i], c.v[i], op) for i in range(c.U)]
    return (np.stack([o["scores32"] for o in ora]),
            np.stack([o["y"].astype(np.float32) for o in ora]), np.stack([o["idx"] for o in ora]))


@pytest.mark.parametrize("w,n,B", [(33, 600, 90), (140, 900, 260)], ids=["m33", "m140"])
def test_ill_conditioned_unit_is_solved_in_fp64(grkv_lib, w, n, B):
    """Two equal window rows and lambda = 1e-9: the second row's Cholesky pivot is about
    2 lambda, far below 2^-20 of its diagonal, so the unit leaves the pair arithmetic.  The equal rows
    have equal residuals, so the merged values stay well determined."""
    wl = _case(1, w, n, B, "f32")
    c = G.Case(wl)
    c.q[0, 0, 7] = c.q[0, 0, 3]
    c.dq = G.to_device(c.q, wl.dtype)
    # without the causal rule the two rows see the same keys
    op = G.oracle_params(wl, lambda_v=1e-9, causal=False)
    p = G.lib_params(wl, c.U, lambda_v=1e-9, causal=False)
    s32, y32, idx = _merge_inputs(c, op)
    y32[0, 7] = y32[0, 3]
    _, vo = G.run_merge(c, p, s32, y32, idx)
    for i in range(c.U):
        ref = O.merge_unit(c.q[i], c.k[i], c.v[i], s32[i], y32[i], idx[i], op)
        G.assert_values(vo[i], ref["v_out"], "f32")


@pytest.mark.parametrize("w,n,B", [(40, 700, 150), (140, 900, 260)], ids=["m40", "m140"])
def test_near_singular_unit_has_fp64_sums(grkv_lib, w, n, B):
    """Half of the window rows differ from the other half by one rounding of one element, and
    lambda = 2^-51: the second half's pivots are below the rounding of sums in pairs of floats (which
    made one non-positive) and above that of fp64 sums."""
    wl = _case(1, w, n, B, "f32")
    c, h = G.Case(wl), w // 2
    c.q[:, 0, h:] = c.q[:, 0, :h]
    c.q[:, 0, h:, 5] = np.nextafter(c.q[:, 0, :h, 5], np.float32(9))
    c.dq = G.to_device(c.q, wl.dtype)
    p = G.lib_params(wl, c.U, lambda_v=2.0 ** -51, causal=False)
    s32, y32, idx = _merge_inputs(c, G.oracle_params(wl, causal=False))
    y32[:, h:] = y32[:, :h]
    _, vo = G.run_merge(c, p, s32, y32, idx)   # the status is GRKV_OK
    assert np.isfinite(vo).all()


@pytest.mark.parametrize("w,n,B", [(40, 700, 150), (140, 900, 260)], ids=["m40", "m140"])
@pytest.mark.parametrize("exp", [-134, 125])
def test_values_at_the_ends_of_fp32(grkv_lib, w, n, B, exp):
    """Values whose products' rounding errors are below fp32's range (subnormal values), and
    values whose Z = N^-1 R is above it: both ends were within an fp64 regression's range."""
    wl = _case(1, w, n, B, "f32")
    c = G.Case(wl)
    c.v = np.ldexp(c.v / np.abs(c.v).max(), exp).astype(np.float32)
    c.dv = G.to_device(c.v, wl.dtype)
    op = G.oracle_params(wl)
    s32, y32, idx = _merge_inputs(c, op)
    _, vo = G.run_merge(c, G.lib_params(wl, c.U), s32, y32, idx)
    for i in range(c.U):
        ref = O.merge_unit(c.q[i], c.k[i], c.v[i], s32[i], y32[i], idx[i], op)["v_out"]
        # the last rounding (half a unit, 2^-150 or 2^-24 relative), and X's fp32 error, a few
        # 1e-6, times |X_G^T N^-1| <= 1 / (2 sqrt(lambda)) = 5 times |R|'s scale
        lim = 2.0 ** -149 + 2.0 ** -23 * np.abs(ref) + 2e-5 * np.abs(c.v[i]).max()
        err = np.abs(vo[i].astype(np.float64) - ref)
        assert (err <= lim).all(), f"{err.max():.3e} against {lim.max():.3e}"
