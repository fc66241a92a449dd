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


def _key_step_fp32(c, i, o, op, V, y, iters):
    """The key step in plain fp32 (matrix products as numpy sums them)."""
    Q, K0 = c.q[i].reshape(op.m, 128), c.k[i][o["idx"]]
    s, lam, free = np.float32(O.effective_scale(op)), np.float32(op.lambda_k), ~o["fixed"]
    seen = np.isfinite(O.window_logits(c.q[i], K0, op, cols=o["idx"]))
    S = np.where(seen, (Q @ K0.T) * s, -np.inf).astype(np.float32)
    X = np.exp(S - S.max(axis=1, keepdims=True))
    X /= X.sum(axis=1, keepdims=True)

    def jt(W):
        dA = W @ V.T
        dK = s * ((X * (dA - (X * dA).sum(axis=1, keepdims=True))).T @ Q)
        dK[~free] = 0
        return dK

    def jvp(dK):
        dS = s * (Q @ dK.T)
        return (X * (dS - (X * dS).sum(axis=1, keepdims=True))) @ V

    r = y - X @ V
    p, alpha, rs = r.copy(), np.zeros_like(r), (r * r).sum()
    for _ in range(iters):
        Ap = jvp(jt(p)) + lam * p
        step = rs / (p * Ap).sum()
        alpha += step * p
        r -= step * Ap
        rs, last = (r * r).sum(), rs
        p = r + (rs / last) * p
    K = K0.copy()
    K[free] += jt(alpha)[free]
    return K


@pytest.mark.parametrize("g,w,n,B", [(2, 8, 400, 64), (4, 32, 1500, 512), (2, 33, 700, 128)])
def test_key_step_is_as_exact_as_fp32(grkv_lib, g, w, n, B):
    """One iteration on fp32 inputs: the update is no further from fp64 (on the same V*, as written)
    than the same steps in plain fp32 are, on the average of four units.  The residual Y - X V* is
    a small difference, so a few units in the last place of its products show."""
    wl = gi.Workload(f"key32_{g}_{w}_{B}", 4, g, n, 128, w, B, 7, 1e-2, "f32", "lowrank", 100)
    c, op = G.Case(wl), G.oracle_params(wl, lambda_k=0.1)
    ora = [O.compress_unit(c.q[i], c.k[i], c.v[i], op) for i in range(c.U)]
    s32, y32, idx = (np.stack([o[k].astype(t) for o in ora])
                     for k, t in (("scores32", np.float32), ("y", np.float32), ("idx", np.int32)))
    p = G.lib_params(wl, c.U)
    p.flags, p.lambda_k, p.cg_iters, p.cg_tol = b.GRKV_UPDATE_K, 0.1, 1, 0.0
    ko, vo = G.run_merge(c, p, s32, y32, idx)
    err, ref = [], []
    for i, o in enumerate(ora):
        K0 = c.k[i][o["idx"]].astype(np.float64)
        want, _ = O.key_step_dual(o["x"], c.q[i].reshape(op.m, 128).astype(np.float64), K0, vo[i],
                                  y32[i], ~o["fixed"], np.float64(np.float32(0.1)),
                                  O.effective_scale(op), 1)
        size = np.linalg.norm(want - K0)
        err.append(np.linalg.norm(ko[i] - want) / size)
        ref.append(np.linalg.norm(_key_step_fp32(c, i, o, op, vo[i], y32[i], 1) - want) / size)
    assert np.mean(err) <= np.mean(ref), f"{err} against {ref} in plain fp32"
