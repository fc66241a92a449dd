"""Selection at the edges of its kernels: positions per thread (n - w around 2048, 4096,
8192, 16384), one CTA against a cluster (32768, 65536, 131072, 262144) and the workspace
kernel past that, pooling radii up to and past a cluster's halo, every budget edge, ties,
and scores over fp32's whole range.  Exact against the oracle."""
import numpy as np
import pytest

import grkv_inputs as gi
import oracle as O
from paper_2605_31105_gb300 import binding as b
from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


def _check(P, w, kk, pool, kind, s):
    wl = gi.Workload("select", s.shape[0], 1, P + w, 128, w, kk + w, pool, 1e-2, "bf16", "lowrank", 1)
    p = G.lib_params(wl, s.shape[0], pool_type=kind)
    op = G.oracle_params(wl, pool_type=kind)
    idx = G.run_select(p, s)
    for i in range(s.shape[0]):
        np.testing.assert_array_equal(idx[i], O.select(O.pool(s[i], op), op))


def _scores(rng, P, style):
    if style == "ties":
        return rng.integers(0, 40, size=(2, P)).astype(np.float32) / 64
    if style == "wide":   # attention mass of peaked rows: many decades, zeros among them
        x = np.exp(rng.normal(size=(2, P)) * 12).astype(np.float32)
        x[:, ::17] = 0
        return x
    x = rng.normal(size=(2, P)).astype(np.float32)   # a caller's own scores, signed
    x[0, P // 2] = np.inf
    x[1, 0] = -np.inf
    x[1, P // 3] = -3.4e38
    return x


@pytest.mark.parametrize("P", [1, 31, 2047, 2049, 4097, 8192, 16385, 32768, 32769, 65537, 131072,
                               131073, 262144, 262145])
@pytest.mark.parametrize("style", ["ties", "wide", "signed"])
def test_prefix_lengths(grkv_lib, P, style):
    rng = np.random.default_rng(P)
    s = _scores(rng, P, style)
    for kk in sorted({1, max(1, P // 10), max(1, P - 1)}):
        _check(P, 8, min(kk, P), 7, "max", s)


@pytest.mark.parametrize("P", [3000, 40000])
@pytest.mark.parametrize("pool", [1, 3, 13, 129, 131])
@pytest.mark.parametrize("kind", ["max", "avg"])
def test_pooling_widths(grkv_lib, P, pool, kind):
    s = _scores(np.random.default_rng(pool), P, "wide")
    _check(P, 32, P // 9, pool, kind, s)


@pytest.mark.parametrize("P", [5000, 50000])
@pytest.mark.parametrize("kk", ["none", "all"])
def test_budget_edges(grkv_lib, P, kk):
    s = _scores(np.random.default_rng(P), P, "ties")
    _check(P, 16, 0 if kk == "none" else P, 7, "max", s)


@pytest.mark.parametrize("P,stride", [(32768, 128), (30000, 128), (65536, 256), (131072, 512)])
@pytest.mark.parametrize("sampled", ["high", "low", "half"])
def test_misleading_sample(grkv_lib, P, stride, sampled):
    """The keys that place the candidates' bound (every `stride`-th position) lie above all
    others (too few candidates), below them (too many), or the cut falls among them."""
    rng = np.random.default_rng(P + len(sampled))
    s = (1 + rng.random((2, P))).astype(np.float32)
    if sampled == "high":
        s[:, ::stride] += 100
    elif sampled == "low":
        s[:, ::stride] *= 1e-6
    else:
        s[:, ::stride] += 0.95
    for kk in (1, P // stride, P // 20, P // 20 + 1):
        _check(P, 8, kk, 1, "max", s)
