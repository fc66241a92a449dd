"""The fp32 solve's shared-memory steps do not depend on the order in which a block's threads
run between two barriers (the kernels' text run on the host, see host_block)."""
import numpy as np
import pytest

from tests import host_block as H


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return H.load(str(tmp_path_factory.mktemp("host_block")))


def _system(m, seed):
    x = np.random.default_rng(seed).random((m, 3 * m + 5))
    x /= x.sum(axis=1, keepdims=True)
    return x @ x.T + 1e-2 * np.eye(m)


def _factor_blocks(n):
    """L below the diagonal blocks of 32 rows, the inverses of L's diagonal blocks on them."""
    L = np.linalg.cholesky(n)
    out = np.tril(L)
    for o in range(0, len(n), 32):
        d = slice(o, min(o + 32, len(n)))
        out[d, d] = np.linalg.inv(L[d, d])
    return out


@pytest.mark.parametrize("m", [1, 32, 33, 77, 128])
def test_factor_in_any_thread_order(lib, m):
    n = _system(m, m)
    want = _factor_blocks(n)
    (up, s0), (down, s1) = H.chol(lib, n, False), H.chol(lib, n, True)
    assert s0 == s1 == 0
    np.testing.assert_array_equal(up, down)
    low = np.tril(np.ones((m, m), bool))
    # 2^-46 per operation, a few hundred of them in a chain, condition number about 1e2
    assert np.abs(up - want)[low].max() <= 2.0 ** -36 * np.abs(want).max()


@pytest.mark.parametrize("m", [1, 32, 33, 128])
def test_substitution_in_any_thread_order(lib, m):
    n, r = _system(m, m), np.random.default_rng(1).standard_normal((m, 128))
    f, _ = H.chol(lib, n, False)
    (up, s0), (down, s1) = H.subst(lib, f, r, False), H.subst(lib, f, r, True)
    assert s0 == s1 == 0
    np.testing.assert_array_equal(up, down)
    want = np.linalg.solve(n, r)
    assert np.abs(up - want).max() <= 2.0 ** -34 * np.abs(want).max()


@pytest.mark.parametrize("flip", [0, 1, 100, 255])
def test_a_block_agrees_on_leaving_a_unit_to_fp64(lib, flip):
    """Another block of the unit finds a value outside fp32's range while this one starts."""
    n, r = _system(40, 7), np.random.default_rng(2).standard_normal((40, 128))
    f, _ = H.chol(lib, n, False)
    z, state = H.subst(lib, f, r, False, flip)
    assert state == 1
    if flip == 0:
        assert np.abs(z - r).max() <= 2.0 ** -46 * np.abs(r).max()   # nothing was solved


@pytest.mark.parametrize("exp,state", [(-99, 0), (-101, 1), (98, 1)])
def test_a_column_outside_the_range_of_pairs(lib, exp, state):
    """One small (or, after N^-1, large) column gives the unit to fp64; a zero column does not."""
    n, r = _system(40, 7), np.random.default_rng(2).standard_normal((40, 128))
    r[:, 3] = 0.0
    r[:, 77] = np.ldexp(np.sign(r[:, 77]), exp)
    f, _ = H.chol(lib, n, False)
    assert H.subst(lib, f, r, False)[1] == state
