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
