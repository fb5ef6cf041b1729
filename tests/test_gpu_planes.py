"""GPU tests of the FP16 digit-plane products (k_zgemm): exact integer cases with three-digit
entries (every group sum has to be exact), and the triangular products of the refined TRSM at the
smallest and larger tiles."""
import numpy as np
import pytest

import oracle
from paper_2410_09819_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2410_09819_gb300 import tile_chol as tc  # noqa: E402

from gpu_util import pack_padded, to_dev, unpack_lower  # noqa: E402


def factor(A, b, mode):
    with tc.Handle(0, fp64_mode=mode) as H:
        At = to_dev(pack_padded(A, b))
        assert tc.tile_chol_factor(H.h, A.shape[0], b, At) == 0
        L = torch.empty_like(At)
        tc.tile_chol_get_factor(H.h, L)
    return unpack_lower(L, A.shape[0], b)


@pytest.mark.parametrize("n,b", [(256, 128), (500, 128), (1024, 256), (1536, 512)])
def test_wide_integer_factor_bit_exact(n, b):
    # entries of 20 bits below a diagonal of 2^20: every intermediate of the factorization is an
    # integer below 2^53, and a product's 128-element group sums reach 3 x 2^21 digits squared
    rng = np.random.default_rng(n + b)
    L = np.tril(rng.integers(-2**20 + 1, 2**20, (n, n)).astype(np.float64), -1) + 2.0**20 * np.eye(n)
    assert np.array_equal(factor(L @ L.T, b, 1), L)


@pytest.mark.parametrize("n,b", [(384, 128), (1000, 256), (1536, 512), (2048, 1024)])
def test_triangular_products_keep_the_backward_error(n, b):
    A = oracle.matern(inputs.uniform_points(n, 23, morton=True), 1.0, 0.05, 1.5, 1e-6)
    be = [np.linalg.norm(A - Lg @ Lg.T) / np.linalg.norm(A) for Lg in (factor(A, b, 1), factor(A, b, 2))]
    assert be[1] <= 1e-14 and be[1] <= 4 * be[0] + 1e-15, be
