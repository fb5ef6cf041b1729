"""GPU test of the sweeps' quotients: with a diagonal factor a substitution is a division an element, which is
rounded once, at ordinary values and where quotient or reciprocal come near the ends of the range."""
import numpy as np
import pytest

from paper_2410_09819_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2410_09819_gb300 import tile_chol as tc  # noqa: E402

from gpu_util import pack_padded, to_dev, unpack_lower  # noqa: E402


# exponents of the diagonal and of the right-hand sides: x = (b / l) / l stays finite and normal
@pytest.mark.parametrize("ea,eb", [(0, 0), (-900, -800), (900, 400), (-1000, -1000), (1000, 1000)])
@pytest.mark.parametrize("nrhs", [1, 4, 9])
def test_diagonal_solve_is_two_divisions(nrhs, ea, eb):
    n, b = 500, 64
    rng = np.random.default_rng(nrhs)
    A = np.diag((1.0 + 3.0 * rng.random(n)) * 2.0 ** ea)
    rhs = inputs.gaussian(n, nrhs, seed=5).T.copy() * 2.0 ** eb
    rhs[:, 7] = 0.0
    with tc.Handle(0, fp64_mode=0) as H:
        At = to_dev(pack_padded(A, b))
        assert tc.tile_chol_factor(H.h, n, b, At) == 0
        L = torch.empty_like(At)
        tc.tile_chol_get_factor(H.h, L)
        X = torch.empty((nrhs, n), dtype=torch.float64, device=At.device)
        tc.tile_chol_solve(H.h, nrhs, to_dev(rhs), n, X, n)
    d = np.diag(unpack_lower(L, n, b))
    assert np.array_equal(X.cpu().numpy(), rhs / d / d)
