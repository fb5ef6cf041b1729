"""GPU tests of the substitution sweeps (k_sweep): one to many right-hand sides, at the edges of
the column groups, from a single 64-row block to more blocks than the grid holds."""
import numpy as np
import pytest

import oracle
from paper_2410_09819_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2410_09819_gb300 import tile_chol as tc  # noqa: E402

from gpu_util import DEV, pack_padded, to_dev, unpack_lower  # noqa: E402

U = 2.0 ** -53


@pytest.mark.parametrize("n,b,nrhs", [(64, 64, 1), (100, 64, 3), (130, 64, 4), (700, 128, 1), (700, 128, 5),
                                      (1000, 192, 16), (1000, 128, 65), (900, 256, 260)])
def test_substitution_is_backward_stable(n, b, nrhs):
    A = oracle.matern(inputs.uniform_points(n, 40 + n, morton=True), 1.0, 0.08, 1.5, 1e-4)
    B = inputs.gaussian(n, nrhs, seed=n)
    ldx = n + 3                                        # a leading dimension of its own
    X = torch.full((nrhs, ldx), float("nan"), dtype=torch.float64, device=DEV)
    with tc.Handle(0) as H:
        At = to_dev(pack_padded(A, b))
        assert tc.tile_chol_factor(H.h, n, b, At) == 0
        L = torch.empty_like(At)
        tc.tile_chol_get_factor(H.h, L)
        tc.tile_chol_solve(H.h, nrhs, to_dev(B.T.copy()), n, X, ldx)
        ll = tc.tile_chol_loglik(H.h, to_dev(B[:, 0].copy()))
    x = X.cpu().numpy()[:, :n].T
    Lg = unpack_lower(L, n, b)
    # two triangular solves of backward error (n + 2) u |L| each (Higham, Theorem 8.5), one extra
    # rounding an element for the scaled triangles: |L L^T x - b| <= 4 (n + 4) u |L| |L^T| |x|
    bound = 4 * (n + 4) * U * (np.abs(Lg) @ (np.abs(Lg.T) @ np.abs(x))) + (n + 2) * U * np.abs(B)
    assert np.all(np.abs(Lg @ (Lg.T @ x) - B) <= bound)
    z = oracle.forward(Lg, B[:, :1])
    ref = -0.5 * n * np.log(2 * np.pi) - np.log(np.diag(Lg)).sum() - 0.5 * float((z * z).sum())
    assert abs(ll - ref) <= 1e-11 * abs(ref)


def test_sweep_with_more_blocks_than_resident_ctas():
    # 164 blocks of 64 rows for two columns, each on half of the 304 resident CTAs: a banded matrix
    # of condition number 3 with a known solution
    n, b = 10496, 128
    with tc.Handle(0, fp64_mode=2) as H:
        T = tc.tile_count(n, b)
        A = torch.zeros(T * b * b, dtype=torch.float64, device=DEV).view(T, b, b)
        i = torch.arange(n // b, device=DEV)
        r = torch.arange(b, device=DEV)
        A[i * (i + 1) // 2 + i] = torch.eye(b, dtype=torch.float64, device=DEV) * 4.0
        A[(i * (i + 1) // 2 + i)[:, None], r[1:], r[:-1]] = -1.0
        A[(i * (i + 1) // 2 + i)[:, None], r[:-1], r[1:]] = -1.0
        A[(i * (i + 1) // 2 + i - 1)[1:], b - 1, 0] = -1.0     # column-major: column b - 1, row 0
        assert tc.tile_chol_factor(H.h, n, b, A.view(-1)) == 0
        x0 = to_dev(inputs.gaussian(n, 2, seed=1).T.copy())
        rhs = 4.0 * x0
        rhs[:, 1:] -= x0[:, :-1]
        rhs[:, :-1] -= x0[:, 1:]
        X = torch.empty_like(rhs)
        tc.tile_chol_solve(H.h, 2, rhs, n, X, n)
    assert float((X - x0).abs().max()) <= 3 * 64 * U * float(x0.abs().max())
