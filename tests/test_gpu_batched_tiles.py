"""GPU test of batched solves and log-likelihoods at tiles that are not a multiple of 128."""
import numpy as np
import pytest

import oracle
from paper_2410_09819_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2410_09819_gb300 import tile_chol as tc  # noqa: E402

from gpu_util import DEV, pack_padded, to_dev  # noqa: E402


@pytest.mark.parametrize("b", [64, 192])
@pytest.mark.parametrize("nrhs", [1, 5])
def test_batched_solve_and_loglik(b, nrhs):
    ns = [b, 3 * b - 20, 500]
    As = [oracle.matern(inputs.uniform_points(n, n, morton=True), 1.0, 0.08, 0.5, 1e-4) for n in ns]
    Bs = [inputs.gaussian(n, nrhs, seed=n) for n in ns]
    X = [torch.empty((nrhs, n), dtype=torch.float64, device=DEV) for n in ns]
    with tc.Handle(0) as H:
        rc, infos, _ = tc.tile_chol_factor_batched(H.h, ns, b, [to_dev(pack_padded(A, b)) for A in As])
        assert rc == 0 and not any(infos)
        tc.tile_chol_solve_batched(H.h, nrhs, [to_dev(B.T.copy()) for B in Bs], X, 0, 1e-13)
        lls = tc.tile_chol_loglik_batched(H.h, [to_dev(B[:, 0].copy()) for B in Bs])
    for A, B, x, ll, n in zip(As, Bs, X, lls, ns):
        L = np.linalg.cholesky(A)
        xr = np.linalg.solve(A, B)
        # two solves of backward error below 10 n u ||A||, and the condition of A
        assert np.abs(x.cpu().numpy().T - xr).max() <= 20 * n * 2.0**-53 * np.linalg.cond(A) * np.abs(xr).max()
        z = np.linalg.solve(L, B[:, 0])
        ref = -0.5 * n * np.log(2 * np.pi) - np.log(np.diag(L)).sum() - 0.5 * float(z @ z)
        assert abs(ll - ref) <= 1e-9 * abs(ref)
