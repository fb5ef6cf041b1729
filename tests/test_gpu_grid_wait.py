"""GPU test: a wait limit short enough for the tensor-core pipelines does not end the longer waits
inside the cooperative POTRF and substitution kernels."""
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


@pytest.mark.parametrize("n,b", [(2048, 256), (4096, 4096)])
def test_short_wait_limit_leaves_factor_and_solve_alone(n, b):
    A = oracle.matern(inputs.uniform_points(n, 9, morton=True), 1.0, 0.05, 0.5, 1e-4)
    B = to_dev(inputs.gaussian(n, 1, seed=3).T.copy())
    out = []
    for us in (0, 1):                                  # the default bound, and one microsecond
        with tc.Handle(0, fp64_mode=0, wait_limit_us=us) as H:
            assert tc.tile_chol_factor(H.h, n, b, to_dev(pack_padded(A, b))) == 0
            X = torch.empty((1, n), dtype=torch.float64, device=DEV)
            tc.tile_chol_solve(H.h, 1, B, n, X, n)
            out.append(X)
    assert torch.equal(out[0], out[1])
