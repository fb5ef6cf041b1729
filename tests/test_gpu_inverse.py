"""GPU test of the column-by-column triangular inverse of mixed maps (k_trinv_batched) at the tiles
the other tests do not reach: an odd number of 128 blocks, and the largest."""
import numpy as np
import pytest

import mxp_local
import oracle
from paper_2410_09819_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2410_09819_gb300 import tile_chol as tc  # noqa: E402

from gpu_util import pack_padded, to_dev, unpack_lower  # noqa: E402


@pytest.mark.parametrize("n,b", [(768, 384), (1920, 640), (4096, 2048)])
def test_fp32_panels_match_one_oracle_step(n, b):
    A = oracle.matern(inputs.uniform_points(n, 17, morton=True), 1.0, 0.05, 0.5, 1e-4)
    nt = n // b
    pm = np.full((nt, nt), oracle.FP32, dtype=np.uint8)
    np.fill_diagonal(pm, oracle.FP64)
    with tc.Handle(0, fp64_mode=2) as H:
        At = to_dev(pack_padded(A, b))
        assert tc.tile_chol_factor(H.h, n, b, At, pm.reshape(-1)) == 0
        L = torch.empty_like(At)
        tc.tile_chol_get_factor(H.h, L)
    fails, close, agree = mxp_local.check_factor(A, unpack_lower(L, n, b), b, pm, "digits", "inverse")
    assert not fails, fails[:8]
    assert close[oracle.FP32] <= 1.0, (close, agree)
