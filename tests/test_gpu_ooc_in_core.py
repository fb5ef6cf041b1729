"""GPU test: out of core the updates and inverses of a mixed map run in another base than in core (fp64_mode 2), so
the two factors differ, but by no more than the map's accuracy level."""
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


@pytest.mark.parametrize("n,b,nu,rg,eps", [(2048, 256, 1.5, 0.03, 1e-9), (2048, 256, 1.5, 0.03, 1e-7),
                                           (2048, 512, 0.5, 0.05, 1e-8), (1500, 128, 0.5, 0.02, 1e-6)])
def test_mixed_factors_agree_to_the_accuracy_level(n, b, nu, rg, eps):
    A = oracle.matern(inputs.uniform_points(n, 31, morton=True), 1.0, rg, nu, 1e-4)
    nt = -(-n // b)
    pm = np.empty(nt * nt, dtype=np.uint8)
    with tc.Handle(0, fp64_mode=2) as H:
        At = to_dev(pack_padded(A, b))
        tc.tile_chol_precision_map(H.h, n, b, At, eps, 1, 4, pm)
        assert tc.tile_chol_factor(H.h, n, b, At, pm) == 0
        L = torch.empty_like(At)
        tc.tile_chol_get_factor(H.h, L)
        Lc = unpack_lower(L, n, b)
    host = torch.from_numpy(pack_padded(A, b)).pin_memory()
    slots = max(8, nt * (nt + 1) // 3)
    with tc.Handle(0, fp64_mode=2, device_cap_bytes=slots * (29 * b * b + 40)) as H:
        assert tc.tile_chol_factor_ooc(H.h, n, b, host, pm) == 0
    Lo = unpack_lower(host, n, b)
    assert np.any(pm.reshape(nt, nt)[np.tril_indices(nt, -1)] != oracle.FP64)
    normA = np.linalg.norm(A)
    assert np.linalg.norm(Lo @ Lo.T - Lc @ Lc.T) <= eps * normA
    # and neither is further from A than its accuracy level
    assert max(np.linalg.norm(A - Lo @ Lo.T), np.linalg.norm(A - Lc @ Lc.T)) <= eps * normA
