"""GPU test of the one-kernel POTRF of a tile (k_potrf_tile) against the launches per 64-column step,
which a captured batch keeps: the same bits and the same failing column."""
import numpy as np
import pytest

import oracle
from paper_2410_09819_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2410_09819_gb300 import tile_chol as tc  # noqa: E402

from gpu_util import pack_padded, to_dev  # noqa: E402


def both(A, b, mode):
    n = A.shape[0]
    At = to_dev(pack_padded(A, b))
    out = []
    for batched in (False, True):
        with tc.Handle(0, fp64_mode=mode) as H:
            L = torch.empty_like(At)
            if batched:
                rc, infos, _ = tc.tile_chol_factor_batched(H.h, [n], b, [At])
                info = int(infos[0])
                if not info:
                    tc.tile_chol_get_factor_batched(H.h, 0, L)
            else:
                info = int(tc.tile_chol_factor(H.h, n, b, At))
                if not info:
                    tc.tile_chol_get_factor(H.h, L)
        out.append((info, L if not info else None))
    return out


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("n,b", [(128, 128), (500, 128), (400, 192), (700, 320), (1000, 512), (1100, 1024), (2048, 2048)])
def test_same_bits_as_the_launches_per_step(n, b, mode):
    if mode and b % 128:
        pytest.skip("digit planes need tiles of a multiple of 128")
    A = oracle.matern(inputs.uniform_points(n, 3 + n, morton=True), 1.0, 0.1, 0.5, 1e-4)
    (i0, L0), (i1, L1) = both(A, b, mode)
    assert i0 == 0 and i1 == 0 and torch.equal(L0, L1)


@pytest.mark.parametrize("n,b,col", [(256, 256, 1), (256, 256, 64), (1024, 512, 300), (1024, 1024, 961), (600, 128, 600)])
def test_reports_the_column_of_a_pivot_that_is_not_positive(n, b, col):
    A = oracle.matern(inputs.uniform_points(n, 5, morton=True), 1.0, 0.1, 0.5, 1e-4)
    A[col - 1, col - 1] = -1.0
    (i0, _), (i1, _) = both(A, b, 0)
    assert i0 == col and i1 == col
