"""GPU test: in a batch that holds a mixed map, the updates of every matrix, also of one that is all FP64, take
their plane budgets from the scale of their own output tiles."""
import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2410_09819_gb300 import tile_chol as tc  # noqa: E402

from gpu_util import pack_padded, to_dev, unpack_lower  # noqa: E402

B, N = 128, 256


def _exp(x):
    """The smallest e with max |x| <= 2^e."""
    f, e = math.frexp(np.abs(x).max())
    return e - 1 if f == 0.5 else e


def _pairs(A, L):
    """Plane pairs of the update of tile (1, 1): planes 14 - floor((e_out - e_x - e_y - 8) / 4) within [1, 14]."""
    su = min(14, max(1, 14 - (_exp(A[B:, B:]) - 2 * _exp(L[B:, :B]) - 8) // 4))
    return su * (su + 1) // 2


def test_fp64_matrix_beside_a_mixed_one():
    rng = np.random.default_rng(4)
    A = 3.0 * np.eye(N)
    A[B:, :B] = 2.0 ** -20 * rng.standard_normal((B, B))
    A[:B, B:] = A[B:, :B].T
    mats = [A, 1e-12 * A, 1e12 * A]
    maps = [np.zeros(4, dtype=np.uint8) for _ in mats]
    maps[0][2] = oracle.FP32                           # tile (1, 0) of the first matrix
    with tc.Handle(0, fp64_mode=2) as H:
        dev = [to_dev(pack_padded(m, B)) for m in mats]
        st = tc.tc_stats()
        assert tc.tile_chol_factor_batched(H.h, [N] * 3, B, dev, maps, st)[0] == 0
        Ls = []
        for i in range(3):
            t = torch.empty_like(dev[i])
            tc.tile_chol_get_factor_batched(H.h, i, t)
            Ls.append(unpack_lower(t, N, B))
    # tile (1, 1) is two items of 128 x 64 with one source each
    pairs = [_pairs(m, L) for m, L in zip(mats, Ls)]
    assert max(pairs) < 105                            # the budgets are below the full count here
    assert st.tensor_flops[tc.TC_FP64] == sum(2 * 2.0 * 128 * 64 * B * p for p in pairs)
