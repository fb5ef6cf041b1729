"""Failure detection of the cooperative kernels (POTRF of a tile, substitution sweeps), on the GPU without a
fault: with tc_config.wait_test = 2 each first waits for work that no CTA does, its bound (100 ms, the
least of these waits) runs out, all its CTAs leave, and the call reports TC_ERR_TIMEOUT naming the
kernel.  The same handle then works with the hook off."""
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

N, B = 700, 128


def _matrix():
    return oracle.matern(inputs.uniform_points(N, 9, morton=True), 1.0, 0.05, 0.5, 1e-4)


def _times_out(what, call, H):
    with pytest.raises(tc.TileCholError) as ei:
        call()
    assert ei.value.code == tc.TC_ERR_TIMEOUT, ei.value
    msg = tc.tc_last_error(H.h)
    assert "timed out" in msg and what in msg and "tensor-core" not in msg, msg


def _is_factor(A, L):
    bound = 2 * (N + 1) * 2.0 ** -53 * np.linalg.norm(np.abs(L) @ np.abs(L.T))
    assert np.linalg.norm(A - L @ L.T) <= bound


def test_potrf_times_out_and_recovers_in_core():
    A = _matrix()
    At = to_dev(pack_padded(A, B))
    with tc.Handle(0, fp64_mode=0, wait_limit_us=1000, wait_test=2) as H:
        _times_out("POTRF", lambda: tc.tile_chol_factor(H.h, N, B, At), H)
        with pytest.raises(tc.TileCholError):          # no factor to solve with
            tc.tile_chol_logdet(H.h)
        tc.tc_set_wait_limit(H.h, 0, 1)                # stops the tensor-core kernels only: none in this mode
        assert tc.tile_chol_factor(H.h, N, B, At) == 0
        L = torch.empty_like(At)
        tc.tile_chol_get_factor(H.h, L)
    _is_factor(A, unpack_lower(L, N, B))


def test_potrf_times_out_and_recovers_out_of_core():
    A = _matrix()
    with tc.Handle(0, fp64_mode=0, wait_limit_us=1000, wait_test=2, device_cap_bytes=14 * B * B * 8) as H:
        host = torch.from_numpy(pack_padded(A, B)).pin_memory()
        _times_out("POTRF", lambda: tc.tile_chol_factor_ooc(H.h, N, B, host), H)
        tc.tc_set_wait_limit(H.h, 0, 0)
        host = torch.from_numpy(pack_padded(A, B)).pin_memory()
        assert tc.tile_chol_factor_ooc(H.h, N, B, host) == 0
    _is_factor(A, unpack_lower(host, N, B))


@pytest.mark.parametrize("nrhs", [1, 5])
def test_sweeps_time_out_and_recover(nrhs):
    A = _matrix()
    b = inputs.gaussian(N, nrhs, seed=3).T.copy()
    Bd = to_dev(b)
    X = torch.empty_like(Bd)
    with tc.Handle(0, fp64_mode=0) as H:
        assert tc.tile_chol_factor(H.h, N, B, to_dev(pack_padded(A, B))) == 0
        tc.tc_set_wait_limit(H.h, 1000, 2)
        _times_out("sweep", lambda: tc.tile_chol_solve(H.h, nrhs, Bd, N, X, N), H)
        _times_out("sweep", lambda: tc.tile_chol_loglik(H.h, Bd[0]), H)
        tc.tc_set_wait_limit(H.h, 0, 0)
        st = tc.tc_stats()
        tc.tile_chol_solve(H.h, nrhs, Bd, N, X, N, 1, 0.0, st)
    x = X.cpu().numpy()
    assert np.linalg.norm(A @ x.T - b.T) <= 1e-12 * np.linalg.norm(A) * np.linalg.norm(x)
