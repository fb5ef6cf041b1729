"""GPU tests of factorizations whose matrix or factor holds tiles that are exactly zero (banded, block
diagonal, arrow-shaped matrices), at scales far from 1: a zero tile has no scale of its own, so it
must not decide the unit of the emulated products or the planes they keep."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2410_09819_gb300 import tile_chol as tc  # noqa: E402

from gpu_util import pack_padded, to_dev, unpack_lower  # noqa: E402

U = 2.0 ** -53
B, NT = 128, 6


def matrix(kind, n):
    """A well-conditioned SPD matrix of scale 1 with zero tiles."""
    rng = np.random.default_rng(11)
    tile = np.arange(n) // B
    i, j = tile[:, None], tile[None, :]
    if kind == "arrow":                                # zero tiles of A that fill in
        V = 0.02 * rng.standard_normal((n, n))
        A = np.where((j == 0) & (i > 0), V, 0.0)
        A = A + A.T + 2.0 * np.eye(n)
        return A
    keep = (i - j <= 1) if kind == "banded" else (i // 3 == j // 3)
    L = np.tril(np.where(keep, 0.05 * rng.standard_normal((n, n)), 0.0), -1) + np.eye(n)
    return L @ L.T


def in_core(A, mode, pm=None):
    n = A.shape[0]
    with tc.Handle(0, fp64_mode=mode) as H:
        At = to_dev(pack_padded(A, B))
        assert tc.tile_chol_factor(H.h, n, B, At, pm) == 0
        L = torch.empty_like(At)
        tc.tile_chol_get_factor(H.h, L)
        return unpack_lower(L, n, B)


def batched(A, mode):
    n = A.shape[0]
    with tc.Handle(0, fp64_mode=mode) as H:
        dev = [to_dev(pack_padded(m, B)) for m in (A, A[:2 * B, :2 * B])]
        assert tc.tile_chol_factor_batched(H.h, [n, 2 * B], B, dev)[0] == 0
        L = torch.empty_like(dev[0])
        tc.tile_chol_get_factor_batched(H.h, 0, L)
        return unpack_lower(L, n, B)


def out_of_core(A, mode, pm=None):
    n = A.shape[0]
    host = torch.from_numpy(pack_padded(A, B)).pin_memory()
    slot = B * B * 8 + 14 * B * B + 16 + (0 if pm is None else 7 * B * B + 24)
    with tc.Handle(0, fp64_mode=mode, device_cap_bytes=14 * slot) as H:
        assert tc.tile_chol_factor_ooc(H.h, n, B, host, pm) == 0
        return unpack_lower(host, n, B)


PATHS = {"core1": lambda A: in_core(A, 1), "core2": lambda A: in_core(A, 2), "batch": lambda A: batched(A, 2),
         "ooc1": lambda A: out_of_core(A, 1), "ooc2": lambda A: out_of_core(A, 2)}


def berr_over_bound(A, L):
    """||A - L L^T|| against 2 (n + 1) u || |L| |L^T| || (Higham, Theorem 10.3; the factor 2 for the digit
    planes' truncation, 2^-54 of a product's scale an element of K)."""
    return np.linalg.norm(A - L @ L.T) / (2 * (A.shape[0] + 1) * U * np.linalg.norm(np.abs(L) @ np.abs(L.T)))


@pytest.mark.parametrize("path", sorted(PATHS))
@pytest.mark.parametrize("kind", ["banded", "blocks", "arrow"])
def test_fp64_factor_at_small_and_large_scales(kind, path):
    A = matrix(kind, NT * B - 30)
    r = {s: berr_over_bound(s * A, PATHS[path](s * A)) for s in (1.0, 1e-10, 1e-20, 1e20)}
    assert all(v <= 1.0 for v in r.values()), r


@pytest.mark.parametrize("path", ["core", "ooc"])
@pytest.mark.parametrize("kind", ["banded", "blocks", "arrow"])
def test_mixed_factor_at_small_and_large_scales(kind, path):
    # tiles of the first column in FP32, the others in FP64: the stored FP32 values add 2^-24 |L| |L^T| each
    A = matrix(kind, NT * B)
    pm = np.zeros((NT, NT), dtype=np.uint8)
    pm[1:, 0] = oracle.FP32
    f = in_core if path == "core" else out_of_core
    r = {}
    for s in (1.0, 1e-10, 1e-20, 1e20):
        L = f(s * A, 2, pm.reshape(-1))
        bound = 2.0 ** -23 * np.linalg.norm(np.abs(L) @ np.abs(L.T)) * 1.01
        r[s] = np.linalg.norm(s * A - L @ L.T) / bound
    assert all(v <= 1.0 for v in r.values()), r


@pytest.mark.parametrize("path", ["core", "batch", "ooc"])
@pytest.mark.parametrize("n", [NT * B - 1, 2 * B + 1])
def test_mixed_factor_of_a_ragged_order_at_small_scales(n, path):
    # the ones on the padded diagonal are not the scale of the last diagonal tile
    i = np.arange(n)
    A = np.exp(-0.05 * np.abs(i[:, None] - i)) + 0.01 * np.eye(n)
    nt = -(-n // B)
    pm = np.zeros((nt, nt), dtype=np.uint8)
    pm[1:, 0] = oracle.FP32
    pm = pm.reshape(-1)
    r = {}
    for s in (1.0, 1e-10, 1e-20):
        if path == "batch":
            with tc.Handle(0, fp64_mode=2) as H:
                dev = [to_dev(pack_padded(s * m, B)) for m in (A[:B, :B], A)]
                one = np.zeros(1, dtype=np.uint8)
                assert tc.tile_chol_factor_batched(H.h, [B, n], B, dev, [one, pm])[0] == 0
                Lt = torch.empty_like(dev[1])
                tc.tile_chol_get_factor_batched(H.h, 1, Lt)
                L = unpack_lower(Lt, n, B)
        else:
            L = (in_core if path == "core" else out_of_core)(s * A, 2, pm)
        r[s] = np.linalg.norm(s * A - L @ L.T) / (2.0 ** -23 * np.linalg.norm(np.abs(L) @ np.abs(L.T)) * 1.01)
    assert all(v <= 1.0 for v in r.values()), r
