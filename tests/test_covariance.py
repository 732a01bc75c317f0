"""The covariance form of the FP32 path, restated in numpy (CPU): beams from the feed
covariance (Eq. Vab) taken over upper-triangle tiles, and the e4m3 encoding of the voltages."""
import numpy as np
import pytest

import oracle
from helpers import make_case, oracle_beams

TILE = 256


def beams_from_covariance(x, w, nx, ny, mx, my):
    """P[A,B] of snapshots x [n][nx * ny] from R = sum x x^H, as the kernel takes it: tiles of
    the upper triangle (off the diagonal twice the real part; on it the imaginary part from
    Im(x_a) Re(x_b) alone, doubled), summed per (ix_a - ix_b mod mx, iy_a - iy_b)."""
    n = nx * ny
    re, im = x.real, x.imag
    V = np.zeros((mx, 2 * ny - 1), np.complex128)
    ix, iy = np.divmod(np.arange(n), ny)
    for i in range(0, n, TILE):
        for j in range(i, n, TILE):
            a, b = np.arange(i, min(i + TILE, n)), np.arange(j, min(j + TILE, n))
            S = re[:, a].T @ re[:, b] + im[:, a].T @ im[:, b]
            C = im[:, a].T @ re[:, b]
            R = S + 2j * C if i == j else 2 * (S + 1j * (C - re[:, a].T @ im[:, b]))
            W = w[a][:, None] * w[b].conj()[None, :] * R
            np.add.at(V, ((ix[a][:, None] - ix[b][None, :]) % mx,
                          iy[a][:, None] - iy[b][None, :] + ny - 1), W)
    A, B = np.arange(mx), np.arange(my)
    ew = np.exp(-2j * np.pi * np.outer(A, np.arange(mx)) / mx)
    ns = np.exp(-2j * np.pi * np.outer(np.arange(-(ny - 1), ny), B) / my)
    return (ew @ V @ ns).real


@pytest.mark.parametrize("shape", [(4, 100, 4, 256), (3, 37, 5, 73), (6, 20, 4, 8), (1, 300, 1, 512),
                                   (16, 18, 16, 16)], ids=lambda s: "x".join(map(str, s)))
def test_beams_from_covariance_match_oracle(shape):
    nx, ny, mx, my = shape
    v, w = make_case(nx, ny, mx, my, 2, 1, 12, 12, weights="random", seed=3)
    ref = oracle_beams(v, w, nx, ny, mx, my, 2, 1, 12)[0, 0]
    x = oracle.unpack(v).reshape(-1, nx * ny)
    got = beams_from_covariance(x, w.reshape(-1).astype(np.complex128), nx, ny, mx, my)
    assert np.abs(got - ref).max() <= 1e-10 * ref.mean()


def test_nibbles_as_e4m3():
    """Sign and magnitude |n| <= 8 as the bit pattern of an e4m3 byte are n 2^-9: the
    subnormals (exponent 0, m 2^-9) and the first binade ((8 + m) 2^-9) are one scale."""
    def e4m3(byte):
        s, e, m = byte >> 7, (byte >> 3) & 15, byte & 7
        val = m * 2.0 ** -9 if e == 0 else (8 + m) * 2.0 ** (e - 10)
        return -val if s else val

    for n in range(-8, 8):
        nib = n & 15
        byte = abs((nib ^ 8) - 8) | ((nib << 4) & 0x80)
        assert e4m3(byte) == n * 2.0 ** -9


@pytest.mark.parametrize("n_int,nwin,want", [
    (64, 4, 1), (64, (2 ** 31 - 65) // 64, 1), (64, 2 ** 31 // 64, 0), (1 << 16, 1 << 16, 0), (384, 2 ** 40, 0)])
def test_calls_past_32_bits_of_samples_load_directly(n_int, nwin, want):
    """A TMA coordinate has 32 bits: calls whose sample index does not fit take the direct loads (the
    same bits), not zeros past the wrap."""
    import ctypes

    import paper_1710_08591_gb300 as fb
    fb.build()
    f = fb.lib().fftbf_corr_staging
    f.restype = ctypes.c_int
    f.argtypes = [ctypes.c_int] * 7 + [ctypes.c_int64, ctypes.c_uint64]
    assert f(1, 32, 1, 64, 1, 1, n_int, nwin, 1 << 20) == want
    assert f(1, 32, 1, 64, 1, 1, n_int, nwin, (1 << 20) + 1) == 0          # off a 16-byte boundary
    assert f(1, 33, 1, 64, 1, 1, n_int, nwin, 1 << 20) == 0                # rows of 33 feeds
