"""Host-side restatement (no GPU) of the block fixed-point transforms' passes
(csrc/chanfs_fix.cuh, fix_x.cu, fix_y.cu): for every supported length the radix
plan multiplies up, every pass writes each padded element once inside its
buffer, and the passes with the mirrored-pair untangling give the transforms
of numpy.fft."""

import numpy as np
import pytest


def smooth(lo, hi):
    return sorted(n for n in (2**a * 3**b for a in range(13) for b in range(8)) if lo <= n <= hi)


def radices(n, pair):
    a = b = 0
    m = n
    while m % 2 == 0:
        m, a = m // 2, a + 1
    while m % 3 == 0:
        m, b = m // 3, b + 1
    tail = 2 if pair and b == 0 else 0
    a -= tail

    def cost(c):
        rest = a - c
        return 2 * (b + rest // 3 + (rest % 3 > 0)) + (rest % 3 == 1 and rest < 4)

    c = min(range(min(a, b) + 1), key=cost)
    a, b = a - c, b - c
    fours = a % 3 == 1 and a >= 4
    r = [8] * (a // 3 - fours)
    if fours:
        r += [4, 4]
    elif a % 3:
        r += [2 if a % 3 == 1 else 4]
    return r + [6] * c + [3] * b + ([4] if tail else [])


def pad(e):
    return e + (e >> 3)


def butterflies(src, R, L, sign):
    """One Stockham pass; checks that the padded places are in bounds and hit once."""
    n = src.size
    Q, out, seen = n // R, np.empty(n, complex), set()
    w = np.exp(sign * 2j * np.pi * np.outer(np.arange(R), np.arange(R)) / R)
    for j in range(Q):
        k = j % L
        v = src[j::Q] * np.exp(sign * 2j * np.pi * np.arange(R) * k / (L * R))
        o = (j - k) * R + k + np.arange(R) * L
        out[o] = w @ v
        seen.update(pad(int(e)) for e in o)
    assert len(seen) == n and max(seen) < n + (n >> 3) + (n % 8 > 0) and min(seen) == 0
    assert max(seen) == pad(n - 1) < n + (n >> 3) + 1
    return out


def fft(z, rad, sign):
    L = 1
    for R in rad:
        z = butterflies(z, R, L, sign)
        L *= R
    return z


def pairs(R, Q, i):
    """(k, uses the butterfly Q/2) of item i's entries, as pair_index / pair_second."""
    if i:
        return [(i + r * Q, False) for r in range(R)]
    return {6: [(3 * Q, False), (Q, False), (2 * Q, False), (Q // 2, True), (Q // 2 + Q, True), (Q // 2 + 2 * Q, True)],
            4: [(2 * Q, False), (Q, False), (Q // 2, True), (Q // 2 + Q, True)],
            3: [(Q + Q // 2, True), (Q, False), (Q // 2, True)],
            2: [(Q, False), (Q // 2, True)]}[R]


@pytest.mark.parametrize("n", smooth(9, 2048))
def test_pair_plans_cover_the_half_spectrum(n):
    rad = radices(n, True)
    assert int(np.prod(rad)) == n and 2 <= len(rad) <= 8 and rad[-1] <= 6
    R, Q = rad[-1], n // rad[-1]
    seen = [0]
    for i in range((Q + 1) // 2):
        for k, second in pairs(R, Q, i):
            if i == 0 and second and Q % 2:
                continue
            assert 0 < k < n
            seen += [k] if 2 * k == n else [k, n - k]
    assert sorted(seen) == list(range(n))


@pytest.mark.parametrize("n", smooth(9, 4096))
def test_column_plans_multiply_up(n):
    rad = radices(n, False)
    assert int(np.prod(rad)) == n and 2 <= len(rad) <= 8


@pytest.mark.parametrize("n", [9, 12, 16, 18, 24, 27, 32, 48, 54, 64, 81, 96, 108, 128, 162, 192, 243,
                               256, 384, 432, 486, 512, 768, 972, 1024, 1728, 2048])
def test_passes_give_the_transforms(n):
    rng = np.random.default_rng(n)
    z = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    for pair in (False, True):
        rad = radices(n, pair)
        assert np.allclose(fft(z, rad, -1), np.fft.fft(z), atol=1e-10 * n)
        assert np.allclose(fft(z, rad[::-1] if pair else rad, 1), np.fft.ifft(z) * n, atol=1e-10 * n)
    # the real transform of nx = 2n values, both ways, through the pairs
    x = rng.standard_normal(2 * n)
    Z = fft(x[0::2] + 1j * x[1::2], radices(n, True), -1)
    X = np.fft.rfft(x)
    W = np.exp(-1j * np.pi * np.arange(n) / n)
    for k in range(1, n):
        E, O = Z[k] + np.conj(Z[n - k]), Z[k] - np.conj(Z[n - k])
        assert abs((E - 1j * W[k] * O) / 2 - X[k]) < 1e-10 * n
        T = X[k] - np.conj(X[n - k])
        assert abs(X[k] + np.conj(X[n - k]) + 1j * np.conj(W[k]) * T - 2 * Z[k]) < 1e-10 * n
    assert abs(Z[0].real + Z[0].imag - X[0].real) + abs(Z[0].real - Z[0].imag - X[n].real) < 1e-10 * n
