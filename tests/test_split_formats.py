"""What the 3xBF16 bars of the GPU tests tell apart: a matrix transform on even / odd halves with its
operands held as two or three BF16 planes, products and sums in 64 bits."""
import numpy as np
import pytest

# relative L2 error of a transform of a random field: three planes (24 bits; the products below 2^-16
# left out) stay below it, two planes (16 bits) do not; FP32 sums add some 3e-7 (test_gpu_tc_mft.py)
BF16_BAR = 1e-6


def planes(x, count):
    out, r = [], x.astype(np.float32)
    for _ in range(count):
        b = r.view(np.uint32).astype(np.uint64)
        h = (((b + 0x7fff + ((b >> 16) & 1)) >> 16) << 16).astype(np.uint32).view(np.float32).reshape(x.shape)
        out.append(h.astype(np.float64))
        r = (r - h).astype(np.float32)
    return out


def product(x, w, count):
    a, b = planes(x, count), planes(w, count)
    return sum(a[i] @ b[j] for i in range(count) for j in range(count - i))


@pytest.mark.parametrize("n,m", [(64, 40), (300, 64), (513, 129)])
def test_two_planes_miss_the_bar_and_three_meet_it(n, m):
    g = np.random.default_rng(n)
    k, u = np.arange(n // 2 + 1), np.arange(m // 2 + 1)
    w = np.cos(2 * np.pi * 0.37 / n * np.outer(k, u))
    x = g.standard_normal((n // 2 + 1, n // 2 + 1))
    ref = (x @ w).T @ w
    err = {c: np.linalg.norm(product(product(x, w, c).T, w, c) - ref) / np.linalg.norm(ref) for c in (2, 3)}
    print(f"n {n} m {m}: two planes {err[2]:.2e}, three {err[3]:.2e}")
    assert err[3] < 0.2 * BF16_BAR and err[2] > 2 * BF16_BAR
