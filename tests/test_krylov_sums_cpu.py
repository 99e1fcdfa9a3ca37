"""The threefold-FP32 sums of Scheme I's complex64 inner products (DotAcc<float> and grid_sums in
unsplit.cu), emulated step by step: products split exactly, two-sums per thread and across a
warp, FP64 over warps and blocks in the kernel's order.

Tolerance: FP64 rounding of the sums beyond the warps. The partial sums' magnitudes add up to
at most 1 for unit vectors (Cauchy-Schwarz) and each takes part in at most 8 (warps) + 19
(blocks of a lane) + 5 (lanes) additions, so the error is at most 32 * 2^-53; the FP32 part
adds about 2^-70 per product.
"""
import math

import numpy as np
import pytest

F = np.float32
TPB, MAX_BLOCKS = 256, 608


class Acc:
    def __init__(self, shape):
        self.s, self.c, self.g = (np.zeros(shape, F) for _ in range(3))

    @staticmethod
    def two_sum(x, p):
        t = x + p
        z = t - x
        return t, (x - (t - z)) + (p - z)

    def add_pair(self, hi, lo):
        self.s, r1 = self.two_sum(self.s, hi)
        lo, r2 = self.two_sum(lo, r1)
        self.c, r3 = self.two_sum(self.c, lo)
        self.g = self.g + (r2 + r3)

    def add(self, a, b):
        p = a * b
        exact = a.astype(np.float64) * b.astype(np.float64)
        self.add_pair(p, (exact - p.astype(np.float64)).astype(F))

    def warp_total(self):
        s, c, g = (x.reshape(-1, 32) for x in (self.s, self.c, self.g))
        for o in (16, 8, 4, 2, 1):
            half = Acc((s.shape[0], o))
            half.s, half.c, half.g = s[:, :o].copy(), c[:, :o].copy(), g[:, :o].copy()
            half.add_pair(s[:, o:2 * o], c[:, o:2 * o])
            half.g = half.g + g[:, o:2 * o]
            s, c, g = half.s, half.c, half.g
        return s[:, 0].astype(np.float64) + (c[:, 0].astype(np.float64) + g[:, 0])


def device_sum(a, b):
    """sum of a * b over [n][4] float32 arrays as the kernel adds it."""
    n = a.shape[0]
    blocks = min((n + 4 * TPB - 1) // (4 * TPB), MAX_BLOCKS)
    stride = blocks * TPB
    assert n % stride == 0 and n <= 8 * stride  # no flush inside a thread
    acc = Acc(stride)
    for k in range(0, n, stride):
        for q in range(4):
            acc.add(a[k:k + stride, q], b[k:k + stride, q])
    warps = acc.warp_total().reshape(blocks, TPB // 32)
    part = np.zeros(blocks)
    for t in range(TPB // 32):
        part = part + warps[:, t]
    lanes = np.zeros(32)
    for i in range(0, blocks, 32):
        v = part[i:i + 32]
        lanes[:v.size] = lanes[:v.size] + v
    for o in (16, 8, 4, 2, 1):
        lanes[:o] = lanes[:o] + lanes[o:2 * o]
    return lanes[0]


def vectors(n, kind, rng):
    if kind == "noise":
        v = rng.standard_normal((n, 4))
    else:
        x = np.linspace(-8.0, 8.0, n)
        ph = 40.0 * x + rng.uniform(0, 6.28)
        v = np.exp(-x ** 2)[:, None] * np.stack([np.cos(ph), np.sin(ph), 0.3 * np.cos(2 * ph),
                                                 -0.7 * np.sin(ph)], axis=1)
    return (v / np.linalg.norm(v)).astype(F)


@pytest.mark.parametrize("kind", ["noise", "packet"])
@pytest.mark.parametrize("n", [4096, 65536, 262144])
def test_products_of_unit_vectors_are_as_good_as_fp64(n, kind):
    rng = np.random.default_rng(n)
    a, b = vectors(n, kind, rng), vectors(n, kind, rng)
    for p, q in ((a, b), (a, a)):
        exact = math.fsum((p.astype(np.float64) * q.astype(np.float64)).ravel())
        err = abs(device_sum(p, q) - exact)
        print(f"n {n} {kind}: error {err:.2e} of {exact:.3e}")
        assert err <= 32 * 2.0 ** -53
