"""The build's Gram matrices by residue products, entry by entry.

Each panel of K' <= 16,384 entries is exact for operands rounded to integers of 56 bits or more below
max sqrt(K') of their row: an entry of X moves by at most 2^-57 max sqrt(K'), so a product sum by
2^-57 sqrt(K') (max_i sum |x_j| + max_j sum |x_i|).  Its reconstruction in fixed point adds at most 1.5 units of
2^55, that is 1.5 2^-57 K' max_i max_j, and there is one FP64 rounding per panel and of each addition."""
import os

import numpy as np
import pytest
import torch

from paper_2212_12737_gb300 import build, gdml

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(build.LIB):
        build.build()
    gdml.load()


def exact_products(X):
    """X X^T with products and sums of 64-bit mantissas and more: X is cut into four parts of 18 bits below its
    row's maximum, whose products are exact in FP64, as are sums of 2^15 of them; the parts' products are added
    in double-double."""
    k, K = X.shape
    e = np.exp2(np.ceil(np.log2(np.abs(X).max(axis=1, keepdims=True))) + 1)
    parts, r = [], X / e
    for i in range(4):
        p = np.rint(r * 2.0 ** 18) / 2.0 ** 18
        parts.append(p)
        r = (r - p) * 2.0 ** 18
    hi = np.zeros((k, k))
    lo = np.zeros((k, k))
    for i in range(4):
        for j in range(4):
            for k0 in range(0, K, 1 << 15):
                t = (parts[i][:, k0:k0 + (1 << 15)] @ parts[j][:, k0:k0 + (1 << 15)].T) * 2.0 ** (-18 * (i + j))
                s = hi + t
                b = s - hi
                lo += (hi - (s - b)) + (t - b)
                hi = s
    return (hi + lo) * e * e.T


# one tile; a ragged one; two and four rows of tiles of 256; K in groups; two and three K panels
@pytest.mark.parametrize("k,K", [(1, 1), (33, 100), (257, 700), (600, 5400), (300, 16385), (70, 40001), (1025, 512)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_entries(k, K, dtype):
    rng = np.random.default_rng(k + K)
    X = (rng.standard_normal((k, K)) * 10.0 ** rng.uniform(-3, 3, (k, 1)) * 10.0 ** rng.uniform(-4, 0, (1, K))).astype(dtype)
    got = gdml.test_oz_syrk(torch.from_numpy(X).cuda()).cpu().numpy()
    X = X.astype(np.float64)
    ref = np.tril(exact_products(X))
    panels = -(-K // 16384)
    Kp = min(K, 16384)
    m, s = np.abs(X).max(axis=1), np.abs(X).sum(axis=1)
    bound = 2.0 ** -57 * np.sqrt(Kp) * (np.outer(m, s) + np.outer(s, m)) + panels * 1.5 * 2.0 ** -57 * Kp * np.outer(m, m)
    bound += panels * EPS * (np.abs(X) @ np.abs(X).T) + 2 * EPS * np.abs(ref)
    worst = (np.abs(got - ref) / bound).max()
    print(f"k={k} K={K} {np.dtype(dtype).name}: max error / bound = {worst:.3f}")
    assert worst <= 1.0
    assert np.array_equal(got, np.tril(got))
