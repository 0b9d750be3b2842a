"""G = Y S Y^T and Z = Y^T G^{-1} of mixed levels: FP32 entries, sums that hold FP64's digits whatever their length.

Exact products, summed in three FP32 parts whose first two are updated without loss, so only the last additions round:
    |fl(g_ab) - g_ab| <= 2^-52 sum_c |y_ac| |y_bc|      (the parts are added in FP64, two roundings).
For Z the FP64 matrix enters as a pair of FP32 numbers (2^-48 of each entry at most), a product's second part is
rounded once (2^-47 of the product) and the sum is rounded to FP32:
    |fl(z_cq) - z_cq| <= 2^-24 |z_cq| + 2^-46 sum_p |y_pc| |h_pq|.
Sums in two parts miss the first bound by a factor of 2^6 at 64 terms and 2^12 at 6,000.  Sizes: one tile, ragged
tiles, several of them, long sums; signed levels; and moduli in very small and very large units, whose square root
the rows carry."""
import numpy as np
import pytest

pytest.importorskip("torch")

from paper_1201_5991_gb300.solver import gram_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("positive", [False, True])
@pytest.mark.parametrize("n,nc,rho", [(64, 64, 1.0), (1, 3, 1.0), (130, 65, 1.0), (777, 200, 1e3), (6001, 97, 1.0),
                                      (500, 70, 1e-34), (500, 70, 1e34)])
def test_sums_keep_fp64_digits(n, nc, rho, positive):
    rng = np.random.default_rng(n + nc)
    y = rng.standard_normal((nc, n)) * 10.0 ** rng.uniform(-2, 0, size=(nc, 1)) / np.sqrt(rho * n)
    if positive:
        y = np.abs(y)
    y = y.astype(np.float32)
    sgn = (np.ones(n) if positive else rng.choice([-1.0, 1.0], size=n)).astype(np.float32)
    h = rng.standard_normal((nc, nc)) * rho
    h = (np.abs(h) if positive else h) + (np.abs(h.T) if positive else h.T)
    g, z = gram_check(y, sgn, h, rho)
    Y, S, H = y.astype(np.longdouble), sgn.astype(np.longdouble), h.astype(np.longdouble)
    eg, ez = (Y * S) @ Y.T, Y.T @ H
    ag, az = np.abs(y).astype(float) @ np.abs(y).astype(float).T, np.abs(y).astype(float).T @ np.abs(h)
    dg, dz = np.abs((g - eg).astype(float)), np.abs((z - ez).astype(float))
    print(f"n {n} n_c {nc} rho {rho:g} positive {positive}: G rms 2^{np.log2(max(np.sqrt(np.mean((dg / ag) ** 2)), 1e-30)):.1f}, "
          f"max 2^{np.log2(max((dg / ag).max(), 1e-30)):.1f}; Z beyond its rounding at most 2^"
          f"{np.log2(max(((dz - 2.0 ** -24 * np.abs(ez.astype(float))) / az).max(), 1e-30)):.1f}")
    assert np.all(dg <= 2.0 ** -52 * ag)
    assert np.all(dz <= 2.0 ** -24 * np.abs(ez.astype(float)) + 2.0 ** -46 * az)
    np.testing.assert_array_equal(g, g.T)
