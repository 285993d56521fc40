"""The native FP64 far field's expanded form, emulated on the CPU (an FMA is its exact product and
sum by two-products and two-sums, rounded once).

Pairs at least 1.5 (R_i + R_j) apart take |x_a - y_b|^2 = E_a + n_b - 2 e_a.o_b about the column
triangle's centroid, the reciprocal root as an FP32 estimate on a grid and a correction of two
terms.  Against extended precision on the same points its entries err no more than those of the
sum of FP64 reciprocal roots of differences: r.m.s. within 10% of that sum's, and below the bound
of the expansion, 54 roundings (4 of terms of at most 3 |d|^2 in a square of at least |d|^2 / 9,
halved by the root)."""
import numpy as np
import pytest

from paper_1901_08393_gb300 import inputs
from tests.test_far_grid_form import BARY, W, grid_pairs

L, F = np.longdouble, np.float32
U = 2.0 ** -53


def two_prod(a, b):
    p, c = a * b, 134217729.0
    ah, bh = a * c, b * c
    ah, bh = ah - (ah - a), bh - (bh - b)
    al, bl = a - ah, b - bh
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def fma(a, b, c):
    a, b, c = np.broadcast_arrays(a, b, c)
    p, e = two_prod(a, b)
    s = p + c
    t = s - p
    return s + (((p - (s - t)) + (c - t)) + e)


def truncated(v):
    """A positive double truncated to FP32."""
    return (np.ascontiguousarray(v).view(np.uint64) & ~np.uint64((1 << 29) - 1)).view(np.float64).astype(F)


def entries(m, pairs, mufu):
    P = m.verts[m.tris]
    c = ((P[:, 0] + P[:, 1]) + P[:, 2]) / 3.0
    X = np.einsum("ak,nkc->nac", BARY, P)
    I, J = pairs[:, 0], pairs[:, 1]
    radius = np.linalg.norm(X - c[:, None], axis=2).max(axis=1)
    D2 = ((c[I] - c[J]) ** 2).sum(axis=1)
    take = D2 >= 2.2505 * (radius[I] + radius[J]) ** 2
    I, J, D2 = I[take], J[take], D2[take]
    exact, plain = np.zeros(len(I), L), np.zeros(len(I))
    for a in range(7):
        s = np.zeros(len(I))
        for b in range(7):
            d = X[I, a].astype(L) - X[J, b].astype(L)
            exact += L(W[a]) * L(W[b]) / np.sqrt((d * d).sum(axis=1))
            e = X[I, a] - X[J, b]
            r2 = fma(e[:, 2], e[:, 2], fma(e[:, 1], e[:, 1], e[:, 0] * e[:, 0]))
            s = fma(W[b], (1 / np.sqrt(r2.astype(L))).astype(np.float64), s)
        plain = fma(W[a], s, plain)
    y0 = (1 / np.sqrt(truncated(D2).astype(np.float64))).astype(F)
    big = (((y0.view(np.uint32) & np.uint32(0x7F800000)) + np.uint32(6 << 23)) | np.uint32(0x400000)).view(F)
    o = (X - c[:, None])[J]
    n = fma(o[..., 2], o[..., 2], fma(o[..., 1], o[..., 1], o[..., 0] * o[..., 0]))
    cls = ((0, 1, 2), (1, 3, 4), (2, 4, 5))
    s, q, l = np.zeros((6, len(I)), F), np.zeros((6, len(I)), F), np.zeros((6, len(I)))
    whole = True
    for a in range(7):
        e = X[I, a] - c[J]
        E = fma(e[:, 2], e[:, 2], fma(e[:, 1], e[:, 1], e[:, 0] * e[:, 0]))
        for b in range(7):
            k = cls[(a + 2) // 3][(b + 2) // 3]
            S = E + n[:, b]
            for x in range(3):
                S = fma(-2 * e[:, x], o[:, b, x], S)
            y = ((1 / np.sqrt(truncated(S).astype(np.float64))) * mufu(len(I))).astype(F)
            y = ((y + big).astype(F) - big).astype(F)
            yd = y.astype(np.float64)
            t = fma(-S, yd * yd, 1.0)
            tf = truncated(np.maximum(np.abs(t), 2.0 ** -127))
            new = (s[k] + y).astype(F)
            whole &= bool(np.array_equal(new.astype(np.float64), s[k].astype(np.float64) + yd))
            s[k] = new
            l[k] = fma(yd, t, l[k])
            q[k] = ((y * tf).astype(F).astype(np.float64) * tf + q[k]).astype(F)
    w = [W[0] * W[0], W[0] * W[1], W[0] * W[4], W[1] * W[1], W[1] * W[4], W[4] * W[4]]
    acc = np.zeros(len(I))
    for k in range(6):
        acc = fma(w[k], fma(0.5, l[k], s[k].astype(np.float64)) + (F(0.375) * q[k]).astype(np.float64), acc)
    return (acc / exact - 1).astype(np.float64), (plain / exact - 1).astype(np.float64), whole


@pytest.mark.parametrize("make", [lambda: inputs.graded_cube_mesh(8), lambda: inputs.cube_mesh(6),
                                  lambda: inputs.workload_polycube_adaptive(),
                                  lambda: inputs.transformed(inputs.graded_cube_mesh(14),
                                                             inputs.random_rotation(inputs.SplitMix64(11)), 0.7, (1, 2, 3))],
                         ids=["graded-needles", "cube6", "polycube", "graded-rotated"])
@pytest.mark.parametrize("bias", [-1, 0, 1], ids=["low", "random", "high"])
def test_entry_error_is_that_of_fp64_sums(make, bias):
    """bias: the reciprocal square root's estimate 2^-22 low, high, or anywhere between."""
    rng = np.random.default_rng(5)
    mufu = (lambda n: 1.0 + bias * 2.0 ** -22) if bias else (lambda n: 1.0 + rng.uniform(-1, 1, n) * 2.0 ** -22)
    m = make()
    pairs = grid_pairs(m, 6000, 3)
    err, plain, whole = entries(m, pairs[::max(1, len(pairs) // 12000)], mufu)
    assert whole, "a sum of estimates was rounded"
    rms, rms_plain = np.sqrt((err ** 2).mean()), np.sqrt((plain ** 2).mean())
    assert len(err) > 1000 and rms <= 1.1 * rms_plain, (len(err), rms, rms_plain)
    assert np.abs(err).max() <= 54 * U, np.abs(err).max() / U
