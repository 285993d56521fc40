"""The double-float far field's expanded form, emulated on the CPU in FP32 (numpy float32
arithmetic is IEEE single precision, round to nearest; an FMA is its exact product and
sum, rounded once).

For a pair of triangles whose centroids are at least 1.5 (R_i + R_j) apart the form expands
|x_a - y_b|^2 = |d|^2 + A_a + B_b - C_ab, d = c_i - c_j, into dot products of d and of the
offsets of one quadrature orbit, each split on one power-of-two grid per pair so that every
sum of hi parts is exact.  These tests pin the properties that the kernel relies on: the hi
sums are exact, the estimates' sums are exact, and the entry sums stay within 1e-12 of FP64 (the two-sum
form's are within 3e-13), their mean error within 5e-14, on seeded meshes with needles.
"""
import numpy as np
import pytest

from paper_1901_08393_gb300 import inputs
from tests.test_far_grid_form import BARY, F, W, fma, grid_pairs, pos_two_sum, snap, two_sum, fast_two_sum

SQ15 = np.sqrt(15.0)
T1 = (1.0 + SQ15) / 7.0              # first orbit: offset T1 (vertex - centroid)
S1 = (1.0 - SQ15) / (1.0 + SQ15)     # second orbit: S1 times the first
SPREAD = 1.5                         # least |d| / (R_i + R_j)


def split(v):
    h = np.asarray(v, np.float64).astype(F)
    return h, (np.asarray(v, np.float64) - h.astype(np.float64)).astype(F)


S1H, S1L = split(S1)
S2H, S2L = split(S1 * S1)


def exponent_field(v, up):
    """1.5 * 2^(e + up), 2^e <= v < 2^(e + 1)."""
    return (((v.view(np.uint32) & np.uint32(0x7F800000)) + np.uint32(up << 23)) | np.uint32(0x400000)).view(F)


class Grid:
    """hi parts are multiples of the pair's q: every plain sum of them must be exact."""

    def __init__(self, big):
        self.big, self.exact = big, True

    def add(self, *hs):
        s = hs[0]
        for h in hs[1:]:
            t = (s + h).astype(F)
            self.exact &= bool(np.array_equal(t.astype(np.float64), s.astype(np.float64) + h.astype(np.float64)))
            s = t
        return s

    def prod(self, ah, al, bh, bl):
        """(ah + al) (bh + bl) as a multiple of q and the rest."""
        h = (fma(ah, bh, self.big) - self.big).astype(F)
        r = fma(ah, bh, -h)
        r = fma(al, bh, r)
        return h, fma(ah, bl, r)

    def snap(self, h, l):
        g = snap(h, self.big)
        return g, ((h - g).astype(F) + l).astype(F)

    def dot(self, a, b):
        hs, ls = zip(*(self.prod(*x, *y) for x, y in zip(a, b)))
        return self.add(*hs), ((ls[0] + ls[1]).astype(F) + ls[2]).astype(F)


def expanded_form(m, pairs, mufu):
    P = m.verts[m.tris]
    c = (P[:, 0] + P[:, 1] + P[:, 2]) / 3.0
    V = T1 * (P - c[:, None, :])
    n1 = (V ** 2).sum(axis=2)
    n2h = [split(n1[:, k]) for k in range(3)]
    n2s = [split(S1 * S1 * n1[:, k]) for k in range(3)]
    off = np.einsum("ak,nkc->nac", BARY, P - c[:, None, :])
    R = np.nextafter(np.linalg.norm(off, axis=2).max(axis=1).astype(F), F(np.inf))
    c0 = c.astype(F)
    r1 = c - c0.astype(np.float64)
    c1 = r1.astype(F)
    c2 = (r1 - c1.astype(np.float64)).astype(F)
    I, J = pairs[:, 0], pairs[:, 1]
    s1, e1 = two_sum(c0[I], -c0[J])
    s2, e2 = two_sum(c1[I], -c1[J])
    hh, ll = two_sum(s1, s2)
    dh, dl = fast_two_sum(hh, (ll + ((e1 + e2).astype(F) + (c2[I] - c2[J]).astype(F)).astype(F)).astype(F))
    D2 = (dh * dh).sum(axis=1, dtype=F)
    Rs = (R[I] + R[J]).astype(F)
    take = D2 >= F(SPREAD * SPREAD * 1.0001) * (Rs * Rs)
    I, J, dh, dl, D2 = I[take], J[take], dh[take], dl[take], D2[take]
    g = Grid(exponent_field((F(1.34) * D2).astype(F), 2))
    d = [(dh[:, k], dl[:, k]) for k in range(3)]
    d2 = [((F(2) * h).astype(F), (F(2) * l).astype(F)) for h, l in d]
    # |d|^2
    Dp = [(lambda h: (h, fma(b[0], a[1], fma(a[0], a[0], -h))))((fma(a[0], a[0], g.big) - g.big).astype(F))
          for a, b in zip(d, d2)]
    Dh = g.add(*[x[0] for x in Dp])
    Dl = ((Dp[0][1] + Dp[1][1]).astype(F) + Dp[2][1]).astype(F)

    def vec(T, k, sign):
        return [tuple((sign * x).astype(F) for x in split(V[T, k, q])) for q in range(3)]

    def side(T, sign):
        """The 6 terms sign 2 d.o + |o|^2 of a triangle's offsets o, orbit 1 then 2."""
        out1, out2 = [], []
        p = [g.dot(d2, vec(T, k, F(sign))) for k in range(2)]
        p.append((-g.add(p[0][0], p[1][0]), -(p[0][1] + p[1][1]).astype(F)))
        for k in range(3):
            nh, nl = g.snap(n2h[k][0][T], n2h[k][1][T])
            out1.append((g.add(p[k][0], nh), (p[k][1] + nl).astype(F)))
            nh, nl = g.snap(n2s[k][0][T], n2s[k][1][T])
            h, l = g.prod(S1H, S1L, *p[k])
            out2.append((g.add(h, nh), (l + nl).astype(F)))
        return [(np.zeros_like(D2), np.zeros_like(D2))] + out1 + out2

    A, B = side(I, 1), side(J, -1)
    two = [[tuple((F(2) * x).astype(F) for x in q) for q in vec(I, k, F(1))] for k in range(2)]
    G = [[g.dot(two[k], vec(J, l, F(1))) for l in range(2)] for k in range(2)]
    neg = lambda x, y: (-g.add(x[0], y[0]), -(x[1] + y[1]).astype(F))
    for k in range(2):
        G[k].append(neg(G[k][0], G[k][1]))
    G.append([neg(G[0][l], G[1][l]) for l in range(3)])
    C = [[None] * 7 for _ in range(7)]
    for k in range(3):
        for l in range(3):
            C[1 + k][1 + l] = G[k][l]
            C[1 + k][4 + l] = C[4 + k][1 + l] = g.prod(S1H, S1L, *G[k][l])
            C[4 + k][4 + l] = g.prod(S2H, S2L, *G[k][l])
    y0 = (1.0 / np.sqrt(Dh.astype(np.float64))).astype(F)
    gy = Grid(exponent_field(y0, 6))
    classes = {}
    for a in range(7):
        eh, el = g.add(Dh, A[a][0]), (Dl + A[a][1]).astype(F)
        for b in range(7):
            H, L = g.add(eh, B[b][0]), (el + B[b][1]).astype(F)
            if C[a][b] is not None:
                H, L = g.add(H, -C[a][b][0]), (L - C[a][b][1]).astype(F)
            y = ((1.0 / np.sqrt(H.astype(np.float64))) * mufu(len(H))).astype(F)
            y = snap(y, gy.big)
            y2 = (y * y).astype(F)
            y2e = fma(y, y, -y2)
            t = fma(-H, y2, F(1))
            t = fma(-H, y2e, t)
            t = fma(-L, y2, t)
            corr = (t * fma(t, F(0.375), F(0.5))).astype(F)
            key = tuple(sorted(((a + 2) // 3, (b + 2) // 3)))
            s, l = classes.get(key, (np.zeros_like(y), np.zeros_like(y)))
            classes[key] = (gy.add(s, y), fma(y, corr, l))
    acc_h, acc_l = np.zeros_like(y0), np.zeros_like(y0)
    for (p, q), (s, l) in classes.items():
        w = W[3 * p] * W[3 * q]
        wh, wl = split(w)
        ph = (wh * s).astype(F)
        pe = fma(wl, s, fma(wh, l, fma(wh, s, -ph)))
        u, ue = pos_two_sum(acc_h, ph)
        acc_h, acc_l = u, (acc_l + (pe + ue).astype(F)).astype(F)
    x = c[:, None, :] + off
    ref = np.einsum("a,b,nab->n", W, W,
                    1.0 / np.linalg.norm(x[I][:, :, None, :] - x[J][:, None, :, :], axis=3))
    return (acc_h.astype(np.float64) + acc_l.astype(np.float64)) / ref - 1.0, g.exact, gy.exact, take.mean()


@pytest.mark.parametrize("make", [lambda: inputs.graded_cube_mesh(8), lambda: inputs.cube_mesh(6),
                                  lambda: inputs.fichera_mesh(2), lambda: inputs.workload_polycube_adaptive()],
                         ids=["graded-needles", "cube6", "fichera2", "polycube"])
@pytest.mark.parametrize("bias", [-1, 0, 1], ids=["low", "random", "high"])
def test_expanded_form_exact_hi_sums_and_entry_error(make, bias):
    """bias: the reciprocal square root's estimate 2^-22 low, high, or anywhere between."""
    m = make()
    rng = np.random.default_rng(7)
    mufu = (lambda n: 1.0 + bias * 2.0 ** -22) if bias else (lambda n: 1.0 + rng.uniform(-1, 1, n) * 2.0 ** -22)
    err, exact, exact_y, frac = expanded_form(m, grid_pairs(m, 4000, 3), mufu)
    assert exact, "a sum of hi parts was rounded"
    assert exact_y, "a sum of estimates was rounded"
    assert frac > 0.2 and len(err) > 1000, (frac, len(err))
    assert np.abs(err).max() < 1e-12 and abs(err.mean()) < 5e-14, (np.abs(err).max(), err.mean(), err.std())
