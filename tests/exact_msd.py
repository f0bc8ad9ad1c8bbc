"""Trial quantities in 60 decimal digits, for walkers whose determinants cancel or
differ in scale by more than FP64 oracles hold: every determinant's overlap, Green's
function and energy by its own inverse (Sec. II A), then the CI sums. Slow: small
systems and a handful of walkers. Also the minors of a matrix and how far a pivoted
LU may be from them."""
import decimal

import numpy as np

decimal.getcontext().prec = 60
_D = np.frompyfunc(lambda x: decimal.Decimal(float(x)), 1, 1)
_F = np.frompyfunc(float, 1, 1)


class Z:
    """Complex array of Decimals."""
    def __init__(self, re, im):
        self.re, self.im = np.asarray(re, dtype=object), np.asarray(im, dtype=object)

    @staticmethod
    def of(x):
        x = np.asarray(x)
        return Z(_D(x.real), _D(x.imag if np.iscomplexobj(x) else np.zeros(x.shape)))

    def __getitem__(self, k):
        return Z(self.re[k], self.im[k])

    def __add__(self, o):
        return Z(self.re + o.re, self.im + o.im)

    def __sub__(self, o):
        return Z(self.re - o.re, self.im - o.im)

    def __mul__(self, o):
        return Z(self.re * o.re - self.im * o.im, self.re * o.im + self.im * o.re)

    def __truediv__(self, o):
        d = o.re * o.re + o.im * o.im
        return Z((self.re * o.re + self.im * o.im) / d, (self.im * o.re - self.re * o.im) / d)

    def __matmul__(self, o):
        return Z(self.re.dot(o.re) - self.im.dot(o.im), self.re.dot(o.im) + self.im.dot(o.re))

    @property
    def T(self):
        return Z(self.re.T, self.im.T)

    def sum(self):
        return Z(self.re.sum(), self.im.sum())

    def num(self):
        return np.asarray(_F(self.re)).astype(float) + 1j * np.asarray(_F(self.im)).astype(float)


def det_inverse(a):
    """Determinant and inverse (None where singular) of a square Z, by Gauss-Jordan."""
    n = a.re.shape[0]
    re = np.concatenate([a.re, _D(np.eye(n))], 1)
    im = np.concatenate([a.im, _D(np.zeros((n, n)))], 1)
    det = Z.of(1.0)
    for k in range(n):
        p = k + int(np.argmax([max(abs(re[i, k]), abs(im[i, k])) for i in range(k, n)]))
        if re[p, k] == 0 and im[p, k] == 0:
            return Z.of(0.0), None
        if p != k:
            for m in (re, im):
                m[[k, p]] = m[[p, k]]
            det = Z.of(-1.0) * det
        piv = Z(re[k, k], im[k, k])
        det = det * piv
        row = Z(re[k], im[k]) / piv
        re[k], im[k] = row.re, row.im
        for i in range(n):
            if i != k:
                r = Z(re[i], im[i]) - Z(re[i, k], im[i, k]) * row
                re[i], im[i] = r.re, r.im
    return det, Z(re[:, n:], im[:, n:])


def minor(a):
    """(determinant, bound of a pivoted LU's error) of a square complex array: the
    computed determinant is that of a + e, so off by |e| times the cofactors; |e| below
    2 k u max|a| per entry in complex arithmetic, times a growth of the pivots that for
    k <= 6 stays below 4."""
    d, inv = det_inverse(Z.of(a))
    if inv is None:
        return 0j, 0.0
    cof = np.abs((inv * d).num()).sum()
    return complex(d.num()), 8 * a.shape[0] * 2.0 ** -53 * float(np.abs(a).max()) * float(cof)


def msd(s, phi_a, phi_b):
    """Per walker: det_ovlp (n_det,), G_I and det_e per determinant, ovlp, e_loc, vbias,
    G_T, as FP64 arrays of the exact values."""
    M, G = s.M, s.n_chol
    h1, L = [Z.of(s.h1[i]) for i in (0, 1)], [Z.of(s.L[g]) for g in range(G)]
    out = []
    for w in range(phi_a.shape[0]):
        det = []
        cache = [{}, {}]
        for I in range(s.n_det):
            o, gs, tr, ex, e1 = Z.of(1.0), [], [], Z.of(0.0), Z.of(0.0)
            for sp, (occ, phi) in enumerate(((s.occ_a, phi_a), (s.occ_b, phi_b))):
                key = tuple(occ[I])
                if key not in cache[sp]:
                    p = Z.of(phi[w])
                    d, inv = det_inverse(p[occ[I]])
                    g = np.zeros((M, M)).astype(object)
                    th = p @ inv                                  # [M][N]; G[occ_j][q] = theta[q][j]
                    gz = Z(_D(g), _D(g))
                    gz.re[occ[I]], gz.im[occ[I]] = th.re.T, th.im.T
                    lg = [x @ gz for x in L]
                    t = [Z(np.trace(x.re), np.trace(x.im)) for x in lg]
                    q = Z.of(0.0)
                    for x in lg:
                        q = q + (x * x.T).sum()
                    cache[sp][key] = (d, gz, t, q, (h1[sp] * gz.T).sum())
                d, gz, t, q, e = cache[sp][key]
                o = o * d
                gs.append(gz)
                tr.append(t)
                ex = ex + q
                e1 = e1 + e
            half = Z.of(0.5)
            cl = Z.of(0.0)
            for g in range(G):
                v = tr[0][g] + tr[1][g]
                cl = cl + v * v
            det.append((o, gs, tr, Z.of(s.e0) + e1 + half * (cl - ex)))
        c = [Z.of(float(x)) for x in s.coeff]
        ov = Z.of(0.0)
        for x, y in zip(c, det):
            ov = ov + x * y[0]
        e, vb, gt = Z.of(0.0), [Z.of(0.0) for _ in range(G)], [Z.of(np.zeros((M, M))) for _ in (0, 1)]
        for x, (o, gs, tr, ei) in zip(c, det):
            f = x * o / ov
            e = e + f * ei
            vb = [v + f * (tr[0][g] + tr[1][g]) for g, v in enumerate(vb)]
            gt = [a + f * b for a, b in zip(gt, gs)]
        out.append(dict(det_ovlp=np.array([complex(y[0].num()) for y in det]),
                        det_e=np.array([complex(y[3].num()) for y in det]),
                        det_g=np.array([[g.num() for g in y[1]] for y in det]),
                        ovlp=complex(ov.num()), e_loc=complex(e.num()),
                        vbias=np.array([complex(v.num()) for v in vb]), G_T=np.stack([g.num() for g in gt])))
    return {k: np.array([o[k] for o in out]) for k in out[0]}


def with_strings(s, n_o, n_act, pairs, rng):
    """System s with `count` random determinants of each (level_a, level_b, count)
    over n_o active occupied of n_act active orbitals, no core."""
    ref = tuple(range(n_o))
    occ = {(ref, ref): 1.0}

    def string(k):
        keep = np.delete(np.arange(n_o), rng.choice(n_o, k, replace=False))
        return tuple(sorted(np.concatenate([keep, n_o + rng.choice(n_act - n_o, k, replace=False)]).tolist()))

    for ka, kb, count in pairs:
        for _ in range(count):
            occ.setdefault((string(ka), string(kb)), rng.normal() / np.sqrt(count))
    s.occ_a = np.array([a for a, _ in occ], np.int32)
    s.occ_b = np.array([b for _, b in occ], np.int32)
    s.coeff = np.array(list(occ.values()))
    return s


def levels(occ):
    """Holes and particles (orbital numbers) of every row against row 0."""
    ref = set(occ[0].tolist())
    return [(sorted(ref - set(r.tolist())), sorted(set(r.tolist()) - ref)) for r in occ]
