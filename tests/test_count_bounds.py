"""count_bound and count_bound2 (render_common.cuh) by their formulas, operation for
operation, on the CPU: both squares, both moduli, with the kernels' own |c| (the
norm of its eight components) and their decisions.  The distance of an orbit in
floats, or in pairs of floats, from the exact one stays within the bound at every
step, and a count that is certain is the exact orbit's."""
import numpy as np
import pytest

F, D = np.float32, np.float64
L = np.longdouble  # at least 64 bits of mantissa: the exact orbit beside pairs of floats (48 bits)
U = 2.0 ** -24


def fma(a, b, c):  # FP32: the product of two floats is exact in double
    return (a.astype(D) * b.astype(D) + np.asarray(c, D)).astype(F)


def qmul(a, b):
    return np.stack([a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3],
                     a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2],
                     a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1],
                     a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0]])


def square(x, sq):
    r, d = x[:4], x[4:]
    return np.concatenate([qmul(r, r), qmul(r, d) + qmul(d, r) if sq == 0 else qmul(d, d)])


def norm(h):
    return np.sqrt((h * h).sum(0))


def modulus(x, mod):
    return (x[:4] ** 2).sum(0) + ((x[4:] ** 2).sum(0) if mod == 0 else 0)


def step32(z, sp, c, sq):  # dq_iter<float>, term by term
    t, td, one = z[0] + z[0], z[4] + z[4], np.full_like(z[0], 1)
    w = np.empty_like(z)
    w[0] = fma(z[0], z[0], fma(sp, -one, c[0]))
    for i in (1, 2, 3):
        w[i] = fma(t, z[i], c[i])
    if sq == 0:
        q = fma(z[3], z[7], fma(z[2], z[6], z[1] * z[5]))
        w[4] = fma(q, -2 * one, fma(t, z[4], c[4]))
        for i in (5, 6, 7):
            w[i] = fma(t, z[i], fma(td, z[i - 4], c[i]))
    else:
        w[4] = fma(z[4], z[4], fma(fma(z[7], z[7], fma(z[6], z[6], z[5] * z[5])), -one, c[4]))
        for i in (5, 6, 7):
            w[i] = fma(td, z[i], c[i])
    return w, fma(w[3], w[3], fma(w[2], w[2], w[1] * w[1]))


class Sum2:  # render_common.cuh: Sum2
    def __init__(self, h, l):
        self.h, self.l = h.copy(), l.copy()

    def add_product(self, ah, al, bh, bl):
        p = ah * bh
        e = fma(ah, bl, fma(al, bh, fma(ah, bh, -p)))
        s = self.h + p
        b = s - self.h
        self.l = self.l + (((self.h - (s - b)) + (p - b)) + e)
        self.h = s

    def done(self):
        oh = self.h + self.l
        return oh, self.l - (oh - self.h)


def step2(zh, zl, c, sq):
    ch = c.astype(F)
    cl = (c - ch.astype(D)).astype(F)
    out = []
    t0h, t0l, s0h, s0l = zh[0] + zh[0], zl[0] + zl[0], zh[4] + zh[4], zl[4] + zl[4]
    a = Sum2(ch[0], cl[0])
    a.add_product(zh[0], zl[0], zh[0], zl[0])
    for i in (1, 2, 3):
        a.add_product(-zh[i], -zl[i], zh[i], zl[i])
    out.append(a.done())
    for i in (1, 2, 3):
        a = Sum2(ch[i], cl[i])
        a.add_product(t0h, t0l, zh[i], zl[i])
        out.append(a.done())
    a = Sum2(ch[4], cl[4])
    if sq == 0:
        a.add_product(t0h, t0l, zh[4], zl[4])
        for i in (1, 2, 3):
            a.add_product(F(-2) * zh[i], F(-2) * zl[i], zh[4 + i], zl[4 + i])
    else:
        a.add_product(zh[4], zl[4], zh[4], zl[4])
        for i in (5, 6, 7):
            a.add_product(-zh[i], -zl[i], zh[i], zl[i])
    out.append(a.done())
    for i in (5, 6, 7):
        a = Sum2(ch[i], cl[i])
        if sq == 0:
            a.add_product(t0h, t0l, zh[i], zl[i])
            a.add_product(s0h, s0l, zh[i - 4], zl[i - 4])
        else:
            a.add_product(s0h, s0l, zh[i], zl[i])
        out.append(a.done())
    return np.stack([o[0] for o in out]), np.stack([o[1] for o in out])


def bound_step(er, ed, ar, ad, rounding, sq, mod):
    ner = er * (2 * ar + er) + rounding
    if mod == 0:
        ed = 2 * (ar * ed + ad * er + er * ed) + rounding if sq == 0 else ed * (2 * ad + ed) + rounding
    return ner, ed


CASES = [(sq, mod, pair) for sq in (0, 1) for mod in (0, 1) for pair in (False, True)]


@pytest.mark.parametrize("sq,mod,pair", CASES)
@pytest.mark.parametrize("scale,radius", [(0.05, 0.7), (0.5, 2.0), (2.0, 4.0)])
def test_bound_and_decision(sq, mod, pair, scale, radius):
    rng = np.random.default_rng(17)
    n, steps = 3000, 24
    c = rng.uniform(-0.8, 0.8, (8, n))
    c[:, : n // 4] *= 0.2  # bounded orbits
    c[4:, n // 2:] *= rng.choice([0.0, 1.0], (1, n - n // 2))
    c = c.astype(F).astype(D) + (rng.uniform(-1, 1, c.shape) * U * np.abs(c))  # doubles near a float, on either side
    x0 = rng.uniform(-scale, scale, (8, n))
    R2 = radius * radius
    x = x0.astype(L)
    zh = x0.astype(F)
    zl = (x0 - zh.astype(D)).astype(F)
    c32 = c.astype(F)
    cn = norm(c)  # of all eight components, as the kernels' settle_cn
    u = U * U if pair else U
    if pair:
        er = 4 * u * ((x0 ** 2)[:4].sum(0) + ((x0 ** 2)[4:].sum(0) if mod == 0 else 0) + 1)
        ed = er.copy()
    else:
        er = 6.1e-8 * norm(x0)
        ed = er.copy()
    sp = fma(zh[3], zh[3], fma(zh[2], zh[2], zh[1] * zh[1]))
    open_, count, exact, certain = np.ones(n, bool), np.zeros(n, int), np.zeros(n, int), np.ones(n, bool)
    going = np.ones(n, bool)  # the exact orbit has not escaped
    worst = 0.0
    for k in range(1, steps + 1):
        with np.errstate(all="ignore"):
            r2 = (zh[:4].astype(D) ** 2).sum(0)
            d2 = (zh[4:].astype(D) ** 2).sum(0)
            rounding = (128 * u if pair else 5.6 * u) * ((r2 + d2 if mod == 0 else r2) + cn)
            er, ed = bound_step(er, ed, np.sqrt(r2), np.sqrt(d2), rounding, sq, mod)
            if pair:
                zh, zl = step2(zh, zl, c, sq)
            else:
                zh, sp = step32(zh, sp, c32, sq)
            x = square(x, sq) + c
            z = zh.astype(L) + (zl if pair else 0)
            dr, dd = norm((x - z)[:4]), norm((x - z)[4:])
            sure = going & open_
            assert np.all(dr[sure] <= er[sure]), k
            if mod == 0:
                assert np.all(dd[sure] <= ed[sure]), k
            worst = max(worst, float((dr[sure] / er[sure]).max(initial=0)))
            m = modulus(zh.astype(D), mod)
            dev = er * (2 * np.sqrt((zh[:4].astype(D) ** 2).sum(0)) + er)
            if mod == 0:
                dev = dev + ed * (2 * np.sqrt((zh[4:].astype(D) ** 2).sum(0)) + ed)
            dev = 1.01 * dev + (14 if pair else 10) * U * m
            esc = open_ & (m - dev > R2 * (1 + 2 * U))
            undecided = open_ & ~esc & ~(m + dev < R2 * (1 - 2 * U))
            exact_esc = going & ~(modulus(x, mod) <= R2)
        count[esc] = k
        certain[undecided] = False
        open_ &= ~(esc | undecided)
        exact[exact_esc] = k
        going &= ~exact_esc
        if not open_.any():
            break
    count[~certain] = -1
    done = certain & ~(open_ & ~going)
    assert np.array_equal(count[done], exact[done]) and np.all(done[certain])
    assert certain.mean() > (0.99 if pair else 0.9) or scale < 0.1 and certain.mean() > 0.8
    assert 1e-4 < worst <= 1.0  # the bound is met, and not by orders of magnitude
