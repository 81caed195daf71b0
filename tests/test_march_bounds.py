"""The two bounds behind the march's settled blocks and its recheck (no GPU), by
their formulas on random orbits.

count_bound (render_common.cuh): an FP32 orbit lies within er (real half) and ed
(dual half) of the exact one.  settle_box (settle.cuh): every point of a box goes
to z + sum u_a g_a + e with |e_r| <= er, |e_d| <= ed.  Both must hold at every step,
whatever the orbit: the comparison is exact up to FP64, whose rounding the 1e-12
covers (orbits below |zeta| = 8, at most 10 steps)."""
import numpy as np
import pytest

U = 2.0 ** -24
F = np.float32


def qmul(a, b):
    return np.stack([a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3],
                     a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2],
                     a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1],
                     a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0]])


def mul(a, b):  # dual quaternions, eps^2 = 0
    return np.concatenate([qmul(a[:4], b[:4]), qmul(a[:4], b[4:]) + qmul(a[4:], b[:4])])


def norm(h):
    return np.sqrt((h * h).sum(0))


def fma(a, b, c):  # FP32: the product of two floats is exact in double
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def step32(z, sp, c):  # dq_iter<float, algebraic>, term by term
    t, td, one = z[0] + z[0], z[4] + z[4], np.full_like(z[0], -1)
    w = np.empty_like(z)
    w[0] = fma(z[0], z[0], fma(sp, one, c[0]))
    for i in (1, 2, 3):
        w[i] = fma(t, z[i], c[i])
    q = fma(z[3], z[7], fma(z[2], z[6], z[1] * z[5]))
    w[4] = fma(q, 2 * one, fma(t, z[4], c[4]))
    for i in (5, 6, 7):
        w[i] = fma(t, z[i], fma(td, z[i - 4], c[i]))
    return w, fma(w[3], w[3], fma(w[2], w[2], w[1] * w[1]))


@pytest.mark.parametrize("seed", range(4))
@pytest.mark.parametrize("scale", [0.05, 0.5, 2.0])
def test_rounding_bound(seed, scale):
    rng = np.random.default_rng(seed)
    n = 2000
    c = rng.uniform(-0.8, 0.8, (8, n))
    x = rng.uniform(-scale, scale, (8, n))
    z, c32 = x.astype(F), c.astype(F)
    er, ed = norm(x[:4] - z[:4]), norm(x[4:] - z[4:])
    sp = fma(z[3], z[3], fma(z[2], z[2], z[1] * z[1]))
    cn = norm(c[:4]) + norm(c[4:])
    live = np.ones(n, bool)
    for _ in range(10):
        zr, zd = norm(z[:4].astype(np.float64)), norm(z[4:].astype(np.float64))
        live &= zr ** 2 + zd ** 2 <= 16.0
        rounding = 5.6 * U * (zr ** 2 + zd ** 2 + cn)
        er, ed = 2 * zr * er + er ** 2 + rounding, 2 * (zr * ed + zd * er + er * ed) + rounding
        with np.errstate(all="ignore"):
            z, sp = step32(z, sp, c32)
            x = mul(x, x) + c
        assert np.all(norm(x[:4] - z[:4])[live] <= er[live] * (1 + 1e-12))
        assert np.all(norm(x[4:] - z[4:])[live] <= ed[live] * (1 + 1e-12))


@pytest.mark.parametrize("seed", range(4))
@pytest.mark.parametrize("half", [0.002, 0.02, 0.2])
def test_box_bound(seed, half):
    rng = np.random.default_rng(seed)
    n, pts = 200, 64
    c = rng.uniform(-0.8, 0.8, (8, n, 1))
    z = rng.uniform(-1.5, 1.5, (8, n, 1))
    basis = np.stack([np.linalg.qr(rng.standard_normal((8, 3)))[0].T for _ in range(n)])
    g = [half * rng.uniform(0.1, 1, (n,)) * basis[:, a].T for a in range(3)]
    g = [v[:, :, None] for v in g]
    u = rng.uniform(-1, 1, (3, n, pts))
    u[:, :, :8] = np.sign(u[:, :, :8])  # corners too
    x = z + sum(u[a] * g[a] for a in range(3))
    er = np.zeros((n, 1))
    ed = np.zeros((n, 1))
    for _ in range(6):
        gr, gd = sum(norm(v[:4]) for v in g), sum(norm(v[4:]) for v in g)
        zr, zd = norm(z[:4]), norm(z[4:])
        er, ed = (2 * zr * er + (gr + er) ** 2, 2 * (zr * ed + zd * er) + 2 * (gr + er) * (gd + ed))
        g = [mul(z, v) + mul(v, z) for v in g]
        z = mul(z, z) + c
        x = mul(x, x) + c
        live = (norm(z[:4]) + norm(z[4:]) < 8) & (er < 1) & (ed < 1)
        e = x - z - sum(u[a] * g[a] for a in range(3))
        scale = 1 + norm(x[:4]) ** 2 + norm(x[4:]) ** 2
        assert np.all((norm(e[:4]) <= er + 1e-12 * scale) | ~live)
        assert np.all((norm(e[4:]) <= ed + 1e-12 * scale) | ~live)
