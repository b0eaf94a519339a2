"""Mixed precision: the gap of spheres that touch to a billionth of their radii,
read off the contact force, against the double-float sums it is to be taken
from, each renormalised, restated in numpy's FP32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

f4, f8 = np.float32, np.float64


def two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def fast_two_sum(a, b):
    s = a + b
    return s, b - (s - a)


def add(a, b):
    s, t = two_sum(a[0], b[0]), two_sum(a[1], b[1])
    s = fast_two_sum(s[0], s[1] + t[0])
    return fast_two_sum(s[0], s[1] + t[1])


def add_loose(a, b):
    """A sum without the second renormalisation (what the gap is not taken by)."""
    s = two_sum(a[0], b[0])
    return fast_two_sum(s[0], s[1] + (a[1] + b[1]))


def fma(a, b, c):
    return (a.astype(np.longdouble) * b + c).astype(f4)   # (the product is exact)


def sqr(a):
    p = a[0] * a[0]
    return fast_two_sum(p, fma(f4(2) * a[0], a[1], fma(a[0], a[0], -p)))


def split(v):
    hi = v.astype(f4)
    return hi, (v - hi).astype(f4)


def touching_pairs(m, seed):
    """m^3 isolated pairs at random places, overlapping by 0.7e-9 to 1e-9 of a_i + a_j."""
    rng = np.random.default_rng(seed)
    n = m ** 3
    c = 8.0 * (np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij")).reshape(3, -1) + 0.5)
    c += rng.uniform(-1.5, 1.5, size=(3, n))
    a = rng.uniform(1.0, 1.4, size=(2, n))
    S = a[0] + a[1]
    v = rng.standard_normal((3, n))
    v *= S * (1.0 - rng.uniform(0.7e-9, 1.0e-9, size=n)) / np.linalg.norm(v, axis=0)
    L = 8.0 * m
    x = np.stack([(c - 0.5 * v) % L, (c + 0.5 * v) % L])      # (2, 3, n)
    return x, a, L


def gap(x, a, L, ncell, plus):
    """The gap of each pair as the kernel takes it, and its exact value."""
    n = x.shape[2]
    cs = f8(L) / ncell
    csh = f4(cs)
    csl = f4(cs - f8(csh))
    D, exact = [], []
    for d in range(3):
        k = np.minimum(np.floor(x[:, d] / cs), ncell - 1)
        loc = (x[:, d].astype(np.longdouble) - k * np.longdouble(cs)).astype(f8)
        (ih, jh), (il, jl) = split(loc)
        w = k[1] - k[0]
        w -= ncell * np.round(w / ncell)
        wf = w.astype(f4)
        p = wf * csh
        shift = (p, fma(wf, csl, fma(wf, csh, -p)))
        low = (jl - il, np.zeros(n, f4))
        r = add(two_sum(jh, -ih), add(shift, low)) if plus is add else plus(two_sum(jh, -ih), (p, shift[1] + low[0]))
        D.append(r)
        e = x[1, d].astype(np.longdouble) - x[0, d]
        exact.append(e - L * np.round(e / L))
    S = plus(split(a[0]), split(a[1]))
    q = sqr(S)
    num = plus(plus(plus(sqr(D[0]), sqr(D[1])), sqr(D[2])), (-q[0], -q[1]))
    num = num[0].astype(f8) + num[1]
    Sx = a[0].astype(np.longdouble) + a[1]
    rr = np.sqrt(exact[0] ** 2 + exact[1] ** 2 + exact[2] ** 2)
    return (num / (2.0 * (a[0] + a[1]))).astype(f8), (rr - Sx).astype(f8)


# |F| = k_n |d| |n| in FP32: the rounding of the numerator, the reciprocal root
# (2 ulp) in r + S and n, the quotient (2 ulp), three products
TOL = 2.5 * 2.0 ** -22 + 5 * 2.0 ** -24


def test_gap_of_touching_spheres():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2108_01013_gb300 as dss
    dss.build()
    x, a, L = touching_pairs(20, 3)
    X, A = np.concatenate([x[0], x[1]], axis=1), np.concatenate([a[0], a[1]])
    z = np.zeros_like(X)
    p = dss.default_params(precision="mixed", kn=1.0, shear_rate=0.0, dt=1e-6)
    s = dss.Suspension(X, A, [L] * 3, p, u=z, w=z, alpha_lin=z, alpha_ang=z)
    nc = s.counters()["ncell"]
    assert nc[0] == nc[1] == nc[2]
    F, _ = s.forces()
    F = F.cpu().numpy()
    s.close()
    n = x.shape[2]
    np.testing.assert_array_equal(F[:, :n], -F[:, n:])
    want, _ = gap(x, a, L, nc[0], add)
    got = -np.sqrt((F[:, :n] ** 2).sum(0))
    assert np.abs(got / want - 1.0).max() <= TOL
