"""The float test that spares the double-precision fallback most of its triangles rejects none that the
double test accepts: emulated in float32 on rays aimed at points inside, on and just off triangles of all
shapes (slivers and needles among them), from origins up to several scene sizes away."""
import numpy as np

f = np.float32


def cross(a, b):
    return np.array([f(a[1] * b[2]) - f(a[2] * b[1]), f(a[2] * b[0]) - f(a[0] * b[2]), f(a[0] * b[1]) - f(a[1] * b[0])], f)


def dot(a, b):
    return f(f(f(a[0] * b[0]) + f(a[1] * b[1])) + f(a[2] * b[2]))


def rejected(o, d, v):
    of, df = o.astype(f), d.astype(f)
    A = v[0]
    e1, e2 = (v[1] - v[0]).astype(f), (v[2] - v[0]).astype(f)
    pv, tv = cross(df, e2), (of - A).astype(f)
    qv = cross(tv, e1)
    det = dot(e1, pv)
    sg = f(1) if det > 0 else f(-1)
    un, vn = f(sg * dot(tv, pv)), f(sg * dot(df, qv))
    m1, m2 = np.abs(e1).max(), np.abs(e2).max()
    mo = f(np.abs(of).max() + np.abs(A).max())
    k = f(2.0 ** -16)
    eu, ev, ed = f(k * mo * m2), f(k * mo * m1), f(k * m1 * m2)
    return abs(det) > ed and (un < -eu or vn < -ev or f(un + vn) > f(f(abs(det) + eu) + f(ev + ed)))


def inside(o, d, v):
    v = v.astype(np.float64)
    e1, e2 = v[1] - v[0], v[2] - v[0]
    p = np.cross(d, e2)
    det = e1 @ p
    if det == 0.0:
        return False
    t = o - v[0]
    u = (t @ p) / det
    q = np.cross(t, e1)
    w = (d @ q) / det
    return u >= 0.0 and w >= 0.0 and u + w <= 1.0


def test_prefilter_keeps_every_hit():
    rng = np.random.default_rng(5)
    hits = kept_far = 0
    with np.errstate(over="ignore"):
        for i in range(20000):
            M = 10.0 ** rng.uniform(-3, 0)
            size = M * 10.0 ** rng.uniform(-4, 0)
            c = rng.uniform(-M, M, 3)
            v = c + rng.uniform(-size, size, (3, 3))
            if i % 4 == 1:
                v[2] = v[0] + (v[1] - v[0]) * rng.uniform(0.2, 0.8) + rng.normal(size=3) * size * 10.0 ** rng.uniform(-5, -1)
            v = v.astype(f)
            a, b = rng.uniform(0, 1, 2)
            if a + b > 1:
                a, b = 1 - a, 1 - b
            if i % 3 == 0:
                a = rng.choice([0.0, 1e-9, 1e-7])
            X = v[0].astype(float) * (1 - a - b) + v[1].astype(float) * a + v[2].astype(float) * b
            d = rng.normal(size=3)
            if i % 5 == 0:                                       # nearly in the triangle's plane
                n = np.cross((v[1] - v[0]).astype(float), (v[2] - v[0]).astype(float))
                n /= np.linalg.norm(n) + 1e-300
                d -= n * (d @ n) * (1 - 10.0 ** rng.uniform(-6, -2))
            d /= np.linalg.norm(d)
            o = X - d * M * 10.0 ** rng.uniform(-2, 0.7)
            if inside(o, d, v):
                hits += 1
                assert not rejected(o, d, v), i
            kept_far += not rejected(o + np.cross(d, rng.normal(size=3)) * 20 * size, d, v)
    assert hits > 8000
