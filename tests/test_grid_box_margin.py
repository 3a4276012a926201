"""The BVH's grid boxes are conservative: a node's child box is stored as a 16-bit centre and a binary16
half extent on the scene's 65536-step grid, and tested in float32 with one rounded offset per ray and
axis.  For any ray that meets a primitive's box at some t >= 0, that test must pass.  This emulates the
builder's rounding and the kernel's arithmetic (each FMA rounded once from the exact product) on boxes
from a step to the whole scene wide, points on their faces, edges and corners, axis-parallel and
nearly axis-parallel directions, scenes flat along an axis, and the widened form of the
double-precision fallback."""
import numpy as np

f32 = np.float32


def fma32(a, b, c):
    # exact product in float64; the sum's double rounding costs at most one ulp of float32 more than
    # the kernel's single one, inside the margin under test
    return (np.asarray(a, f32).astype(np.float64) * np.asarray(b, f32).astype(np.float64) + np.asarray(c, f32).astype(np.float64)).astype(f32)


def half_up(e):
    v = np.asarray(e, np.float64).astype(np.float16)
    up = np.nextafter(v, np.float16(np.inf))
    return np.where(v.astype(np.float64) < e, up, v)


def grid_of(all_lo, all_hi, pad):
    lo = (all_lo - pad).astype(f32)
    step = ((all_hi.astype(np.float64) + np.float64(pad) - lo.astype(np.float64)) / 65534.0).astype(f32)
    return lo, step


def quantise(lo, hi, pad, glo, step):
    s = step.astype(np.float64)
    l = (lo.astype(np.float64) - np.float64(pad) - glo) / s - 1.0
    u = (hi.astype(np.float64) + np.float64(pad) - glo) / s + 1.0
    c = np.clip(np.floor(0.5 * (l + u) + 0.5), 0, 65535)
    return c, half_up(np.maximum(u - c, c - l)).astype(f32)


def slab(o, d, c, h, glo, step, w=None):
    of, df = o.astype(f32), d.astype(f32)
    inv = np.where(np.abs(df) > f32(1e-20), f32(1) / np.where(df == 0, f32(1), df), np.copysign(f32(1e20), df)).astype(f32)
    st = (step * inv).astype(f32)
    k = fma32(f32(-8388608.0), st, ((glo - of).astype(f32) * inv).astype(f32))
    hh = h if w is None else (h + (w / step).astype(f32)).astype(f32)
    t = fma32((c + 8388608.0).astype(f32), st, k)
    near, far = fma32(hh, -np.abs(st), t), fma32(hh, np.abs(st), t)
    return max(near.max(), f32(0)), far.min()


def _run(fallback):
    rng = np.random.default_rng(11 + fallback)
    misses = 0
    for i in range(6000):
        M = 10.0 ** rng.uniform(-3, 0)
        ext = M * 10.0 ** rng.uniform(-3, 0, 3)
        if i % 5 == 0:
            ext[rng.integers(3)] = 0.0                          # a scene flat along an axis
        mid = rng.uniform(-1, 1, 3) * np.maximum(M - ext, 0) * 0.5
        all_lo, all_hi = (mid - ext / 2).astype(f32), (mid + ext / 2).astype(f32)
        max_abs = f32(max(np.abs(all_lo).max(), np.abs(all_hi).max()))
        pad = f32(f32(2e-6) * max_abs + f32(1e-12))
        glo, step = grid_of(all_lo, all_hi, pad)
        half = ext * 10.0 ** rng.uniform(-5, 0) * rng.uniform(0, 0.5, 3)
        ctr = rng.uniform(all_lo.astype(float), all_hi.astype(float))
        lo = np.clip(ctr - half, all_lo, all_hi).astype(f32)
        hi = np.maximum(np.clip(ctr + half, all_lo, all_hi).astype(f32), lo)
        X = rng.uniform(lo.astype(float), hi.astype(float))
        for k in rng.choice(3, size=rng.integers(1, 4), replace=False):
            X[k] = float(lo[k] if rng.random() < 0.5 else hi[k])
        d = rng.normal(size=3)
        if i % 4 == 1:
            d[rng.integers(3)] = 0.0
        elif i % 4 == 2:
            d[rng.integers(3)] *= 1e-9
        d /= np.linalg.norm(d)
        dist = rng.uniform(0, 2) * float(max_abs)
        o = X - dist * d
        if not fallback:
            # the float traversal's rays are the float ones
            o = o.astype(f32).astype(np.float64)
            d = d.astype(f32).astype(np.float64)
            t = (X - o) @ d / (d @ d)
            P = o + t * d                                       # the ray's point nearest X ...
            if t < 0:
                continue
            lo = np.minimum(lo, np.floor(P / 2.0 ** -40) * 2.0 ** -40).astype(f32)   # ... is in the box
            lo = np.where(lo.astype(float) > P, np.nextafter(lo, f32(-np.inf)), lo)
            hi = np.maximum(hi, P.astype(f32))
            hi = np.where(hi.astype(float) < P, np.nextafter(hi, f32(np.inf)), hi)
            if (lo < all_lo).any() or (hi > all_hi).any():
                continue
        c, h = quantise(lo, hi, pad, glo, step)
        w = None
        if fallback:
            bound = f32(max_abs + pad)
            w = f32((f32(np.abs(o.astype(f32)).max()) + bound) * f32(2.0 ** -17))
        tn, tf = slab(o, d, c, h, glo, step, w)
        misses += not (tn <= tf)
    return misses


def test_float_traversal_box_is_conservative():
    assert _run(False) == 0


def test_fallback_box_is_conservative():
    assert _run(True) == 0
