"""The boxes of the BVH reach every ray that meets them, wherever it starts: the scene's box code and the
kernels' box test, compiled with the host compiler, with reciprocals off by up to the 2 ulp of the device's
approximate division, origins from inside the scene to 1e5 times its largest coordinate away (where first rays
start near the geometry instead), scenes flat along an axis, and grids that leave out a few huge triangles (whose boxes then reach to infinity).  The rays go
through points on faces, edges and corners of boxes, so they graze them; the scene's padding and the grid's
rounding are all the slack there is."""
import ctypes as C

import numpy as np
import pytest

from paper_2606_14173_gb300 import scenes as S
from tests.native import load

f32 = np.float32
P = C.POINTER(C.c_float)


def _p(a):
    assert a.dtype == f32 and a.flags.c_contiguous
    return a.ctypes.data_as(P)


def _missed(lib, coder, far, lo, hi, o, d, inv):
    n = len(lo)
    tn, tf = np.empty(n, f32), np.empty(n, f32)
    lib.box_test.argtypes = [C.c_void_p, C.c_int, C.c_int, P, P, P, P, P, P, P]
    assert lib.box_test(coder, far, n, _p(lo), _p(hi), _p(o), _p(d), _p(inv), _p(tn), _p(tf)) == 0   # the empty child
    return int((~(tn <= tf)).sum())


def _near(lib, coder, o):
    lib.coder_near.argtypes = [C.c_void_p, P, P]
    return bool(lib.coder_near(coder, _p(np.ascontiguousarray(o.min(0))), _p(np.ascontiguousarray(o.max(0)))))


def _boxes(rng, kind):
    """Boxes of a scene inside a cube of half side M (but for the huge ones)."""
    M = 10.0 ** rng.uniform(-3, 0)
    ext = M * 10.0 ** rng.uniform(-2, 0, 3)
    if kind == "flat":
        ext[rng.integers(3)] = 0.0
    mid = rng.uniform(-1, 1, 3) * np.maximum(M - ext / 2, 0)
    n = 64
    half = ext * 10.0 ** rng.uniform(-5, -0.5, (n, 1)) * rng.uniform(0, 0.5, (n, 3))
    ctr = mid + rng.uniform(-0.5, 0.5, (n, 3)) * ext
    lo, hi = (ctr - half).astype(f32), (ctr + half).astype(f32)
    if kind == "huge":                # a few huge triangles beside them, up to 3000 times as wide
        for _ in range(3):
            a, b = np.sort(rng.uniform(-1, 1, (2, 3)), 0) * M * 10.0 ** rng.uniform(2, 3.5)
            lo, hi = np.vstack([lo, a.astype(f32)]), np.vstack([hi, b.astype(f32)])
    return lo, np.maximum(lo, hi), M


def _coder(lib, lo, hi, wide=0):
    lib.coder_new.restype = C.c_void_p
    lib.coder_new.argtypes = [C.c_int, P, P, C.c_float, C.c_int]
    lib.coder_free.argtypes = lib.coder_wide.argtypes = [C.c_void_p]
    return lib.coder_new(len(lo), _p(lo), _p(hi), float(max(np.abs(lo).max(), np.abs(hi).max())), wide)


def _grazing_rays(rng, lo, hi, dist, X=None, d=None):
    """Float rays through points X (on the boxes' faces, edges and corners), and the boxes grown by what rounding the
    ray's origin moved it past them (the geometry that a float ray meets is where that ray goes)."""
    n = len(lo)
    if X is None:
        X = rng.uniform(lo.astype(float), hi.astype(float))
        for i in range(n):
            for k in rng.choice(3, size=rng.integers(1, 4), replace=False):
                X[i, k] = lo[i, k] if rng.random() < 0.5 else hi[i, k]
        d = rng.normal(size=(n, 3))
        d[np.arange(1, n, 4), rng.integers(3)] = 0.0
        d[np.arange(2, n, 4), rng.integers(3)] *= 1e-9
    d /= np.linalg.norm(d, axis=1)[:, None]
    o = (X - dist[:, None] * d).astype(f32)
    d = d.astype(f32)
    of, df = o.astype(np.longdouble), d.astype(np.longdouble)
    t = np.maximum(((X - of) * df).sum(1) / (df * df).sum(1), 0)
    Y = of + t[:, None] * df
    glo = np.minimum(lo, Y.astype(f32))
    ghi = np.maximum(hi, Y.astype(f32))
    glo = np.where(glo > Y, np.nextafter(glo, f32(-np.inf)), glo).astype(f32)
    ghi = np.where(ghi < Y, np.nextafter(ghi, f32(np.inf)), ghi).astype(f32)
    return glo, ghi, o, d


def _reciprocals(rng, d):
    """1 / d off by up to 2 ulp, or 1e20 as the traversal takes it where d vanishes."""
    inv = (f32(1) / np.where(d == 0, f32(1), d)).astype(f32)
    for _ in range(2):
        s = rng.integers(-1, 2, d.shape)
        inv = np.where(s > 0, np.nextafter(inv, f32(np.inf)), np.where(s < 0, np.nextafter(inv, f32(-np.inf)), inv))
    return np.where(np.abs(d) > f32(1e-20), inv, np.copysign(f32(1e20), d)).astype(f32)


@pytest.mark.parametrize("wide", [0, 1])
@pytest.mark.parametrize("kind", ["plain", "flat", "huge"])
@pytest.mark.parametrize("far", [2.0, 40.0, 300.0, 1e5])
def test_no_grazing_ray_misses_its_box(kind, far, wide):
    lib = load("boxes")
    rng = np.random.default_rng([ord(kind[0]), int(far)])
    missed, n_far = 0, 0
    for _ in range(150):
        lo, hi, M = _boxes(rng, kind)
        dist = M * (rng.uniform(0, far, len(lo)) if far <= 300 else 10.0 ** rng.uniform(2, 5, len(lo)))
        lo, hi, o, d = _grazing_rays(rng, lo, hi, dist)
        coder = _coder(lib, lo, hi, wide)
        use_far = not _near(lib, coder, o)          # as the host decides for a job's origins
        n_far += use_far
        missed += _missed(lib, coder, use_far, lo, hi, o, d, _reciprocals(rng, d))
        lib.coder_free(coder)
    assert missed == 0
    assert kind == "huge" or n_far > 0
    assert far > 2.0 or wide or n_far < 150


@pytest.mark.parametrize("wide", [0, 1])
@pytest.mark.parametrize("kind", ["plain", "flat", "huge"])
def test_rays_from_the_geometry_need_no_reach(kind, wide):
    """Rays that leave a point of the geometry (every ray but a job's first) never miss."""
    lib = load("boxes")
    rng = np.random.default_rng([ord(kind[0]), 3])
    missed = 0
    for _ in range(150):
        lo, hi, _ = _boxes(rng, kind)
        o = rng.uniform(lo.astype(float), hi.astype(float))[rng.permutation(len(lo))]
        X = rng.uniform(lo.astype(float), hi.astype(float))
        k = rng.integers(3, size=len(lo))
        X[np.arange(len(lo)), k] = lo[np.arange(len(lo)), k]
        lo, hi, o, d = _grazing_rays(rng, lo, hi, np.linalg.norm(X - o, axis=1), X, X - o)
        coder = _coder(lib, np.vstack([lo, o]), np.vstack([hi, o]), wide)
        missed += _missed(lib, coder, 0, lo, hi, o, d, _reciprocals(rng, d))
        lib.coder_free(coder)
    assert missed == 0


def test_ordinary_origins_are_near():
    """Origins within 0.6 times the scene's largest coordinate of the scene's origin, and a hologram plane at z = 0
    before scenes of the seeded generators' proportions."""
    lib = load("boxes")
    rng = np.random.default_rng(7)
    for kind in ("plain", "flat", "huge"):
        for _ in range(40):
            lo, hi, _ = _boxes(rng, kind)
            coder = _coder(lib, lo, hi, -1)
            m = max(np.abs(lo).max(), np.abs(hi).max())
            assert _near(lib, coder, rng.uniform(-1, 1, lo.shape).astype(f32) * f32(0.6) * m)
            lib.coder_free(coder)
    for make in (S.config0_scene, S.config1_scene, S.config3_scene):
        v = make().verts.astype(f32)
        t = v[make().tris.reshape(-1)].reshape(-1, 3, 3)
        coder = _coder(lib, np.ascontiguousarray(t.min(1)), np.ascontiguousarray(t.max(1)), -1)
        assert not lib.coder_wide(coder)                          # the grid is fine enough for them
        half = np.array([7.2e-3, 4.1e-3, 0.0], f32)              # 3840 x 2160 at 3.74 um
        for shift in (0.0, 0.03, -0.03):
            assert _near(lib, coder, np.stack([-half, half]).astype(f32) + np.array([5e-3, -5e-3, shift], f32))
        lib.coder_free(coder)


@pytest.mark.parametrize("apart,wide", [(0.0, 0), (0.02, 0), (0.5, 1), (3.0, 1)])
def test_scenes_too_large_for_their_triangles_are_wide(apart, wide):
    """Two spheres of 20480 triangles with edges of some 26 um: together on the grid, metres apart with float boxes."""
    lib = load("boxes")
    b = S._Builder("two")
    m = b.material(S.LAMBERT, albedo=(0.5, 0.5, 0.5))
    b.sphere(np.array([0.0, 0.0, 8e-3]), 0.8e-3, 5, m)
    b.sphere(np.array([2e-3 + apart, 0.7 * apart, 8e-3 + apart]), 0.8e-3, 5, m)
    s = b.build()
    t = s.verts.astype(f32)[s.tris.reshape(-1)].reshape(-1, 3, 3)
    coder = _coder(lib, np.ascontiguousarray(t.min(1)), np.ascontiguousarray(t.max(1)), -1)
    assert lib.coder_wide(coder) == wide
    lib.coder_free(coder)
