"""Scenes whose extents are hard for a 65536-step box grid, against the oracle: flat along an axis, tiny
triangles beside a huge one, a scene far from the origin for its size, and triangles whose sizes and
places fall off geometrically (the surface-area splits then peel one triangle at a time, and the
builder has to bound the depth); and two scenes of different depth traced through one output buffer."""
import numpy as np
import pytest

from paper_2606_14173_gb300 import scenes as S
from tests.parity import assert_parity

pytestmark = pytest.mark.gpu
MM = 1e-3


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_14173_gb300 import build, hpt
    build.build()
    c = hpt.Context(0)
    yield c
    c.close()


def _tri_scene(name, tris):
    """Emissive triangles ([n][3][3], metres), the normals facing the SLM (-z)."""
    b = S._Builder(name)
    m = b.material(S.LAMBERT, albedo=(0.0, 0.0, 0.0), Le=(1.0, 0.7, 0.4))
    V = np.asarray(tris, np.float64)
    n = np.cross(V[:, 1] - V[:, 0], V[:, 2] - V[:, 0])
    flip = n[:, 2] > 0
    V[flip] = V[flip][:, ::-1]
    b.mesh(V.reshape(-1, 3), np.tile([0.0, 0.0, -1.0], (3 * len(V), 1)), np.zeros((3 * len(V), 2)),
           np.arange(3 * len(V)).reshape(-1, 3), m)
    return b.build()


def _cells(rng, n, half, z, size, zs=0.0):
    c = np.stack([rng.uniform(-half, half, n), rng.uniform(-half, half, n), z + rng.uniform(-1, 1, n) * zs], 1)
    d = rng.uniform(-size, size, (n, 3, 3))
    d[..., 2] *= 0.0 if zs == 0.0 else 0.3
    return c[:, None, :] + d


def _flat(rng):
    return _cells(rng, 400, 0.6 * MM, 4 * MM, 0.08 * MM)


def _huge_and_tiny(rng):
    t = _cells(rng, 600, 0.25 * MM, 4 * MM, 0.004 * MM, 0.05 * MM)
    return np.concatenate([t, [[[-900 * MM, -900 * MM, 9 * MM], [1800 * MM, -900 * MM, 9 * MM], [-900 * MM, 1800 * MM, 9 * MM]]]])


def _far(rng):
    return _cells(rng, 300, 6 * MM, 900 * MM, 1.0 * MM, 2 * MM)


def _geometric(rng):
    t = []
    for i in range(400):
        s = 0.5 * MM * 0.95 ** i + 1e-7
        x = 0.6 * MM * 0.97 ** i
        t.append([[x, -s, 4 * MM + x], [x + 0.2 * s, s, 4 * MM + x], [x - 0.2 * s, s, 4 * MM + x]])
    return np.array(t)


@pytest.mark.parametrize("make", [_flat, _huge_and_tiny, _far, _geometric])
def test_scene_extents(ctx, oracle_mod, make):
    from paper_2606_14173_gb300 import hpt
    sc = _tri_scene(make.__name__, make(np.random.default_rng(3)))
    sid = ctx.upload_scene(sc)
    assert ctx.scene_info(sid)["depth"] <= 31
    for prec in (hpt.PREC_FP64, hpt.PREC_DF32):
        r = S.Render(W=48, H=40, pitch=8e-6, lambdas=(638e-9, 450e-9), channels=(0, 2), spp=8, max_depth=1, K=2,
                     phase_mode=S.PHASE_ZERO)
        out = hpt.alloc_output(r)
        ctx.trace(sid, r, out, precision=prec)
        ctx.sync()
        ref = oracle_mod.Oracle(sc).trace_full(r)
        assert np.abs(ref).max() > 0
        assert_parity(out.cpu().numpy(), ref, f"{make.__name__} prec {prec}")
    ctx.release_scene(sid)


def test_scenes_of_different_depth_share_an_output(ctx, oracle_mod):
    """One output buffer and launch shape for a shallow and then a deep tree (and back): the captured
    frame of the first must not serve the second with its shorter traversal stack."""
    from paper_2606_14173_gb300 import hpt
    scenes = [S.config0_scene(), S.config1_scene()]
    r = S.config1_render(W=40, H=32, spp=4, max_depth=2, K=1)
    out = hpt.alloc_output(r)
    ids = [ctx.upload_scene(s) for s in scenes]
    refs = [oracle_mod.Oracle(s).trace_full(r) for s in scenes]
    for k in (0, 1, 0, 1):
        ctx.trace(ids[k], r, out)
        ctx.sync()
        assert_parity(out.cpu().numpy(), refs[k], f"scene {k}")
    for i in ids:
        ctx.release_scene(i)
