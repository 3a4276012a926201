"""Small objects seen from a hologram plane posed tens of their sizes away, against the oracle: a ray that
grazes a node's box from afar must still enter it."""
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


def _plate(half, n):
    """A plate of n x n cells (2 n^2 triangles) of three emissive materials across the z axis, at the origin."""
    b = S._Builder("plate")
    mats = [b.material(S.LAMBERT, albedo=(0.0, 0.0, 0.0), Le=e) for e in ((1.0, 0.6, 0.3), (0.4, 1.0, 0.5), (0.7, 0.3, 1.0))]
    x = np.linspace(-half, half, n + 1)
    for i in range(n):
        for j in range(n):
            b.quad(np.array([x[i], x[j], 0.0]), np.array([0.0, x[j + 1] - x[j], 0.0]),
                   np.array([x[i + 1] - x[i], 0.0, 0.0]), mats[(i + 2 * j) % 3])
    return b.build()


@pytest.mark.parametrize("half,n,dist", [(5 * MM, 40, 0.5), (1 * MM, 30, 0.04), (2 * MM, 20, 0.6)])
def test_far_pose(ctx, oracle_mod, half, n, dist):
    from paper_2606_14173_gb300 import hpt
    sc = _plate(half, n)
    sid = ctx.upload_scene(sc)
    r = S.Render(W=64, H=48, pitch=16e-6, lambdas=(638e-9, 450e-9), channels=(0, 2), spp=16, max_depth=1, K=1,
                 phase_mode=S.PHASE_ZERO, T=S.pose_T(0.0, 0.0, -dist))
    ref = oracle_mod.Oracle(sc).trace_full(r)
    assert np.abs(ref).max() > 0
    for prec in (hpt.PREC_FP64, hpt.PREC_DF32):
        out = hpt.alloc_output(r)
        ctx.trace(sid, r, out, precision=prec)
        ctx.sync()
        assert_parity(out.cpu().numpy(), ref, f"{half} {dist} prec {prec}")
    ctx.release_scene(sid)


def test_bake_of_far_cells(ctx, oracle_mod):
    """Cells 5 to 8 scene sizes away, against the oracle with the bake's bar: cell-channels beyond 1e-4 are float32-
    sensitive ones, but for at most 0.1 %."""
    sc = S.config1_scene()
    sid = ctx.upload_scene(sc)
    lo, hi = [-20 * MM, 150 * MM, 0 * MM], [20 * MM, 200 * MM, 40 * MM]
    res, spp, depth = 10, 256, 2
    got = ctx.cache_bake(sid, res, lo, hi, spp, depth, seed=11)
    ctx.sync()
    got = got.cpu().numpy().reshape(-1, 3).astype(np.float64)
    lo32, hi32 = np.float32(lo).astype(np.float64), np.float32(hi).astype(np.float64)
    orc = oracle_mod.Oracle(sc)
    ref = orc.bake(res, lo32, hi32, spp, depth, seed=11)
    assert (ref > 0).mean() > 0.5
    tol = 1e-4 * np.maximum(np.abs(ref), 1e-3 * np.abs(ref).mean())
    bad = np.abs(got - ref) > tol
    cells = np.nonzero(bad.any(axis=1))[0]
    sv = np.zeros_like(ref)
    if len(cells):
        sv[cells] = orc.bake(res, lo32, hi32, spp, depth, seed=11, cells=cells, with_sens=True)[1]
    explained = bad & (sv >= tol) & (np.abs(got - ref) <= tol + sv)
    assert int((bad & ~explained).sum()) <= 1e-3 * bad.size, (int(bad.sum()), int((bad & ~explained).sum()))
    ctx.release_scene(sid)
