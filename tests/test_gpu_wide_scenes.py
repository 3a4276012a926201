"""Scenes with float boxes (wide scenes) on a GB300: which boxes a tree has changes the work and no field, so every
entry point gives the grid's bits; a scene that is wide by itself meets the oracle."""
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


def _clusters(apart, level=4, points=False):
    """Spheres of every material under a light, and the same spheres 'apart' metres away."""
    rng = np.random.default_rng(4)
    b = S._Builder("clusters")
    b.rect_light(np.array([-3 * MM, 6 * MM, 4 * MM]), np.array([6 * MM, 0, 0]), np.array([0, 0, 6 * MM]), np.array([20.0, 20.0, 20.0]))
    mats = [b.material(S.LAMBERT, albedo=(0.7, 0.6, 0.5)), b.material(S.GGX, albedo=(0.7, 0.7, 0.7), rough=0.3),
            b.material(S.MIRROR, albedo=(0.8, 0.8, 0.8)), b.material(S.DIELECTRIC, ior=1.5)]
    for i in range(8):
        c = np.array([(i % 4 - 1.5) * 1.0, (i // 4 - 0.5) * 1.2, 8.0 + rng.uniform(-1, 1)]) * MM
        b.sphere(c, 0.45 * MM, level, mats[i % 4])
        b.sphere(c + apart * np.array([1.0, 0.7, 1.0]), 0.45 * MM, level, mats[i % 4])
    sc = b.build()
    if points:
        sc.points = np.array([[0.2 * MM, 0.1 * MM, 11 * MM, 1.0], [-1.1 * MM, 0.4 * MM, 6 * MM, 0.5]], np.float64)
    return sc


def _upload(ctx, monkeypatch, sc, boxes):
    monkeypatch.setenv("HPT_BOXES", boxes)
    sid = ctx.upload_scene(sc)
    monkeypatch.delenv("HPT_BOXES")
    return sid


def _is_wide(ctx, sid, sc, monkeypatch):
    """A wide scene's nodes take twice the bytes."""
    grid = _upload(ctx, monkeypatch, sc, "grid")
    more = ctx.scene_info(sid)["device_bytes"] - ctx.scene_info(grid)["device_bytes"]
    ctx.release_scene(grid)
    return more > 0


def test_a_scene_of_far_groups_is_wide_and_meets_the_oracle(ctx, oracle_mod, monkeypatch):
    from paper_2606_14173_gb300 import hpt
    sc = _clusters(3.0)
    sid = ctx.upload_scene(sc)
    assert _is_wide(ctx, sid, sc, monkeypatch)
    r = S.config1_render(W=64, H=48, spp=8, K=2)
    ref = oracle_mod.Oracle(sc).trace_full(r)
    assert np.abs(ref).max() > 0
    for prec in (hpt.PREC_FP64, hpt.PREC_DF32):
        out = hpt.alloc_output(r)
        ctx.trace(sid, r, out, precision=prec)
        ctx.sync()
        assert_parity(out.cpu().numpy(), ref, f"far groups prec {prec}")
    ctx.release_scene(sid)


def test_the_benchmark_scenes_are_not_wide(ctx, monkeypatch):
    for make in (S.config0_scene, S.config1_scene, S.config3_scene):
        sc = make()
        sid = ctx.upload_scene(sc)
        assert not _is_wide(ctx, sid, sc, monkeypatch)
        ctx.release_scene(sid)


@pytest.mark.parametrize("name,make,render,kw", [
    ("quads", S.config0_scene, S.config0_render, dict(W=203, H=117, spp=8, K=2)),
    ("spheres", S.config1_scene, S.config1_render, dict(W=203, H=117, spp=8, K=4)),
    ("spheres posed", S.config1_scene, S.config1_render, dict(W=96, H=64, spp=8, K=1, T=S.pose_T(1e-3, -1e-3, -8e-3))),
    ("spheres far", S.config1_scene, S.config1_render, dict(W=96, H=64, spp=8, K=1, T=S.pose_T(0.0, 0.0, -2.0))),
    ("slabs", S.config3_scene, S.config3_render, dict(W=160, H=90, spp=8, K=2)),
    ("groups", lambda: _clusters(0.3, points=True), S.config1_render, dict(W=96, H=64, spp=8, K=2))])
def test_fields_do_not_depend_on_the_boxes(ctx, monkeypatch, name, make, render, kw):
    import torch
    from paper_2606_14173_gb300 import hpt
    sc, r = make(), render(**kw)
    ids = {b: _upload(ctx, monkeypatch, sc, b) for b in ("grid", "wide")}
    for prec in (hpt.PREC_DF32, hpt.PREC_FP64):
        ref = hpt.alloc_output(r)
        ctx.trace(ids["grid"], r, ref, precision=prec)
        ctx.sync()
        assert ref.abs().max() > 0
        def same(f, what):
            out = hpt.alloc_output(r)
            out.zero_()
            f(out)
            ctx.sync()
            assert torch.equal(torch.view_as_real(out), torch.view_as_real(ref)), (name, prec, what)
        for k in range(3):                     # direct, captured, replayed
            same(lambda o: ctx.trace(ids["wide"], r, o, precision=prec), k)
        same(lambda o: ctx.trace_timed(ids["wide"], r, o, precision=prec), "timed")
        same(lambda o: ctx.trace_fixed_scratch(ids["wide"], r, o, precision=prec), "fixed scratch")
        out = hpt.alloc_output(r)
        c = [ctx.trace_counters(ids[b], r, out, precision=prec) for b in ("grid", "wide")]
        assert c[0]["rays"] == c[1]["rays"] and c[0]["bounces"] == c[1]["bounces"] and c[0]["shadow_rays"] == c[1]["shadow_rays"]
    lo, hi = sc.verts.min(0), sc.verts.max(0)
    lo, hi = np.maximum(lo, -9 * MM), np.minimum(hi, 30 * MM)
    bakes = [ctx.cache_bake(ids[b], 12, lo, hi, 8, 3) for b in ("grid", "wide")]
    ctx.sync()
    assert torch.equal(bakes[0], bakes[1])
    for i in ids.values():
        ctx.release_scene(i)


def test_wide_and_grid_scenes_share_waves(ctx, monkeypatch):
    """Requests of both kinds of scene in the same serving waves."""
    import torch
    from paper_2606_14173_gb300 import hpt
    sc = [S.config1_scene(), _clusters(3.0), S.config0_scene()]
    ids = [_upload(ctx, monkeypatch, s, b) for s, b in zip(sc, ("grid", "wide", "wide"))]
    rs = [S.config1_render(W=96, H=64, spp=8, K=2, seed=s) for s in (1, 2, 3)]
    refs, outs = [], []
    for i, r in zip(ids, rs):
        out = hpt.alloc_output(r)
        ctx.trace(i, r, out)
        ctx.sync()
        refs.append(out)
        outs.append(hpt.alloc_output(r))
    for _ in range(2):
        reqs = [ctx.submit(i, r, o) for i, r, o in zip(ids, rs, outs)]
        for q in reqs:
            ctx.wait(q, 60000)
        for o, ref in zip(outs, refs):
            assert torch.equal(torch.view_as_real(o), torch.view_as_real(ref))
            o.zero_()
    for i in ids:
        ctx.release_scene(i)
