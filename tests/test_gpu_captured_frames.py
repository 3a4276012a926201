"""Captured frames of the trace on a GB300.  A shape is launched directly at its first frame, captured at its second
and replayed from then on, so every shape here is traced at least three times."""
import numpy as np
import pytest

from paper_2606_14173_gb300 import scenes as S
from tests.parity import assert_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hpt_mod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_14173_gb300 import build, hpt
    build.build()
    return hpt


def test_a_captured_frame_serves_scenes_of_its_depth_only(hpt_mod, oracle_mod):
    """A shallow scene's frame is captured (its traversal stacks are short), then a deep scene is traced with the same
    launch shape into the same buffer, three times, and the shallow one again: the frames keep apart."""
    ctx = hpt_mod.Context(0)
    try:
        scenes = [S.config0_scene(), S.config1_scene()]
        r = S.config1_render(W=40, H=32, spp=4, max_depth=2, K=1)
        out = hpt_mod.alloc_output(r)
        ids = [ctx.upload_scene(s) for s in scenes]
        assert ctx.scene_info(ids[0])["depth"] + 4 < ctx.scene_info(ids[1])["depth"]
        refs = [oracle_mod.Oracle(s).trace_full(r) for s in scenes]
        for k in (0, 0, 0, 1, 1, 1, 0, 1, 0):
            out.zero_()
            ctx.trace(ids[k], r, out)
            ctx.sync()
            assert_parity(out.cpu().numpy(), refs[k], f"scene {k}")
    finally:
        ctx.close()


def test_a_captured_frame_serves_far_and_near_poses_apart(hpt_mod):
    """A far pose launches a kernel that a near one does not: neither replays the other's frame."""
    direct, graphed = hpt_mod.Context(0, graphs=False), hpt_mod.Context(0)
    try:
        sc = S.config1_scene()
        sd, sg = direct.upload_scene(sc), graphed.upload_scene(sc)
        rs = [S.config1_render(W=48, H=32, spp=4, K=2, T=S.pose_T(0.0, 0.0, dz)) for dz in (0.0, -2.0)]
        refs = []
        for r in rs:
            out = hpt_mod.alloc_output(r)
            direct.trace(sd, r, out)
            direct.sync()
            refs.append(out.cpu().numpy())
        assert all(np.abs(x).max() > 0 for x in refs)
        for k in (0, 0, 0, 1, 1, 1, 0, 1):
            out = hpt_mod.alloc_output(rs[k])
            graphed.trace(sg, rs[k], out)
            graphed.sync()
            assert np.array_equal(out.cpu().numpy(), refs[k]), k
    finally:
        direct.close()
        graphed.close()


@pytest.mark.parametrize("paths,cases", [(65536, ((203, 117, 4, 7, 1), (320, 180, 8, 8, 2))),
                                         (4096, ((643, 21, 2, 3, 4), (203, 117, 1, 5, 5)))])
def test_host_rows_equal_the_captured_device_frames(hpt_mod, monkeypatch, paths, cases):
    """The rows that hpt_trace_host copies wave by wave equal the device trace's, direct, captured and replayed, with
    waves that end inside tiles and tile rows."""
    import torch
    monkeypatch.setenv("HPT_WAVE_PATHS", str(paths))
    ctx = hpt_mod.Context(0)
    try:
        sid = ctx.upload_scene(S.config1_scene())
        for W, H, K, spp, seed in cases:
            r = S.config1_render(W=W, H=H, spp=spp, K=K, seed=seed, max_depth=2)
            host = torch.empty(r.out_shape(), dtype=torch.complex64, pin_memory=True).numpy()
            host[...] = np.nan
            ctx.trace_host(sid, r, host)
            for _ in range(4):
                out = hpt_mod.alloc_output(r)
                ctx.trace(sid, r, out)
                ctx.sync()
                assert np.array_equal(out.cpu().numpy(), host), (W, H, K, spp)
    finally:
        ctx.close()
