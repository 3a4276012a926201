"""Coherent rays traced beside the incoherent shading (small waves): the same bits as the kernels one after
the other, which the per-kernel timing runs, for frames of one wave and of several, with and without delta
chains, launched directly and replayed."""
import pytest

from paper_2606_14173_gb300 import scenes as S

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("W,H,spp,depth", [(5, 3, 1, 4), (64, 48, 4, 1), (64, 48, 4, 2), (203, 117, 8, 4), (320, 200, 32, 4)])
def test_side_stream_matches_serial_kernels(ctx, W, H, spp, depth, precision):
    import torch
    from paper_2606_14173_gb300 import hpt
    sid = ctx.upload_scene(S.config1_scene())
    r = S.config1_render(W=W, H=H, spp=spp, K=2, max_depth=depth)
    ref = hpt.alloc_output(r)
    ctx.trace_timed(sid, r, ref, precision=precision)
    assert W < 64 or depth < 2 or ref.abs().max() > 0     # the area light is not seen directly
    for _ in range(3):
        out = hpt.alloc_output(r)
        ctx.trace(sid, r, out, precision=precision)
        ctx.sync()
        assert torch.equal(torch.view_as_real(out), torch.view_as_real(ref))
    ctx.release_scene(sid)
