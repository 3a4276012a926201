"""What hpt_autotune times on a GB300: two full waves of the largest candidate on every lane where the frame has the
paths; on a small frame no wave sizes at all, which would all be the same launch."""
import pytest

from paper_2606_14173_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def test_band_and_candidates():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_14173_gb300 import build, hpt
    build.build()
    ctx = hpt.Context(0)
    try:
        sid = ctx.upload_scene(S.config0_scene())
        big = ctx.autotune(sid, S.config0_render(W=1920, H=1080, spp=128))
        assert 8 << 24 <= big["band_path_samples"] < (8 << 24) + 1920 * 128
        before = big["paths_per_wave"]
        small = ctx.autotune(sid, S.config0_render(W=160, H=90, spp=8))
        assert small["band_path_samples"] == 160 * 90 * 8
        assert small["paths_per_wave"] == before
    finally:
        ctx.close()
