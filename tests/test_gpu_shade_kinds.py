"""The FP64 coherent shading gathers a warp's entries by what they hit (image points, delta vertices): ragged
frames, whose last warps hold part of a chunk of either kind, of one kind only (receiver) and of both, against
the oracle, and through the fixed scratch, whose waves cut the paths elsewhere, to the same bits."""
import numpy as np
import pytest

from paper_2606_14173_gb300 import scenes as S
from tests.parity import assert_parity

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


@pytest.mark.parametrize("scene", ["receiver", "spheres"])
@pytest.mark.parametrize("W,H,spp", [(1, 1, 1), (33, 31, 1), (41, 31, 3), (64, 48, 8)])
def test_fp64_ragged_frames(ctx, oracle_mod, scene, W, H, spp):
    from paper_2606_14173_gb300 import hpt
    sc = S.lit_receiver_scene(kind=S.LAMBERT) if scene == "receiver" else S.config1_scene()
    sid = ctx.upload_scene(sc)
    r = S.config1_render(W=W, H=H, spp=spp, K=1, max_depth=2)
    out, fixed = hpt.alloc_output(r), hpt.alloc_output(r)
    ctx.trace(sid, r, out, precision=hpt.PREC_FP64)
    ctx.trace_fixed_scratch(sid, r, fixed, precision=hpt.PREC_FP64)
    ctx.sync()
    U = out.cpu().numpy()
    assert np.array_equal(U.view(np.uint64), fixed.cpu().numpy().view(np.uint64))
    assert_parity(U, oracle_mod.Oracle(sc).trace_full(r), f"{scene} {W}x{H}x{spp}")
    ctx.release_scene(sid)
