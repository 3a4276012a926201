"""Wave-optics calls on a nearly full device: what 8-field groups and single maps once fitted into is still enough, and
the results are the ones of the full groups, bit for bit."""
import pytest

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


class _Full:
    """Holds the device's memory but for 'left' MB."""

    def __init__(self, torch, left):
        self.torch, self.left, self.held = torch, left << 20, []

    def __enter__(self):
        self.torch.cuda.synchronize()
        while True:
            n = min(self.torch.cuda.mem_get_info()[0] - self.left, 32 << 30) & ~((2 << 20) - 1)
            if n < 4 << 20:
                return self
            self.held.append(self.torch.empty(n, dtype=self.torch.uint8, device="cuda"))

    def __exit__(self, *exc):
        self.torch.cuda.synchronize()
        self.held.clear()
        self.torch.cuda.empty_cache()


def test_smaller_groups_when_memory_is_short(ctx):
    import torch
    lib, ptr = ctx.lib, lambda t: t.data_ptr()
    import ctypes as C
    lams = (638e-9, 520e-9, 450e-9)
    g = torch.Generator(device="cuda").manual_seed(5)
    U = torch.view_as_complex(torch.randn((3, 25, 512, 512, 2), generator=g, device="cuda"))
    out = torch.empty_like(U)
    phi = torch.empty((8, 2048, 4096), dtype=torch.float32, device="cuda")
    lam = (C.c_double * 3)(*lams)

    def grf():
        return lib.hpt_grf_build(ctx.h, C.c_uint64(5), 0, 8, 4096, 2048, 6.4e-6, C.c_void_p(ptr(phi)), None)

    def asm():
        return lib.hpt_asm_propagate(ctx.h, C.c_void_p(ptr(U)), C.c_void_p(ptr(out)), 512, 512, 3, 25, lam, 6.4e-6, 0.02, None)

    # a small call first: the kernels' code is loaded, the pool still small
    tiny = ctx.grf_build(5, 1, 64, 64, 6.4e-6)
    ctx.asm_propagate(U[:, :1, :8, :8].contiguous(), lams, 6.4e-6, 0.02)
    del tiny
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    with _Full(torch, 150):
        assert grf() == 0, lib.hpt_last_error()      # a group of four maps needs 268 MB, one 67 MB
        torch.cuda.synchronize()
        assert asm() == 0, lib.hpt_last_error()      # 75 fields of 4 MB and three transfer functions of 4 MB
        torch.cuda.synchronize()
    small_phi, small_out = phi.clone(), out.clone()
    assert grf() == 0 and asm() == 0
    torch.cuda.synchronize()
    assert torch.equal(small_phi, phi)
    assert torch.equal(torch.view_as_real(small_out), torch.view_as_real(out))


def test_a_call_gets_back_what_the_wave_optics_pool_keeps(ctx):
    """The pool keeps a propagation's 300 MB between calls; any later allocation of the context that would fail
    otherwise has it back: the probes' 64 MB and the autotuner's 17 MB output here."""
    import torch
    from paper_2606_14173_gb300 import scenes as S
    lams = (638e-9, 520e-9, 450e-9)
    sid = ctx.upload_scene(S.config0_scene())
    r = S.config0_render(W=1920, H=1080, spp=2)
    ctx.autotune(sid, r)                             # the wave state is there
    U = torch.zeros((3, 25, 512, 512), dtype=torch.complex64, device="cuda")
    for call in (ctx.probe_peaks, lambda: ctx.autotune(sid, r)):
        ctx.asm_propagate(U, lams, 6.4e-6, 0.02, out=U)
        with _Full(torch, 8):
            call()
    ctx.release_scene(sid)
