"""The angular-spectrum propagation at every transform length it is built for (padded 2 .. 8192 along
either axis), odd windows, windows that fill their half exactly, rows that do not fill a block and
field counts that do not fill a group, against the FP64 oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# A float32 FFT convolution of N points errs by about eps log2 N in the 2-norm (eps = 2^-24): two
# transforms each way over at most 2^26 padded points, with a margin of two for the twiddles and the
# transfer function.
TOL = 2 * 2 * 26 * 2.0 ** -24


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


@pytest.mark.parametrize("W,H,nl,K", [
    (1, 4, 1, 1), (4, 1, 2, 3), (2, 2, 1, 2), (3, 5, 3, 2), (8, 9, 1, 3), (16, 17, 2, 1), (31, 32, 1, 4), (33, 64, 1, 2),
    (64, 65, 3, 1), (127, 128, 1, 3), (129, 255, 1, 2), (256, 257, 1, 1), (511, 300, 2, 2), (513, 512, 1, 1),
    (1023, 100, 1, 5), (1025, 33, 3, 1), (2048, 7, 1, 3), (2049, 3, 1, 1), (4096, 2, 1, 1), (5, 1024, 1, 2),
    (3, 2047, 1, 1), (2, 2049, 2, 1), (1, 4096, 1, 1), (1030, 1100, 1, 9)])
def test_every_length(ctx, W, H, nl, K):
    import torch
    from oracle import waveoptics as wo
    lams = (638e-9, 520e-9, 450e-9)[:nl]
    rng = np.random.default_rng(W * 5000 + H)
    U = (rng.normal(size=(nl, K, H, W)) + 1j * rng.normal(size=(nl, K, H, W))).astype(np.complex64)
    got = ctx.asm_propagate(torch.from_numpy(U).cuda(), lams, 6.4e-6, 7e-3)
    ctx.sync()
    got = got.cpu().numpy()
    ref = wo.asm_propagate(U, 6.4e-6, lams, 7e-3)
    for l in range(nl):
        for k in range(K):
            d = np.linalg.norm(got[l, k] - ref[l, k]) / np.linalg.norm(ref[l, k])
            assert d <= TOL, (l, k, d)
