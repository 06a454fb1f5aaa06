"""Gradients of the training kernels at batch sizes around a block's 32 samples
and with more blocks than the reduction has segments, against the FP64
reference (tolerances of a float sum over 32 samples and 64 units: 1e-4 of a
block's largest gradient)."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 7, 31, 32, 33, 255, 257, 1000])
def test_gradients_match_the_reference(B):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_06015_gb300 import bbx
    vec = mlp.pack(mlp.init_params(3)).astype(np.float32)
    rng = np.random.default_rng(B)
    x, t = rng.normal(size=(2, B, 8)).astype(np.float32)
    m = bbx.bbx_mlp_create(5)
    try:
        bbx.bbx_mlp_set_params(m, vec)
        g, loss = bbx.bbx_mlp_gradients(m, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), B)
        q = mlp.unpack(vec.astype(np.float64))
        ref = mlp.pack(mlp.grads(q, x.astype(np.float64), t.astype(np.float64)))
        assert loss == pytest.approx(mlp.loss(q, x, t), rel=1e-5)
        o = 0
        for size in (512, 64, 4096, 64, 512, 8):
            a, b = g[o:o + size], ref[o:o + size]
            assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max() + 1e-9
            o += size
    finally:
        bbx.bbx_mlp_destroy(m)
