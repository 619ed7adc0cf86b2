"""Loss gradients where the weight gradients' sum over the 128-sample tiles is cut
into all of its 15 slices (csrc/mlp_kernels.cu, kMaxSlices): one tile each, two
each, and one tile more than either."""

import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2108_07031_gb300 import surrogate as S  # noqa: E402


@pytest.mark.parametrize("n", [1920, 1921, 3840, 3841])
def test_gradients_with_all_slices(n):
    """2e-2 of a layer's largest entry, as at the tiles' edges: a BF16 rounding on
    the other side of a boundary moves an entry by 2^-8 of itself."""
    rng = np.random.Generator(np.random.PCG64(n))
    feat = rng.normal(0, 1, (n, 32)).astype(np.float32)
    feat[:, 21:] = 0.0
    T = rng.normal(0, 0.5, (n, 4)).astype(np.float32)
    p = S.init_params(7)
    p[-4:] = [0.1, -0.2, 0.05, 0.3]
    net = S.MLP(capacity=n, seed=1)
    try:
        net.set_params(p)
        loss, g = net.gradients(torch.from_numpy(feat).cuda(), torch.from_numpy(T).cuda())
    finally:
        net.close()
    loss_o, g_o = M.loss_and_grad(p, feat, T, emulate=True)
    assert abs(loss - loss_o) < 1e-3 * loss_o
    off = 0
    for rows, k in M.layer_shapes():
        for size in (rows * k, rows):
            gl, gol = g[off:off + size], g_o[off:off + size]
            assert np.abs(gl - gol).max() <= 2e-2 * np.abs(gol).max() + 1e-9, (rows, k, size)
            off += size
