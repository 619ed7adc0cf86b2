"""Loss gradients at the edges of the 128-sample tiles and of the 16 slices that
the weight gradients' sum over the tiles is cut into."""

import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2108_07031_gb300 import surrogate as S  # noqa: E402


def _batch(n):
    rng = np.random.Generator(np.random.PCG64(n))
    feat = rng.normal(0, 1, (n, 32)).astype(np.float32)
    feat[:, 21:] = 0.0
    return feat, rng.normal(0, 0.5, (n, 4)).astype(np.float32)


@pytest.mark.parametrize("n", [1, 128, 129, 2048, 2049, 4225])
def test_gradients_at_tile_and_slice_edges(n):
    """One row, whole tiles, one row more, a tile a slice, and slices of two and
    three tiles with a short last one; a larger batch runs before, so that
    what it left in the workspaces must not count. Against the FP64 reference
    with the same BF16 rounding points: a rounding on the other side of a
    boundary moves an entry by 2^-8 of itself, 2e-2 of a layer's largest
    covers five of them in one entry. Repeated calls give the same bits."""
    p = S.init_params(7)
    p[-4:] = [0.1, -0.2, 0.05, 0.3]
    net = S.MLP(capacity=6000, seed=1)
    try:
        net.set_params(p)
        for k in (6000, n):
            feat, T = _batch(k)
            fd, Td = torch.from_numpy(feat).cuda(), torch.from_numpy(T).cuda()
            loss, g = net.gradients(fd, Td)
        assert np.array_equal(g, net.gradients(fd, Td)[1])
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
