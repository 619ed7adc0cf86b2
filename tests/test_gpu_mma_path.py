"""The network's forward pass on mma.sync, as lskum_mlp_set_gemm selects it: against
the FP64 reference at the edges of its 64-row tiles, and another kernel than the
default one."""

import numpy as np
import pytest

from oracle import mlp_oracle as M
from parity_utils import normwise

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2108_07031_gb300 import surrogate as S  # noqa: E402


def _case(n):
    rng = np.random.Generator(np.random.PCG64(n))
    feat = rng.normal(0, 1, (n, 32)).astype(np.float32)
    feat[:, 21:] = 0.0
    p = S.init_params(9)
    p[-4:] = [0.1, -0.2, 0.05, 0.3]
    return feat, rng.normal(0, 0.5, (n, 4)).astype(np.float32), p


@pytest.mark.parametrize("n", [1, 63, 64, 65, 127, 129, 1000])
def test_forward_and_gradients_on_mma_sync(n):
    """The bounds of the other path's tests: 5e-3 norm-wise and 2e-2 a layer (a
    BF16 rounding on the other side of a boundary)."""
    feat, T, p = _case(n)
    net = S.MLP(capacity=1200, seed=1)
    try:
        net.set_params(p)
        net.set_gemm(S.GEMM_MMA_SYNC)
        for k in (1200, n):  # what a larger batch left in the workspaces must not count
            f, t, _ = _case(k) if k != n else (feat, T, p)
            fd, Td = torch.from_numpy(f).cuda(), torch.from_numpy(t).cuda()
            Y = net.predict(fd).cpu().numpy()
            loss, g = net.gradients(fd, Td)
    finally:
        net.close()
    Y_o, _ = M.forward(p, feat, emulate=True)
    assert normwise(Y, Y_o) < 5e-3
    loss_o, g_o = M.loss_and_grad(p, feat, T, emulate=True)
    assert abs(loss - loss_o) < 1e-3 * loss_o
    off = 0
    for rows, k in M.layer_shapes():
        for size in (rows * k, rows):
            gl, gol = g[off:off + size], g_o[off:off + size]
            assert np.abs(gl - gol).max() <= 2e-2 * np.abs(gol).max() + 1e-9, (rows, k, size)
            off += size


def test_the_choice_selects_a_kernel():
    """The two sum 256 products in different orders: of 16,384 outputs some differ in
    the last place. The default is tcgen05."""
    feat, _, p = _case(4096)
    net = S.MLP(capacity=4096, seed=1)
    try:
        net.set_params(p)
        fd = torch.from_numpy(feat).cuda()
        default = net.predict(fd).cpu().numpy()
        net.set_gemm(S.GEMM_MMA_SYNC)
        mma = net.predict(fd).cpu().numpy()
        net.set_gemm(S.GEMM_TCGEN05)
        tc = net.predict(fd).cpu().numpy()
    finally:
        net.close()
    assert np.array_equal(default, tc)
    assert not np.array_equal(mma, tc)
    assert normwise(mma, tc) < 1e-2
