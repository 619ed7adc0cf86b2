"""The two layouts of the flux kernels and of the mixed sweeps (four threads or one
thread a point, by the number of (point, condition) pairs) give the same bits: a batch large enough
for one thread a point against its conditions solved alone. Neighbour counts
1-4 modulo the four classes, a wall, a far field and entries of both the
pair form and FP64 all occur in these clouds."""

import numpy as np
import pytest

from paper_2108_07031_gb300 import cloud as Cl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2108_07031_gb300 import lskum as L  # noqa: E402


@pytest.mark.parametrize("n_c, n_r, conditions, opts", [
    (130, 41, 64, {}), (46, 23, 256, dict(order=1, inner_iters=0)), (131, 47, 64, dict(outer_mode=0)),
    (130, 41, 64, dict(precision=L.MIXED)), (131, 47, 64, dict(precision=L.MIXED, outer_mode=0, gamma=1.3))])
def test_both_layouts_agree_bitwise(n_c, n_r, conditions, opts):
    cloud = Cl.naca0012_cloud(n_c, n_r, shuffle=True, seed=5)
    assert cloud.n <= 1 << 18 < cloud.n * conditions
    mach, alpha = Cl.conditions(conditions, seed=3)
    W = np.stack([Cl.perturbed_state(cloud, m, a, seed=k)
                  for k, (m, a) in enumerate(zip(mach, alpha))])
    with L.Solver.from_cloud(cloud, n_conditions=conditions, **opts) as b:
        b.set_conditions(mach, alpha)
        b.set_state(W)
        R = b.eval_residual()
        b.step(2)
        W2 = b.get_state()
    for k in (0, conditions - 1):
        with L.Solver.from_cloud(cloud, **opts) as s:
            s.set_freestream(mach[k], alpha[k])
            s.set_state(W[k])
            assert np.array_equal(R[k], s.eval_residual())
            s.step(2)
            assert np.array_equal(W2[k], s.get_state())
