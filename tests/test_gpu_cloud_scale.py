"""FP64 on clouds of any size: the residual of a cloud scaled by a power of two is the
unscaled one's divided by it, also where offsets, weights and derivatives lie
outside the floats' range."""

import dataclasses

import numpy as np
import pytest

from paper_2108_07031_gb300 import cloud as Cl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2108_07031_gb300 import lskum as L  # noqa: E402


def _residual(cloud, log2_scale, W, **opts):
    scaled = dataclasses.replace(cloud, xy=np.ldexp(cloud.xy, log2_scale))
    with L.Solver.from_cloud(scaled, **opts) as s:
        s.set_freestream(0.63, 2.0)
        s.set_state(W)
        return np.ldexp(s.eval_residual(), log2_scale)


@pytest.mark.parametrize("inner", [0, 1, 2, 3])
def test_residual_scales_with_the_cloud(inner):
    """Within the pair form's sizes every operation scales exactly: the same bits.
    Beyond them FP64 throughout: the two forms' errors are some 1e-13 of the
    residual's largest entry at this size; 1e-11 leaves room."""
    cloud = Cl.naca0012_cloud(46, 23, shuffle=True, seed=5)
    W = Cl.perturbed_state(cloud, 0.63, 2.0, seed=7)
    R = _residual(cloud, 0, W, inner_iters=inner)
    for k in (-8, 12):
        assert np.array_equal(_residual(cloud, k, W, inner_iters=inner), R)
    for k in (-200, -140, 40, 140):
        assert np.abs(_residual(cloud, k, W, inner_iters=inner) - R).max() <= 1e-11 * np.abs(R).max()
