"""A residual that leaves the floats' range in mixed precision is reported: the
step returns the divergence code and the residue is not finite (no finite number
of 1e38 in its place), for the layouts with one and four threads a point."""

import numpy as np
import pytest

from paper_2108_07031_gb300 import cloud as Cl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2108_07031_gb300 import lskum as L  # noqa: E402


@pytest.mark.parametrize("conditions, opts", [(1, {}), (1, dict(gamma=1.3)), (64, {})])
def test_overflowing_residual_is_reported(conditions, opts):
    cloud = Cl.naca0012_cloud(128, 40)
    mach, alpha = Cl.conditions(conditions) if conditions > 1 else (np.array([0.63]), np.array([2.0]))
    W = np.stack([Cl.perturbed_state(cloud, m, a, seed=k) for k, (m, a) in enumerate(zip(mach, alpha))])
    inside = np.flatnonzero(cloud.flags == 0)[2000]
    W[:, inside] = [1e38, 25.0, 0.0, 0.7e38]  # a mass flux of 2.5e39
    with L.Solver.from_cloud(cloud, precision=L.MIXED, n_conditions=conditions, **opts) as s:
        s.set_conditions(mach, alpha)
        s.set_state(W if conditions > 1 else W[0])
        with pytest.raises(L.LskumError) as e:
            s.step(1)
        assert e.value.code == -5
        assert not np.any(np.isfinite(s.residual_norm()))
        s.set_conditions(mach, alpha)  # the context stays usable
        s.step(1)
        assert np.all(np.isfinite(s.residual_norm()))
