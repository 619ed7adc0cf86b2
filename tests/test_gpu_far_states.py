"""Flows with |S| beyond the fixed-point form's tables (Mach 8 and 12: FP64 formulas,
whole points and entry by entry) in both layouts of the FP64 flux: the same bits,
and as near binary128 as the parity tests ask."""

import numpy as np
import pytest

from oracle import oracle as O
from paper_2108_07031_gb300 import cloud as Cl
from parity_utils import exact_errors

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2108_07031_gb300 import lskum as L  # noqa: E402


@pytest.mark.parametrize("amplitude", [0.05, 0.002])  # large steps and small ones
def test_far_states_in_both_layouts(amplitude):
    cloud = Cl.naca0012_cloud(130, 41, shuffle=True, seed=5)
    mach, alpha = np.tile([8.0, 12.0], 32), np.linspace(-4.0, 6.0, 64)
    assert cloud.n <= 1 << 18 < cloud.n * 64
    W = np.stack([Cl.perturbed_state(cloud, m, a, amplitude=amplitude, seed=k)
                  for k, (m, a) in enumerate(zip(mach, alpha))])
    with L.Solver.from_cloud(cloud, n_conditions=64) as b:
        b.set_conditions(mach, alpha)
        b.set_state(W)
        R = b.eval_residual()
    oc = O.OracleCloud.from_cloud(cloud)
    for k in (0, 63):
        with L.Solver.from_cloud(cloud) as s:
            s.set_freestream(mach[k], alpha[k])
            s.set_state(W[k])
            assert np.array_equal(R[k], s.eval_residual())
        e = exact_errors(oc, W[k], {"R": R[k]}, idx=np.arange(0, cloud.n, 7))
        assert np.all(e["R"]["gpu_rms"] <= 2.0 * e["R"]["oracle_rms"]), e
