"""The FP64 residual where its large steps take the fixed-point form (Mach 0.63),
the general FP64 formulas (Mach 12, |S| about 10) and, entry by entry, one or
the other (Mach 7, |S| about the table's end at 6): within twice the FP64
oracle's own distance from the binary128 reference, the bar of the parity
tests."""

import numpy as np
import pytest

from oracle import oracle as O
from paper_2108_07031_gb300 import cloud as Cl
from parity_utils import describe, exact_errors

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2108_07031_gb300 import lskum as L  # noqa: E402


@pytest.mark.parametrize("mach", [0.63, 7.0, 12.0])
def test_residual_over_the_forms_ranges(mach):
    cloud = Cl.naca0012_cloud(46, 23, shuffle=True, seed=5)
    oc = O.OracleCloud.from_cloud(cloud)
    W = Cl.perturbed_state(cloud, mach, 2.0, seed=7)
    with L.Solver.from_cloud(cloud) as s:
        s.set_freestream(mach, 2.0)
        s.set_state(W)
        e = exact_errors(oc, W, {"R": s.eval_residual()})
    print(describe(e))
    assert np.all(e["R"]["gpu_rms"] <= 2.0 * e["R"]["oracle_rms"]), e
