"""The adjoint's boundary items at the smallest meshes, where an interface is next to two walls, a
cell next to both ends, or an axis its own periodic image: against the oracle's complex-step
derivatives, with the tolerances of test_gpu_adjoint.py (FP64)."""
import pytest

from paper_1411_6121_gb300 import workloads as W

from . import test_gpu_adjoint as A

pytestmark = pytest.mark.gpu

PER = [W.periodic(), W.periodic()]
XWALLS = [W.bounce_back((0.0, 0.01, 0.0)), W.wall((0.0, 0.02, 0.0))]
YWALLS = [W.wall((0.03, 0.0, 0.0)), W.bounce_back()]
FLOWS = {"walls": XWALLS + YWALLS, "x_periodic": PER + YWALLS, "y_periodic": XWALLS + PER, "periodic": PER + PER,
         "pressure": [W.pressure(2e-3, 1e-3), W.pressure(-1e-3)] + YWALLS}


@pytest.mark.parametrize("flow", sorted(FLOWS))
@pytest.mark.parametrize("shape", [(1, 1), (1, 4), (2, 2), (2, 3), (3, 2), (4, 3)])
def test_adjoint_smallest_meshes(shape, flow, monkeypatch):
    bcs = FLOWS[flow]
    if any(n == 1 and bcs[2 * d][0] != 0 for d, n in enumerate(shape)):
        pytest.skip("a wall axis needs two cells")
    cfg = dict(shape=shape, q=9, nu=0.05, dt=0.5, g=(2e-5, -1e-5, 0.0), omega=0.07, bcs=bcs)
    monkeypatch.setitem(A.CASES, "small", cfg)
    A.test_adjoint_equals_oracle_complex_step("small")
