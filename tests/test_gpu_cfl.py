"""The time-step bound, whose points are screened in FP32, against the oracle's FP64 evaluation on
the metrics the block holds: flows where the screen has little to go by (uniform, hypersonic
with the pressure a small difference of energies, a point without a pressure, values near the
end of the FP32 range), and point counts around the 1024 points of a CTA.  Both evaluate one
FP64 formula in different order: at most 12 roundings, 1e-13."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2101_05886_gb300 import inputs as I

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_2101_05886_gb300 import binding as B  # noqa: E402
from paper_2101_05886_gb300.solver import Block  # noqa: E402

F64, F32 = B.FP_F64, B.FP_F32_MIXED


@pytest.mark.parametrize("precision", [F64, F32])
@pytest.mark.parametrize("n,flow", [((16, 16, 4), "smooth"), ((41, 25, 1), "smooth"), ((33, 31, 1), "uniform"),
                                    ((30, 20, 11), "mach50"), ((30, 20, 11), "no_pressure"), ((21, 17, 9), "tiny")])
def test_cfl_bound_equals_the_fp64_maximum(n, flow, precision):
    Gn = O.node_ghost(6)
    g = I.periodic_wavy_2d(max(n[:2]), amp=0.05, Gn=Gn) if n[2] == 1 else I.periodic_wavy_3d(n, amp=0.05, Gn=Gn)
    qinf = I.uniform_qinf(50.0 if flow == "mach50" else 0.7, 20.0)
    q = I.uniform_state(g, qinf) if flow == "uniform" else I.random_smooth_state(g, qinf, amp=1e-4 if flow == "mach50" else 0.05, seed=2)
    if flow == "no_pressure":
        # the largest momentum of the block, and so little energy that its pressure is negative
        q[1:4, -1, 3, 5] *= 20.0
    if flow == "tiny":
        q *= 1e-31                                   # density and energy below the screen's range
    if precision == F32:
        q = np.float32(q).astype(np.float64)
    blk = Block(g, metric_order=6, precision=precision, q_inf=qinf)
    cfg = O.cfg_for(g, M=6, qinf=qinf)
    want = O.cfl_dt(cfg, blk.metrics(), q, 0.5)
    assert abs(blk.cfl_dt(blk.to_device(q), 0.5) - want) <= 1e-13 * want
    blk.close()
