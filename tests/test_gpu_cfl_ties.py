"""The time-step bound where its FP32 screen decides least: density and pressure at opposite ends
of the FP32 range (their quotient below it), metrics and cell volumes likewise, and flows in which
every point ties.  The value is the oracle's FP64 maximum, to 1e-13 as in the other tests of the
bound."""
import dataclasses

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
SIZES = [(17, 13, 9), (41, 37, 29), (41, 25, 38)]     # 1,989, 43,993 and 38,950 points


def _check(g, q, qinf, precision):
    if precision == F32:
        q = np.float32(q).astype(np.float64)
    blk = Block(g, metric_order=6, precision=precision, q_inf=qinf)
    want = O.cfl_dt(O.cfg_for(g, M=6, qinf=qinf), blk.metrics(), q, 0.5)
    assert abs(blk.cfl_dt(blk.to_device(q), 0.5) - want) <= 1e-13 * want
    blk.close()


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("precision", [F64, F32])
@pytest.mark.parametrize("rho,cold,hot", [(1e20, 1e-27, 1e-25), (1e15, 1e-24, 1e-22), (1e10, 1e-22, 1e-19)])
def test_dense_and_cold(rho, cold, hot, precision, n):
    """A slow uniform stream with one hot point at rest, whose sound speed is the block's largest
    speed; p/rho of every point is below the FP32 range, or the lowest values in it."""
    g = I.periodic_wavy_3d(n, amp=0.05, Gn=O.node_ghost(6))
    u = np.sqrt(cold / rho)
    q = np.zeros((5, n[2], n[1], n[0]))
    q[0], q[1], q[4] = rho, rho * u, cold + 0.5 * rho * u * u
    q[:, 4, 6, 8] = (rho, 0, 0, 0, hot)
    _check(g, q, I.uniform_qinf(0.5), precision)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("precision", [F64, F32])
@pytest.mark.parametrize("length,energy", [(2.0 ** 30, 1e-25), (2.0 ** -30, 1e25)])
def test_large_and_small_grids(length, energy, precision, n):
    """Lengths and energies of opposite extremes, one point faster than the rest."""
    g = I.periodic_wavy_3d(n, amp=0.05, Gn=O.node_ghost(6))
    g = dataclasses.replace(g, nodes=g.nodes * length)
    qinf = I.uniform_qinf(0.5, 10.0)
    q = I.random_smooth_state(g, qinf, amp=0.02, seed=4)
    q[1:4] *= np.sqrt(energy)
    q[4] *= energy
    q[1:4, 3, 5, 7] *= 2.0
    _check(g, q, qinf, precision)


@pytest.mark.parametrize("precision", [F64, F32])
@pytest.mark.parametrize("n", [(32, 32, 4), (61, 47, 1), (31, 23, 17), (38, 32, 32), (39, 32, 32), (211, 203, 1)])
def test_uniform_stream_on_a_uniform_grid(n, precision):
    """Every point has the same value, or the same but for the rounding of the metrics."""
    if n[2] == 1:
        g = I.cartesian_2d(n[:2], 0.1, O.node_ghost(6))
    else:
        g = I.cartesian_3d(n, 0.1, O.node_ghost(6))
    qinf = I.uniform_qinf(0.7, 20.0)
    _check(g, I.uniform_state(g, qinf), qinf, precision)
    q = I.uniform_state(g, qinf)
    q[4, -1, -1, -1] *= 1.0 + 1e-6                      # the last point, within the screen's width
    _check(g, q, qinf, precision)


@pytest.mark.parametrize("precision", [F64, F32])
@pytest.mark.parametrize("n", [(41, 37, 29), (41, 25, 38), (197, 199, 1)])
@pytest.mark.parametrize("flow", ["smooth", "mach50", "no_pressure", "tiny"])
def test_the_screen(flow, n, precision):
    """Flows of the other tests of the bound, on blocks that are screened."""
    Gn = O.node_ghost(6)
    g = I.periodic_wavy_2d(max(n[:2]), amp=0.05, Gn=Gn) if n[2] == 1 else I.periodic_wavy_3d(n, amp=0.05, Gn=Gn)
    qinf = I.uniform_qinf(50.0 if flow == "mach50" else 0.7, 20.0)
    q = I.random_smooth_state(g, qinf, amp=1e-4 if flow == "mach50" else 0.05, seed=2)
    if flow == "no_pressure":                           # large momenta, and no pressure, at one point
        q[1:4, -1, 3, 5] *= 20.0
    if flow == "tiny":
        q *= 1e-31                                      # density and energy below the screen's range
    _check(g, q, qinf, precision)
