"""Sweeps whose CTAs march over several lines: blocks with more tiles along eta or zeta than the
device holds CTAs (several rounds of tiles per CTA, then equal pieces of what is left), lines
shorter than a chunk, and boundary ghosts that are loaded in the middle of a stream.  Against
the oracle, with the bounds of the parity suite: 1e-5 in FP32; in FP64 1e-12 or twice the
oracle's own response to one-ulp input changes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2101_05886_gb300 import inputs as I
from tests.helpers import f32, rhs_err, ulp_sensitivity

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_2101_05886_gb300 import binding as B  # noqa: E402
from paper_2101_05886_gb300.solver import Block  # noqa: E402

F64, F32 = B.FP_F64, B.FP_F32_MIXED


@pytest.mark.parametrize("kind,n,scheme,precision", [
    ("wavy", (180, 8, 170), 0, F32), ("wavy", (180, 170, 8), 1, F32), ("wavy", (9, 150, 200), 0, F32),
    ("wavy", (130, 9, 100), 0, F64), ("wall", (130, 12, 100), 1, F64)])
def test_streams_over_many_lines_match_the_oracle(kind, n, scheme, precision):
    Gn = O.node_ghost(6)
    if kind == "wall":
        g = I.cylinder_ogrid(n, Lz=3.0, Gn=Gn, wall=True)
        qinf = I.uniform_qinf(0.5, 0.0)
    else:
        g = I.periodic_wavy_3d(n, amp=0.05, Gn=Gn)
        qinf = I.uniform_qinf(0.8, 0.0)
    q = I.random_smooth_state(g, qinf, amp=0.05, seed=5)
    if precision == F32:
        q, qinf = f32(q), f32(qinf)
    blk = Block(g, metric_order=6, scheme=scheme, precision=precision, q_inf=qinf)
    dq = blk.rhs(blk.to_device(q)).cpu().numpy()
    cfg = O.cfg_for(g, M=6, scheme=scheme, qinf=qinf)
    met = O.metrics(cfg, g.nodes, g.Gn)
    tol = 1e-5 if precision == F32 else max(1e-12, 2.0 * ulp_sensitivity(cfg, met, q))
    assert precision == F32 or tol <= 2e-11, tol
    errs = rhs_err(dq, cfg, met, q, per_component=True)
    assert np.isfinite(dq).all() and max(errs) <= tol, errs
    assert blk.status() == B.FP_OK
    blk.close()


def test_a_cell_without_pressure_has_no_acoustic_speed():
    """A cell whose pressure is negative has no sound speed (NaN): like the oracle, the sweep leaves
    it out of the local Lax-Friedrichs maxima, and its faces stay finite where their Roe state
    is.  The pattern of finite values is the oracle's; the finite ones agree to 1e-10 of the
    largest (about 1e-13 of rounding, and residual terms up to 1e2 times their sum)."""
    Gn = O.node_ghost(6)
    g = I.periodic_wavy_3d((16, 14, 12), amp=0.05, Gn=Gn)
    qinf = I.uniform_qinf(0.8, 10.0)
    q = I.random_smooth_state(g, qinf, amp=0.02, seed=3)
    ke = 0.5 * (q[1:4, 5, 6, 7] ** 2).sum() / q[0, 5, 6, 7]
    q[4, 5, 6, 7] = 0.9 * ke                             # p < 0 there only
    blk = Block(g, metric_order=6, scheme=1, precision=F64, q_inf=qinf)
    dq = blk.rhs(blk.to_device(q)).cpu().numpy()
    cfg = O.cfg_for(g, M=6, scheme=1, qinf=qinf)
    _, ref = O.rhs(cfg, O.metrics(cfg, g.nodes, g.Gn), q)
    fine = np.isfinite(ref)
    assert fine.any() and (np.isfinite(dq) == fine).all()
    assert np.abs(dq[fine] - ref[fine]).max() <= 1e-10 * np.abs(ref[fine]).max()
    blk.close()
