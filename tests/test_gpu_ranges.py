"""Units far from 1: the sweep's intermediate products stay in range wherever its inputs do.

Scaling by powers of two is exact, so a problem in other units has the same significands, and the
residuals are compared bit for bit after scaling back."""
import dataclasses

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
from paper_2101_05886_gb300.solver import Batch, Block  # noqa: E402

N = (22, 14, 11)


def _case(precision, seed):
    g = I.periodic_wavy_3d(N, amp=0.05, Gn=O.node_ghost(6, 2))
    qinf = I.uniform_qinf(0.8, 10.0)
    q = I.random_smooth_state(g, qinf, amp=0.05, seed=seed)
    return (g, f32(qinf), f32(q)) if precision == B.FP_F32_MIXED else (g, np.asarray(qinf), q)


def _rhs(g, q, qinf, **kw):
    blk = Block(g, metric_order=6, q_inf=tuple(qinf), **kw)
    dq = blk.rhs(blk.to_device(q)).cpu().numpy()
    assert blk.status() == B.FP_OK
    blk.close()
    return dq


@pytest.mark.parametrize("characteristic,global_lf,length,speed", [
    (1, 0, 27, 17), (0, 0, 27, 17), (1, 1, 27, 17), (0, 1, 27, 17), (0, 0, 40, 0), (0, 0, -40, 0), (0, 1, 40, 0), (0, 1, -40, 0)])
def test_fp32_linear_upwind_in_large_units(characteristic, global_lf, length, speed):
    """Lengths in units of 2^-27 and speeds in units of 2^-17 (metres and metres per second on a
    planet-sized grid): |k| is about 2^53 and the sound speed about 2^17, so |k|^2, 1/J and all
    fluxes are FP32 numbers but c^2 |k|^2, about 2^140, is not.  Component-wise, which needs no
    unit normal, also lengths whose |k|^2 is not one.  Linear upwind and its speeds have no
    constant with a unit, so the residual has the bits of the problem in units of 1; with 1/J near
    2^-120, where products with small differences of the state are subnormal, it agrees to the FP32
    bound of the parity suite, 1e-5 of the largest of each component."""
    g, qinf, q = _case(B.FP_F32_MIXED, 7)
    big = dataclasses.replace(g, nodes=g.nodes * 2.0 ** length)
    unit = 2.0 ** np.array([0, speed, speed, speed, 2 * speed])
    kw = dict(scheme=B.FP_LINEAR_UPWIND5, precision=B.FP_F32_MIXED, characteristic=characteristic, global_lf=global_lf)
    want = _rhs(g, q, qinf, **kw)
    got = _rhs(big, q * unit[:, None, None, None], qinf * unit, **kw)
    assert np.isfinite(want).all() and np.abs(want).max() > 1e-3
    got = got / (unit * 2.0 ** (speed - length))[:, None, None, None]
    if length > 0:
        assert np.array_equal(got, want)
    else:
        assert (np.abs(got - want).reshape(5, -1).max(1) <= 1e-5 * np.abs(want).reshape(5, -1).max(1)).all()


@pytest.mark.parametrize("characteristic", [1, 0])
@pytest.mark.parametrize("power", [130, 240])
def test_fp64_weno5_of_large_states(power, characteristic):
    """The Euler fluxes and the WENO5 weights (where the constant 1e-6 is negligible) do not depend
    on the unit of the conserved variables: a state times 2^130 or 2^240, whose squared indicators
    (2^500, 2^940) are FP64 numbers though their products are not, has the residual of the state
    times 2^100, and the oracle's."""
    g, qinf, q = _case(B.FP_F64, 8)
    kw = dict(scheme=B.FP_WENO5_JS, precision=B.FP_F64, characteristic=characteristic)
    want = _rhs(g, q * 2.0 ** 100, qinf * 2.0 ** 100, **kw)
    got = _rhs(g, q * 2.0 ** power, qinf * 2.0 ** power, **kw)
    assert np.isfinite(want).all() and np.abs(want).max() > 0
    assert np.array_equal(got * 2.0 ** (100 - power), want)
    # the oracle in the same units; its error bound is that of the parity suite
    cfg = O.cfg_for(g, M=6, scheme=0, charwise=characteristic, qinf=qinf * 2.0 ** 130)
    met = O.metrics(cfg, g.nodes, g.Gn)
    q130 = q * 2.0 ** 130
    tol = max(1e-12, 2.0 * ulp_sensitivity(cfg, met, q130))
    assert tol <= 2e-11, tol
    assert max(rhs_err(got * 2.0 ** (130 - power), cfg, met, q130, per_component=True)) <= tol


@pytest.mark.parametrize("scheme,power,base", [(1, -80, -50), (1, 70, 60), (0, -80, -60), (2, -80, -60), (0, 200, 100)])
@pytest.mark.parametrize("characteristic,global_lf", [(1, 0), (0, 0), (1, 1)])
@pytest.mark.parametrize("precision", [B.FP_F32_MIXED, B.FP_F64])
def test_states_in_other_units(precision, characteristic, global_lf, scheme, power, base):
    """Densities far from 1 (a thin gas in kg/m^3: 2^-80 is 8e-25) at ordinary velocities: the residual
    has the bits of the state in other units, for linear upwind at any two units, for WENO5 and WENO7
    where the constant 1e-6 of the weights is far above every indicator (2^-60 and below) or, in FP64,
    far below (2^100 and above); and it is the oracle's, with the bounds of the parity suite."""
    if power > 100 and precision == B.FP_F32_MIXED:
        pytest.skip("beyond the FP32 range")
    g, qinf, q = _case(B.FP_F32_MIXED, 9)               # float values in both precisions
    kw = dict(scheme=scheme, precision=precision, characteristic=characteristic, global_lf=global_lf)
    u = 2.0 ** base
    want = _rhs(g, q * u, qinf * u, **kw)
    got = _rhs(g, q * 2.0 ** power, qinf * 2.0 ** power, **kw)
    assert np.isfinite(want).all() and np.abs(want).max() > 0
    assert np.array_equal(got * 2.0 ** (base - power), want)
    if power > 100:
        return                                          # test_fp64_weno5_of_large_states
    cfg = O.cfg_for(g, M=6, scheme=scheme, charwise=characteristic, global_lf=global_lf, qinf=qinf * 2.0 ** power)
    met, qp = O.metrics(cfg, g.nodes, g.Gn), q * 2.0 ** power
    tol = 1e-5 if precision == B.FP_F32_MIXED else max(1e-12, 2.0 * ulp_sensitivity(cfg, met, qp))
    assert max(rhs_err(got, cfg, met, qp, per_component=True)) <= tol


def test_batches_of_states_in_other_units():
    """A batch with one block far from unit scale runs all of them by that sweep; blocks of ordinary
    units keep to the bounds of the parity suite, and the others have their single-block bits."""
    g, qinf, q = _case(B.FP_F32_MIXED, 10)
    scale = [2.0 ** -70, 1.0, 2.0 ** -80]
    for scheme in (0, 1, 2):
        blks = [Block(g, metric_order=6, scheme=scheme, precision=B.FP_F32_MIXED, q_inf=tuple(qinf * s)) for s in scale]
        for order in ((0, 1, 2), (1, 0, 2)):
            bs = [blks[k] for k in order]
            qs = [b.to_device(q * scale[k]) for b, k in zip(bs, order)]
            for tune in (False, True):
                bat = Batch(bs, qs, autotune=tune)
                outs = bat.rhs([torch.full_like(x, float("nan")) for x in qs])
                for b, k, x, o in zip(bs, order, qs, outs):
                    if k != 1:
                        assert torch.equal(o, b.rhs(x))
                    cfg = O.cfg_for(g, M=6, scheme=scheme, qinf=qinf * scale[k])
                    met = O.metrics(cfg, g.nodes, g.Gn)
                    assert max(rhs_err(o.cpu().numpy(), cfg, met, q * scale[k], per_component=True)) <= 1e-5
                before = [x.clone() for x in qs]
                bat.rk3_step(1e-3)
                torch.cuda.synchronize()
                assert all(torch.isfinite(x).all() and not torch.equal(x, y) for x, y in zip(qs, before))
                for x, y in zip(qs, before):
                    x.copy_(y)
                torch.cuda.synchronize()
                bat.close()
        for b in blks:
            assert b.status() == B.FP_OK
            b.close()
