"""fp_get_metrics and fp_get_face_metrics read the packed arrays back through a buffer of limited size:
blocks whose ghosted values are more than that (thin ones, in one piece or many), 2-D ones with
their zero third vector, both precisions, before and after a step.  Against the oracle's metrics with
the bounds of the parity suite (1e-12 of the largest), and one rounding to float."""
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


@pytest.mark.parametrize("precision", [B.FP_F64, B.FP_F32_MIXED])
@pytest.mark.parametrize("n", [(33, 33, 1), (4, 5, 1), (4, 4, 4), (40, 4, 5), (21, 18, 13)])
def test_metrics_read_back(n, precision):
    M = 8
    Gn = O.node_ghost(M)
    if n[2] == 1:
        g = I.cartesian_2d(n[:2], 0.1, Gn)
        y = g.nodes[1]
        g.nodes[0] += 0.02 * np.sin(3 * y)
    else:
        g = I.periodic_wavy_3d(n, amp=0.03, Gn=Gn)
    qinf = I.uniform_qinf(0.5, 10.0)
    blk = Block(g, metric_order=M, precision=precision, q_inf=qinf)
    met = O.metrics(O.cfg_for(g, M=M, qinf=qinf), g.nodes, g.Gn).reshape(10, -1)
    tol = np.abs(met).max() * (1e-12 + (2.0 ** -24 if precision == B.FP_F32_MIXED else 0.0))
    q = blk.to_device(I.uniform_state(g, qinf))
    want = blk.rhs(q)
    for _ in range(2):
        got = blk.metrics()
        assert np.abs(got.reshape(10, -1) - met).max() <= tol
        faces = [blk.face_metrics(d) for d in range(g.dims)]
        assert torch.equal(blk.rhs(q), want)
        blk.rk3_step(q.clone(), 1e-4)
    assert np.array_equal(blk.metrics(), got)
    if n[2] == 1:
        assert not got[6:9].any() and not got[2].any() and not got[5].any()
    # a face's metric is the order-M midpoint value of the cells' along its line
    c, G = O.interp_coef(M), O.ghost(M)
    cells = met.reshape(got.shape)
    for d in range(g.dims):
        ax = 2 - d
        for a in range(3):
            arr = cells[3 * d + a]
            for e in range(g.dims):
                if e != d:
                    arr = np.take(arr, np.arange(G, G + n[e]), axis=2 - e)
            ref = sum(c[m] * np.take(arr, np.arange(-1, n[d]) - M // 2 + 1 + m + G, axis=ax) for m in range(M))
            assert np.abs(faces[d][a] - ref).max() <= 4 * tol
    blk.close()
