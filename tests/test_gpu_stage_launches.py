"""The ways a stage is launched give the same bits: all directions in one launch with a sum behind it
(blocks up to a limit by scheme and precision), chained passes in turn (beyond it, and in
every batch), and the unchained passes of fp_rhs_noalloc; with boundary rules compiled into all
directions or only into those that have such a side."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2101_05886_gb300 import inputs as I

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_2101_05886_gb300 import binding as B  # noqa: E402
from paper_2101_05886_gb300.solver import Batch, Block  # noqa: E402

F64, F32 = B.FP_F64, B.FP_F32_MIXED
LIMIT = {(0, F32): 3 << 19, (1, F32): 7 << 17, (2, F32): 3 << 18, (0, F64): 3 << 19}   # points, by scheme and precision


def _setup(kind, n, scheme, precision, **kw):
    Gn = O.node_ghost(6, scheme)
    if kind == "wall":
        g, qinf = I.cylinder_ogrid(n, Lz=3.0, Gn=Gn, wall=True), I.uniform_qinf(0.5, 3.0)
    else:
        g, qinf = I.periodic_wavy_3d(n, amp=0.05, Gn=Gn), I.uniform_qinf(0.8, 10.0)
    blk = Block(g, metric_order=6, scheme=scheme, precision=precision, q_inf=qinf, **kw)
    return blk, blk.to_device(I.random_smooth_state(g, qinf, amp=0.03, seed=6))


def _noalloc(blk, q):
    out = torch.full_like(q, float("nan"))
    st = B.lib().fp_rhs_noalloc(blk.ctx, ctypes.c_void_p(q.data_ptr()), ctypes.c_void_p(out.data_ptr()),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == B.FP_OK, B.lib().fp_last_error(blk.ctx)
    return out


def _close(*objs):
    torch.cuda.synchronize()
    for o in objs:
        o.close()


# every scheme, precision and switch on blocks whose launches differ in their work items: where an
# item starts, its first cells are staged by other code than the rest
@pytest.mark.parametrize("kw", [{}, dict(characteristic=0), dict(fp=0), dict(global_lf=1), dict(fp=0, characteristic=0)],
                         ids=lambda kw: "-".join(kw) or "default")
@pytest.mark.parametrize("precision", [F32, F64], ids=["f32", "f64"])
@pytest.mark.parametrize("scheme", [0, 1, 2, 3])
@pytest.mark.parametrize("kind,n", [("wall", (96, 40, 34)), ("wavy", (9, 150, 60))], ids=["wall", "wavy"])
def test_one_launch_or_passes_in_turn(kind, n, scheme, precision, kw):
    blk, q = _setup(kind, n, scheme, precision, **kw)
    bat = Batch([blk], [q], autotune=False)
    ref = blk.rhs(q)
    assert torch.isfinite(ref).all() and ref.abs().max() > 0
    assert torch.equal(bat.rhs([torch.full_like(q, float("nan"))])[0], ref)
    assert torch.equal(_noalloc(blk, q), ref)
    S, T = ctypes.c_int(), ctypes.c_int()
    for d in (1, 2):                                      # other tiles, other items
        assert B.lib().fp_get_tile(blk.ctx, d, ctypes.byref(S), ctypes.byref(T)) == B.FP_OK
        faces = 8 if S.value != 8 else 16
        assert B.lib().fp_set_tile(blk.ctx, d, faces, S.value * T.value // faces) == B.FP_OK
    assert torch.equal(blk.rhs(q), ref)
    _close(bat, blk)


# more tiles along eta than two rounds of the resident CTAs: whole rounds, then equal pieces
@pytest.mark.parametrize("n,scheme,precision", [((180, 8, 170), 0, F32), ((180, 8, 170), 1, F32), ((130, 9, 100), 0, F64)])
def test_many_rounds_of_tiles(n, scheme, precision):
    blk, q = _setup("wavy", n, scheme, precision)
    ref = blk.rhs(q)
    assert torch.isfinite(ref).all() and ref.abs().max() > 0
    assert torch.equal(_noalloc(blk, q), ref)
    _close(blk)


# just below and just above each limit
@pytest.mark.parametrize("n,scheme,precision", [
    ((181, 97, 89), 0, F32), ((181, 97, 90), 0, F32), ((181, 97, 52), 1, F32), ((181, 97, 53), 1, F32),
    ((181, 97, 44), 2, F32), ((181, 97, 45), 2, F32), ((181, 97, 89), 0, F64), ((181, 97, 90), 0, F64)])
def test_steps_on_either_side_of_the_limit(n, scheme, precision):
    blk, q = _setup("wall", n, scheme, precision)
    assert B.lib().fp_launches_per_rhs(blk.ctx) == (2 if np.prod(n) <= LIMIT[scheme, precision] else 3)
    dt = blk.cfl_dt(q, 0.4)
    a, b = q.clone(), q.clone()
    bat = Batch([blk], [b], autotune=False)
    for _ in range(2):
        blk.rk3_step(a, dt)
    torch.cuda.synchronize()                              # the batch and the block share the stage states
    for _ in range(2):
        bat.rk3_step(dt)
    torch.cuda.synchronize()
    assert torch.isfinite(a).all() and not torch.equal(a, q)
    assert torch.equal(a, b)
    assert blk.status() == B.FP_OK
    _close(bat, blk)
