"""fp_set_tile under allocation failures (injected on the host): a failed call leaves the context as
it was, with its tile, its launch form and the work items that belong to them."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2101_05886_gb300 import inputs as I

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_2101_05886_gb300 import binding as B  # noqa: E402
from paper_2101_05886_gb300.solver import Block  # noqa: E402


def _tiles(blk):
    S, T = ctypes.c_int(), ctypes.c_int()
    out = []
    for d in range(3):
        assert B.lib().fp_get_tile(blk.ctx, d, ctypes.byref(S), ctypes.byref(T)) == B.FP_OK
        out.append((S.value, T.value))
    return out


def _noalloc(blk, q):
    out = torch.full_like(q, float("nan"))
    st = B.lib().fp_rhs_noalloc(blk.ctx, ctypes.c_void_p(q.data_ptr()), ctypes.c_void_p(out.data_ptr()),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == B.FP_OK
    return out


# WENO5 FP32: the primary shape has 64 threads, the alternative 128 (a block with tiles of both runs
# its directions in turn); FP64: one shape
@pytest.mark.parametrize("precision,tiles", [(B.FP_F32_MIXED, [(1, 8, 8), (2, 16, 8), (2, 8, 8)]),
                                             (B.FP_F64, [(1, 8, 16), (2, 16, 8)])])
def test_failed_set_tile_changes_nothing(precision, tiles):
    g = I.periodic_wavy_3d((33, 26, 21), amp=0.05, Gn=O.node_ghost(6))
    qinf = I.uniform_qinf(0.8, 0.0)
    blk = Block(g, metric_order=6, precision=precision, q_inf=qinf)
    q = blk.to_device(I.random_smooth_state(g, qinf, amp=0.03, seed=3))
    ref = blk.rhs(q)
    assert torch.isfinite(ref).all()
    for d, faces, lines in tiles:
        before, launches = _tiles(blk), B.lib().fp_launches_per_rhs(blk.ctx)
        for k in range(8):
            B.fp_debug_fail_allocation(k)
            st = B.lib().fp_set_tile(blk.ctx, d, faces, lines)
            B.fp_debug_fail_allocation(-1)
            if st == B.FP_OK:
                break
            assert st == B.FP_ERR_OOM
            assert _tiles(blk) == before and B.lib().fp_launches_per_rhs(blk.ctx) == launches
            assert torch.equal(blk.rhs(q), ref) and torch.equal(_noalloc(blk, q), ref)
        assert st == B.FP_OK and k >= 1
        assert _tiles(blk) == before[:d] + [(faces, lines)] + before[d + 1:]
        assert torch.equal(blk.rhs(q), ref) and torch.equal(_noalloc(blk, q), ref)
    assert blk.status() == B.FP_OK
    blk.close()
