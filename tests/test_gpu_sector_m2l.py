"""The tensor-core M2L kernels on mirror sectors (k_m2l_sec: mixed form, k_m2l_oz: FP64 form
and its transpose) at the edges of their tiles, next to the SIMT five-table kernel, which
shares no code with them.  GPU."""
import numpy as np
import pytest
import torch

from paper_2507_18491_gb300 import lmfmm
from paper_2507_18491_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _op(p, **kw):
    # ragged: 1503 points in two layers, pair counts per geometry from 1 to beyond a work item
    w = W.three_layer(n=1503, p=p, depth=3)
    return w, lmfmm.Operator(w.d, w.k, w.xyz, p=p, depth=3, theta=0.5, **kw).build()


def _simt(p):
    w, op = _op(p, precision=lmfmm.MIXED, tensor_cores=0)
    assert op.stats()["m2l_kernel"] == 1
    a = op.matvec(torch.from_numpy(w.J).cuda()).cpu().numpy()
    op.close()
    return a


# one tile per sector with three accumulators (p <= 8; 8: 126 of 128 rows), with two (9, 10: 187 of
# 192), two tiles (11, 12: 260 = 128 + 132 rows); p = 1: 7 rows
@pytest.mark.parametrize("p", [1, 7, 8, 10, 11, 12])
def test_mixed_form(p):
    ref = _simt(p)
    w, op = _op(p, precision=lmfmm.MIXED, tensor_cores=1)
    assert op.stats()["m2l_kernel"] == 3
    a = op.matvec(torch.from_numpy(w.J).cuda()).cpu().numpy()
    op.check()
    op.close()
    # FP32 expansions on both sides: the bar of the mixed form's M2L against the FP64 form
    assert rel(a, ref) < 5e-6


# matrix tiles of 64 rows: one (p = 1), full and 16-row remainders (4: 40; 7: 100 = 64 + 48;
# 10: 187 = 2 x 64 + 64), the largest order (16: 442 = 6 x 64 + 64)
@pytest.mark.parametrize("p", [1, 4, 7, 10, 16])
def test_fp64_form(p):
    w, op = _op(p)
    # FP32 expansions overflow beyond p = 13 (NaN in the SIMT mixed form): the sum over all pairs there
    ref = _simt(p) if p <= 13 else op.direct(torch.from_numpy(w.J).cuda()).cpu().numpy()
    rng = np.random.default_rng(p)
    mv = lambda x: op.matvec(torch.from_numpy(x).cuda()).cpu().numpy()  # noqa: E731
    a = mv(w.J)
    assert rel(a, ref) < 5e-6
    # currents ten orders of magnitude apart in neighbouring boxes: every box has its own grid, so
    # the sum of the parts is the whole to FP64 rounding (three results of ~1e-15)
    near = (w.xyz[:, :1] > 0)
    big, small = np.where(near, 1e10 * w.J, 0), np.where(near, 0, w.J)
    whole, b, s = mv(big + small), mv(big), mv(small)
    assert np.linalg.norm(whole - b - s) < 1e-13 * np.linalg.norm(whole)
    # a power of two goes through the digits exactly; the output atomics leave ~1e-15
    assert rel(mv(2.0 ** 40 * w.J), 2.0 ** 40 * a) < 1e-13
    # the transpose runs on the images of the transposed blocks
    y = rng.standard_normal((w.N, 3)) + 1j * rng.standard_normal((w.N, 3))
    at = op.tmatvec(torch.from_numpy(y).cuda()).cpu().numpy()
    assert abs(np.sum(y * a) - np.sum(at * w.J)) < 1e-12 * np.linalg.norm(y) * np.linalg.norm(a)
    # a current that is not a number does not come out as one
    bad = w.J.copy()
    bad[3, 1] = np.nan
    assert np.isnan(mv(bad)).any()
    assert rel(mv(w.J), a) < 1e-13
    op.check()
    op.close()


@pytest.mark.parametrize("p", [2, 8, 12])
def test_p2m_of_crowded_leaves(p):
    # 69 points per unit on average, above the 5 p at which the kernel for many points takes over;
    # units of a partial pass (69 = 2 x 32 + 5) and of one pass both occur.  FP32 expansions
    # against the FP64 form: the mixed form's bar
    w = W.paper_table_uniform(m=50000, layers=2, p=p)
    J = torch.from_numpy(w.J).cuda()
    out = []
    for kw in (dict(), dict(precision=lmfmm.MIXED, tensor_cores=1)):
        op = lmfmm.Operator(w.d, w.k, w.xyz, p=p, depth=4, theta=0.55, **kw).build()
        out.append(op.matvec(J).cpu().numpy())
        op.close()
    assert rel(out[1], out[0]) < 2e-6
