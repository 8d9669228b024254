"""Set-up and products on a stream that is not ordered behind the legacy one.  GPU."""
import pytest
import torch

from paper_2507_18491_gb300 import lmfmm
from paper_2507_18491_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(), dict(precision=lmfmm.MIXED, tensor_cores=1),
                                dict(precision=lmfmm.MIXED, tensor_cores=3), dict(components=lmfmm.TOTAL)])
def test_build_on_a_side_stream(kw):
    """The same operator as one built on the default stream: every table, phase and translation
    matrix is formed by kernels of the side stream from arrays uploaded just before.  Sums of
    atomics differ by rounding: 1e-13 (FP64), 1e-6 (FP32 expansions)."""
    w = W.three_layer(n=1503, p=6, depth=3)
    J = torch.from_numpy(w.J).cuda()
    torch.cuda.synchronize()
    out = []
    for st in (None, torch.cuda.Stream()):
        op = lmfmm.Operator(w.d, w.k, w.xyz, p=6, depth=3, theta=0.5, **kw).build(st)
        out.append(op.matvec(J, stream=st))
        op.check(st)
        op.close()
    torch.cuda.synchronize()
    tol = 1e-6 if kw.get("precision") == lmfmm.MIXED else 1e-13
    assert (out[0] - out[1]).norm() < tol * out[0].norm()
