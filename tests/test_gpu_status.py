"""The device status word over calls of several passes.  GPU; failures are injected from the host."""
import pytest
import torch

from paper_2507_18491_gb300 import lmfmm
from paper_2507_18491_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_a_gradient_keeps_the_status_of_its_forward_pass():
    """A wait that gives up in the gradient's forward M2L leaves incomplete local expansions:
    the transposed pass must not clear the word; the next call starts from a clear one."""
    w = W.two_layer_small(n=300, seed=3)
    op = lmfmm.Operator(w.d, w.k, w.xyz, p=4, depth=2).build()
    try:
        J = torch.from_numpy(w.J).cuda()
        op.vjp(J, J)
        op.check()
        for call in (lambda: op.matvec(J), lambda: op.vjp(J, J)):
            lmfmm.test_fail_m2l(op.ctx, 4)
            call()
            with pytest.raises(lmfmm.LmfmmError) as ei:
                op.check()
            assert ei.value.code == lmfmm.ERR_TIMEOUT
            op.vjp(J, J)
            op.check()
        # one pass, not cleared by what the forward pass left
        lmfmm.test_fail_m2l(op.ctx, 4)
        op.vjp(J, J)
        op.rmatvec(J)
        op.check()
    finally:
        op.close()
