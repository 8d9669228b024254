"""Device memory held by an operator.  GPU."""
import pytest
import torch

from paper_2507_18491_gb300 import lmfmm
from paper_2507_18491_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# 48 far pairs in 8 geometries at p = 12: images of 2 x 4.33 MB (FP64) or 1.67 MB (mixed) per
# geometry, scratch of 1.6 MB or 0.27 MB per work item, and some 40 allocations of up to 2 MB
# that round up; a scratch for every SM alone takes 243 MB and 41 MB
@pytest.mark.parametrize("kw,limit", [(dict(), 200e6), (dict(precision=lmfmm.MIXED, tensor_cores=3), 60e6)])
def test_scratch_follows_the_work_items(kw, limit):
    w = W.two_layer_small(n=40, seed=3)
    build = lambda: lmfmm.Operator(w.d, w.k, w.xyz, p=12, depth=1, **kw).build()  # noqa: E731
    J = torch.from_numpy(w.J).cuda()
    warm = build()            # modules and pools of the first build
    warm.matvec(J)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    ops = [build() for _ in range(3)]
    free1 = torch.cuda.mem_get_info()[0]
    ref = warm.matvec(J)
    try:
        assert (free0 - free1) / 3 < limit
        for op in ops:
            a = op.matvec(J)
            op.check()
            assert (a - ref).norm() < 1e-6 * ref.norm()
        # batch of problems whose items together are more than one's scratch has room for
        if kw:
            b = lmfmm.Batch(ops)
            outs = [torch.empty_like(J) for _ in ops]
            for tuned in (False, True):
                if tuned:
                    b.tune()
                b.matvec([J, J, J], outs)
                b.check()
                for a in outs:
                    assert (a - ref).norm() < 1e-6 * ref.norm()
            b.close()
    finally:
        for op in ops + [warm]:
            op.close()
