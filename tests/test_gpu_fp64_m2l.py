"""The digit M2L of the FP64 form (k_m2l_oz) against the FP64 SIMT kernels, which work on the five
tables and share no code with it.  GPU."""
import numpy as np
import pytest
import torch

from paper_2507_18491_gb300 import lmfmm
from paper_2507_18491_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# every number of matrix tiles and remainders (16-row steps) of p = 1..16; all layers' pairs,
# mirrored boxes on either side, item sizes from one pair on.  Both are FP64 sums of the same tables
# (each within K u = 884 x 1.1e-16 of the exact one, in practice sqrt(K) u = 3e-15 before the sums'
# cancellation): 1e-13
@pytest.mark.parametrize("p", [1, 2, 5, 8, 12, 16])
def test_digits_against_simt(p):
    w = W.three_layer(n=1503, p=p, depth=3)
    J = torch.from_numpy(w.J).cuda()
    rng = np.random.default_rng(p)
    y = torch.from_numpy(rng.standard_normal((w.N, 3)) + 1j * rng.standard_normal((w.N, 3))).cuda()
    out = []
    for tc in (1, 0):
        op = lmfmm.Operator(w.d, w.k, w.xyz, p=p, depth=3, theta=0.5, tensor_cores=tc).build()
        assert op.stats()["m2l_kernel"] == 0 and op.stats()["m2l_digits"] == tc
        out.append((op.matvec(J), op.tmatvec(y), op.rmatvec(y)))
        op.check()
        op.close()
    for a, b in zip(*out):
        assert (a - b).norm() < 1e-13 * b.norm()
