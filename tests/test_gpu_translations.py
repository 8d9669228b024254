"""The M2M / L2L matrices that a build forms on the device against those of the host routine
(long double, rounded once per entry).  GPU."""
import math

import numpy as np
import pytest

from paper_2507_18491_gb300 import lmfmm
from paper_2507_18491_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# the smallest and the largest order, real and lossy layers, every octant and level of the tree.
# Both sides round each entry once before the same scaling: two roundings of an entry of a degree
# block, 2^-52 of the block's largest one
@pytest.mark.parametrize("p", [1, 6, 12, 16])
def test_device_matrices(p):
    w = W.three_layer(n=300, p=p, depth=2)
    op = lmfmm.Operator(w.d, w.k, w.xyz, p=p, depth=2, theta=0.5, tensor_cores=0).build()
    groups = 0
    worst = 0.0
    try:
        while True:
            g = lmfmm.built_translation(op.ctx, p, groups)
            if g is None:
                break
            groups += 1
            layer, t, (sc, sp), up, dn = g
            ru, rd = lmfmm.translation_matrix(p, complex(w.k[layer]), tuple(t))
            for n in range(p + 1):
                for n1 in range(p + 1):
                    a, b = slice(n * n, (n + 1) ** 2), slice(n1 * n1, (n1 + 1) ** 2)
                    for got, ref, f in ((up, ru, math.pow(sc, n1) / math.pow(sp, n)),
                                        (dn, rd, math.pow(sc, n) / math.pow(sp, n1))):
                        ref = f * ref[a, b]
                        worst = max(worst, np.max(np.abs(got[a, b] - ref)) / np.max(np.abs(ref)))
    finally:
        op.close()
    print("p = %d: %d groups, worst entry %.2e of its degree block" % (p, groups, worst))
    assert groups >= 16 and worst < 2.0 ** -52
