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


def _near_centre(height, spread, k, offset=0.0):
    """Points within `spread` of the centre of a cell of side 1 that lies `height` above an interface,
    and points elsewhere that span the root cell [-1, 1]^3: the image of the cell's centre is 2 height
    away, a small part of the cell's side, and still far from the points by their radius."""
    rng = np.random.default_rng(9)
    near = 0.5 + offset + spread * rng.uniform(-1, 1, (12, 3))
    wide = np.array([[1, -1, -1], [-1, 1, -1], [-1, -1, 1], [-1, -1, -1]], float) * (1 - 1e-9)
    below = np.array([0.5, 0.5, 0.5 - 2 * height]) + offset + spread * rng.uniform(-1, 1, (12, 3))
    xyz = np.concatenate([near, wide, below])
    J = rng.standard_normal(xyz.shape) + 1j * rng.standard_normal(xyz.shape)
    return [0.5 - height], k, xyz, J


# the tables' entries grow like (side / distance)^(n + nu), the expansions fall like
# (radius / side)^n: the products are of ordinary size, but a grid set by each side's own largest
# entry has no bits left for them (46% of the result at p = 12, height 0.02).  Forward and
# transposed; 1e-13 as above
@pytest.mark.parametrize("p,height,spread", [(8, 0.1, 0.01), (12, 0.1, 0.01), (16, 0.1, 0.01), (12, 0.02, 0.002),
                                             (16, 0.02, 0.002)])
def test_expansions_far_inside_their_cells(p, height, spread):
    _compare(p, height, spread, 1)


# the same through M2M and L2L: at the cell, the expansions' high degrees are what the truncated
# translations leave there, not (radius / side)^n, and a grid that follows the radius gives its bits to
# them (74% off).  The points lie in one octant, so that every box has one child and both operators form the same expansions
@pytest.mark.parametrize("p,height,offset", [(6, 0.4, 4e-6), (8, 0.4, 1.5e-4)])
def test_translated_expansions_far_inside_their_cells(p, height, offset):
    _compare(p, height, offset / 8, 4, offset)


def _compare(p, height, spread, depth, offset=0.0):
    d, k, xyz, J = _near_centre(height, spread, [1.3 + 0.01j, 2.1 + 0.02j], offset)
    Jt = torch.from_numpy(J).cuda()
    out = []
    for tc in (1, 0):
        op = lmfmm.Operator(d, k, xyz, p=p, depth=depth, theta=0.5, tensor_cores=tc).build()
        assert op.stats()["m2l_digits"] == tc
        out.append((op.matvec(Jt), op.tmatvec(Jt)))
        ref = op.direct(Jt)
        op.close()
    for a, b in zip(*out):
        print("p %d height %g: digits against SIMT %.2e" % (p, height, (a - b).norm() / b.norm()))
    print("against the sum over all pairs: digits %.2e SIMT %.2e" %
          ((out[0][0] - ref).norm() / ref.norm(), (out[1][0] - ref).norm() / ref.norm()))
    for a, b in zip(*out):
        assert (a - b).norm() < 1e-13 * b.norm()
