"""Performance cases of the layered-media Maxwell FMM, through its public entry points.

A case is one call that a program using the library makes again and again:

  matvec  Phi = A J of a built operator (an iterative solver's step),
  vjp     (A^H g, Re sum conj(g) dE/dr): the backward pass of an optimisation over
          currents and positions (it runs the forward pass again, so it stands for both),
  cold    set-up of a new geometry, one matvec and release (moving points, a scan over
          media): the quantity the paper's own timings measure,
  batch   many small problems applied together.

The point sets, media, truncations and admissibility parameters are those of the
repository's workloads (paper_2507_18491_gb300/workloads.py) and of its benchmark.
The FP64 form takes complex128 currents and the mixed form complex64 ones, the element
type that its accuracy corresponds to.
"""
import math

import numpy as np
import torch

from paper_2507_18491_gb300 import lmfmm
from paper_2507_18491_gb300 import workloads as W

DEVICE = "cuda:0"


def _case(name, call, points, n, p, depth, theta, form, tensor_cores=1, components="reaction", problems=1):
    return {"name": name, "call": call, "points": points, "n": n, "p": p, "depth": depth, "theta": theta,
            "form": form, "tensor_cores": tensor_cores, "components": components, "problems": problems}


def listed():
    return [
        # the smallest configuration: two layers, 512 points; launches and latency
        _case("matvec_two_layer_n512_fp64", "matvec", "two_layer", 512, 6, 2, 0.4, "fp64"),
        # a small ragged problem in the library's default mixed form
        _case("matvec_three_layer_n10007_mixed", "matvec", "three_layer", 10007, 7, 4, 0.55, "mixed"),
        # the three-layer medium in double precision, the form that meets 1e-6 everywhere
        _case("matvec_three_layer_n4096_fp64", "matvec", "three_layer", 4096, 10, 3, 0.5, "fp64"),
        # the three-layer configuration's points in the mixed form with the default tensor-core M2L
        _case("matvec_three_layer_n65536_mixed", "matvec", "three_layer", 65536, 8, 5, 0.5, "mixed"),
        # the benchmark's order, all translations on the tensor cores, crowded leaves
        _case("matvec_three_layer_n3001_mixed", "matvec", "three_layer", 3001, 12, 3, 0.5, "mixed", 3),
        # the four-layer clustered medium: uneven leaves, points next to the interfaces
        _case("matvec_clusters_n131072_mixed", "matvec", "clusters", 131072, 8, 5, 0.55, "mixed", 3),
        # the largest point set: the paper's two-layer table, 10^6 points per layer
        _case("matvec_paper2_n2000000_mixed", "matvec", "paper2", 2000000, 8, 5, 0.55, "mixed", 3),
        # reaction and free-space parts together (the whole field)
        _case("matvec_total_paper2_n9998_mixed", "matvec", "paper2", 9998, 6, 4, 0.55, "mixed", components="total"),
        # gradient with respect to currents and positions (inverse design), double precision
        _case("vjp_three_layer_n16384_fp64", "vjp", "three_layer", 16384, 6, 4, 0.55, "fp64"),
        # a new geometry each time, at the paper's size (10^4 points per layer)
        _case("cold_paper2_n20000_fp64", "cold", "paper2", 20000, 6, 4, 0.55, "fp64"),
        # a new geometry with near pairs across the interface, mixed form
        _case("cold_three_layer_n8192_mixed", "cold", "three_layer", 8192, 6, 4, 0.55, "mixed"),
        # uneven small problems of several media in one call
        _case("batch_2_mixed", "batch", "batch", 3001, 8, 3, 0.55, "mixed", problems=2),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("two_layer", "three_layer", "clusters", "paper2", "total", "vjp", "cold", "batch"))
    form = rng.choice(("fp64", "mixed"))
    tc = rng.choice((1, 3))
    theta = rng.choice((0.45, 0.5, 0.55))
    p = rng.randint(6, 10)
    if kind == "two_layer":
        n = _log_uniform(rng, 200, 8000)
        c = _case("", "matvec", kind, n, rng.randint(6, 12), 2 if n < 1500 else 3, theta, form, tc)
    elif kind == "three_layer":
        n = _log_uniform(rng, 1500, 40000)
        c = _case("", "matvec", kind, n, rng.randint(6, 12) if n < 4000 else min(p, 8), 3 if n < 4000 else 4, theta,
                  form, tc)
    elif kind == "clusters":
        c = _case("", "matvec", kind, _log_uniform(rng, 20000, 120000), min(p, 8), 5, 0.55, "mixed", tc)
    elif kind == "paper2":
        n = _log_uniform(rng, 3000, 1500000)
        c = _case("", "matvec", kind, n, p, 4 if n < 100000 else 5, theta,
                  "mixed" if n > 100000 else form, tc)
    elif kind == "total":
        c = _case("", "matvec", "paper2", _log_uniform(rng, 3000, 12000), min(p, 7), 4, 0.55, form, tc, "total")
    elif kind == "vjp":
        n = _log_uniform(rng, 1000, 25000)
        c = _case("", "vjp", "three_layer", n, min(p, 7), 3 if n < 4000 else 4, 0.55, "fp64")
    elif kind == "cold":
        n = _log_uniform(rng, 2000, 9000)
        c = _case("", "cold", rng.choice(("paper2", "three_layer")), n, min(p, 7), 3 if n < 4000 else 4, 0.55, form, tc)
    else:
        c = _case("", "batch", "batch", _log_uniform(rng, 1500, 4000), min(p, 8), 3, 0.55, "mixed", tc,
                  problems=rng.randint(2, 3))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _workloads(case, seed):
    """The point sets, media and currents of a case (one, or one per batched problem)."""
    n, p = case["n"], case["p"]
    seed = int(seed) % (1 << 31)
    kind = case["points"]
    if kind == "two_layer":
        return [W.two_layer_small(n=n, seed=seed)]
    if kind == "three_layer":
        return [W.three_layer(n=n, seed=seed, p=p)]
    if kind == "clusters":
        return [W.four_layer_clusters(n=n, seed=seed, p=p)]
    if kind == "paper2":
        return [W.paper_table_uniform(m=n // 2, layers=2, seed=seed, p=p)]
    # uneven sizes: n, n / 2, n / 3, ...; two or three layers, wavenumbers in [0.5, 4]
    return [W.batch_problems(n_problems=1, seed=seed + i, n_min=n // (i + 1), n_max=n // (i + 1), p=p)[0]
            for i in range(case["problems"])]


def _operator(case, w):
    return lmfmm.Operator(w.d, w.k, w.xyz, p=case["p"], depth=case["depth"], theta=case["theta"],
                          precision=lmfmm.FP64 if case["form"] == "fp64" else lmfmm.MIXED,
                          tensor_cores=case["tensor_cores"],
                          components=lmfmm.TOTAL if case["components"] == "total" else lmfmm.REACTION)


def _currents(case, J):
    return torch.from_numpy(J).to(DEVICE).to(torch.complex128 if case["form"] == "fp64" else torch.complex64)


def _upstream(n, seed):
    """dL/dconj(E) of a vjp case."""
    rng = np.random.default_rng([int(seed) % (1 << 31), 7])
    return torch.from_numpy(rng.standard_normal((n, 3)) + 1j * rng.standard_normal((n, 3))).to(DEVICE)


def prepare(case, seed):
    ws = _workloads(case, seed)
    Js = [_currents(case, w.J) for w in ws]
    state = {"call": case["call"], "J": Js}
    if case["call"] == "cold":
        state["new"] = lambda: _operator(case, ws[0])
        return state
    state["ops"] = [_operator(case, w).build() for w in ws]
    state["out"] = [torch.empty_like(J) for J in Js]
    if case["call"] == "vjp":
        state["g"] = _upstream(ws[0].N, seed)
    elif case["call"] == "batch":
        state["batch"] = lmfmm.Batch(state["ops"])
    return state


def run(state):
    call = state["call"]
    if call == "matvec":
        return state["ops"][0].matvec(state["J"][0], out=state["out"][0])
    if call == "vjp":
        return state["ops"][0].vjp(state["J"][0], state["g"])
    if call == "batch":
        return state["batch"].matvec(state["J"], state["out"])
    op = state["new"]().build()
    phi = op.matvec(state["J"][0])
    op.close()
    return phi


# -------------------------------------------------------------------- work
def work(case):
    """Caller's buffers once, and the arithmetic of the FMM's own counts: per far pair the
    3 x 3 helical translation (36 P^2 flops: the pair's vertical plane of symmetry splits the
    operator into two halves of 3P/2), per tree edge and helical component one P x P matrix
    each way, per point the three expansions each way, 9 complex products per near point pair."""
    nbytes = flops = 0.0
    elem = 16 if case["form"] == "fp64" else 8
    P = (case["p"] + 1) ** 2
    for w in _workloads(case, 1):
        rc, pl = lmfmm.plan_check(w.d, w.k, w.xyz, p=case["p"], depth=case["depth"], theta=case["theta"],
                                  components=lmfmm.TOTAL if case["components"] == "total" else lmfmm.REACTION)
        if rc != lmfmm.OK:
            raise ValueError("plan_check: %s" % pl["message"])
        one = (36.0 * P * P * (pl["n_far_pairs"] + pl["n_free_far_pairs"]) +
               2 * 3 * 8.0 * P * P * pl["n_translation_pairs"] + 2 * 3 * 8.0 * P * w.N +
               72.0 * (pl["n_near_point_pairs"] + pl["n_free_near_point_pairs"]))
        if case["call"] == "vjp":
            # forward pass, transposed pass, nine directional derivatives of the leaf sums
            flops += 2 * one + 9 * 8.0 * P * w.N
            nbytes += w.N * (3 * 3 * elem + 24 + 24)
        else:
            flops += one
            nbytes += w.N * (2 * 3 * elem + 24)
        if case["call"] == "cold":
            # every table entry from its p + 2 Chebyshev integrals
            flops += 36.0 * P * P * (case["p"] + 2) * pl["n_geometries"]
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------- exact
# The dyadic Green's function of a layered medium as a sum of plane waves: e^{ikR}/(4 pi R)
# = i/(8 pi^2) int d^2k / k_z e^{i k.(x-x') + i k_z |z-z'|}, transverse electric and magnetic
# parts, the scattered waves of every layer from the interface conditions, the radial integral
# on a path below the real axis.  The kernel is G(r_j, r_i) J_j (first slot summed).
_CUT = 27.0          # e^-27: the relative size of the waves left out
_MOST = 4.0e10       # points x waves: about 20 s


def _waves(d, k, reach, dz):
    """Radial nodes and weights (k dk), and the number of directions of each node."""
    a = 1.5 * np.max(np.abs(k)) + 0.75
    kmax = max(2 * a, _CUT / dz + np.max(np.abs(k)))
    x, w = np.polynomial.legendre.leggauss(16)

    def panels(lo, hi, n):
        e = np.linspace(lo, hi, n + 1)
        h = np.diff(e)[:, None] / 2
        return (e[:-1, None] + h * (1 + x)).ravel(), (h * w).ravel()

    t1, w1 = panels(0.0, a, 12 + int(a * reach / 4))
    dip = min(0.5 * a, 2.0 / reach)
    n1 = t1 - 1j * dip * np.sin(np.pi * t1 / a)
    w1 = w1 * (1 - 1j * dip * np.pi / a * np.cos(np.pi * t1 / a))
    t2, w2 = panels(a, kmax, 4 + int((kmax - a) * reach / 6))
    q = np.concatenate([n1, t2])
    m = 2 * np.ceil((np.abs(q) * reach + 12 * (np.abs(q) * reach) ** (1 / 3) + 40) / 2).astype(int)
    return q, np.concatenate([w1, w2]) * q, m


def _scattered(d, kz, Y):
    """C[(m, b), (l, a)] per node: amplitude, at its interface, of the wave seen from side b (0 top:
    down-going, 1 bottom: up-going) of layer m, for a unit wave from layer l meeting its side a."""
    L, Q = len(d), kz.shape[0]
    e = np.ones((Q, L + 1), complex)
    for j in range(1, L):
        e[:, j] = np.exp(1j * kz[:, j] * (d[j - 1] - d[j]))
    A = np.zeros((Q, 2 * L, 2 * L), complex)   # unknowns: up-going of layers 0..L-1, down-going of 1..L
    R = np.zeros((Q, 2 * L, L + 1, 2), complex)
    for j in range(L):
        up, dn = j, L + j
        A[:, 2 * j, up], A[:, 2 * j + 1, up] = 1, Y[:, j]
        A[:, 2 * j, dn], A[:, 2 * j + 1, dn] = -1, Y[:, j + 1]
        if j >= 1:
            A[:, 2 * j, dn - 1], A[:, 2 * j + 1, dn - 1] = e[:, j], -Y[:, j] * e[:, j]
        if j + 1 < L:
            A[:, 2 * j, up + 1], A[:, 2 * j + 1, up + 1] = -e[:, j + 1], -Y[:, j + 1] * e[:, j + 1]
        R[:, 2 * j, j, 1], R[:, 2 * j + 1, j, 1] = -1, Y[:, j]
        R[:, 2 * j, j + 1, 0], R[:, 2 * j + 1, j + 1, 0] = 1, Y[:, j + 1]
    S = np.linalg.solve(A, R.reshape(Q, 2 * L, -1)).reshape(Q, 2 * L, L + 1, 2)
    C = np.zeros((Q, L + 1, 2, L + 1, 2), complex)
    C[:, :L, 1] = S[:, :L]
    C[:, 1:, 0] = S[:, L:]
    return C


def _reaction(d, k, xyz, J, grads=None):
    """Reaction field of the currents J at the points; with grads = (g, gJ, gx) the gradients of
    Re sum conj(g) E with respect to J and the points are added into gJ and gx instead."""
    d, k = np.asarray(d, float), np.asarray(k, complex)
    L = len(d)
    pts = xyz.detach().cpu().numpy()
    lay = np.sum(pts[:, 2:3] < d[None, :], axis=1)
    reach = float(np.hypot(np.ptp(pts[:, 0]), np.ptp(pts[:, 1])))
    dz = 2 * float(np.min(np.abs(pts[:, 2:3] - d[None, :])))
    q, wq, m = _waves(d, k, reach, dz)
    if float(np.sum(m)) * len(pts) * (4 if grads else 1) > _MOST:
        return None
    kz = np.sqrt(k[None, :] ** 2 - q[:, None] ** 2 + 0j)
    kz = np.where(kz.imag < 0, -kz, kz)
    C = [_scattered(d, kz, Y) for Y in (kz, kz / k[None, :] ** 2)]
    dev, cplx = xyz.device, torch.complex128
    idx = [torch.from_numpy(np.flatnonzero(lay == l)).to(dev) for l in range(L + 1)]
    sides = [(l, s) for l in range(L + 1) if len(idx[l]) for s in (0, 1) if not (l == 0 and s == 0) and not (l == L and s == 1)]
    E = torch.zeros(len(pts), 3, dtype=cplx, device=dev)
    step = max(1, int(2.0e8 / len(pts)))     # waves (of one half circle) at a time
    half = m // 2
    node = np.repeat(np.arange(len(q)), half)
    ang = np.concatenate([np.arange(h) * np.pi / h for h in half])
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)  # noqa: E731
    for at in range(0, len(node), step):
        nd, al = node[at:at + step], ang[at:at + step]
        # each direction and its opposite: e^{ik.x} of one is the other's e^{-ik.x}
        nd2 = np.concatenate([nd, nd])
        ca, sa = np.concatenate([np.cos(al), -np.cos(al)]), np.concatenate([np.sin(al), -np.sin(al)])
        pre = t(1j / (8 * np.pi ** 2) * wq[nd2] * np.pi / half[nd2])
        tca, tsa, tq = t(ca), t(sa), t(q[nd2])
        n = len(nd)

        def chunk(x, j):
            lat = 1j * (x[:, :1] * (tq * tca)[None, :n] + x[:, 1:2] * (tq * tsa)[None, :n])
            F, pol, S = {}, {}, {}
            for l, s in sides:
                tkz = t(kz[nd2, l])
                z = x[idx[l], 2:3]
                vert = 1j * (tkz[None, :n] * ((d[l - 1] - z) if s == 0 else (z - d[l])))
                fwd, bwd = torch.exp(lat[idx[l]] + vert), torch.exp(vert - lat[idx[l]])
                F[l, s] = (bwd, fwd)
                sg = 1.0 if s == 1 else -1.0
                # polarisations of the wave seen at this side (up-going at the bottom side)
                see = torch.stack([-sg * tkz * tca, -sg * tkz * tsa, tq], 1) / complex(k[l])
                src = torch.stack([sg * tkz * tca, sg * tkz * tsa, tq], 1) / complex(k[l])
                pol[l, s] = (see, src)
                S[l, s] = torch.cat([fwd.T @ j[idx[l]], bwd.T @ j[idx[l]]])
            te = torch.stack([-tsa, tca, torch.zeros_like(tca)], 1).to(cplx)
            out = torch.zeros(len(x), 3, dtype=cplx, device=dev)
            for l, a in sides:
                amp = 0
                for mm, b in sides:
                    see, src = pol[mm, b][0], pol[l, a][1]
                    cte, ctm = t(C[0][nd2, mm, b, l, a]), t(C[1][nd2, mm, b, l, a] * k[l] / k[mm])
                    amp = amp + te * (cte * (te * S[mm, b]).sum(1))[:, None] + see * (ctm * (src * S[mm, b]).sum(1))[:, None]
                amp = (pre / t(kz[nd2, l]))[:, None] * amp
                bwd, fwd = F[l, a]
                out = out.index_add(0, idx[l], bwd @ amp[:n] + fwd @ amp[n:])
            return out

        if grads is None:
            E += chunk(xyz, J)
        else:
            g, gJ, gx = grads
            x, j = xyz.clone().requires_grad_(True), J.clone().requires_grad_(True)
            a, b = torch.autograd.grad((g.conj() * chunk(x, j)).sum().real, (j, x))
            gJ += a
            gx += b
    return E


def _free(d, k, xyz, J):
    """Free-space part: closed-form dyad over the other points of the same layer."""
    E = torch.zeros_like(J)
    lay = (xyz[:, 2:3] < torch.as_tensor(np.asarray(d, float), device=xyz.device)[None, :]).sum(1)
    for l in range(len(k)):
        at = torch.nonzero(lay == l)[:, 0]
        x, j, kl = xyz[at], J[at], complex(k[l])
        for c in range(0, len(at), 512):
            r = x[c:c + 512, None, :] - x[None, :, :]
            R = r.square().sum(2).sqrt()
            own = R == 0
            R = torch.where(own, torch.ones_like(R), R)
            g = torch.where(own, torch.zeros_like(R), 1 / (4 * np.pi * R)) * torch.exp(1j * kl * R)
            a = 1 + (1j * kl / R - 1 / R ** 2) / kl ** 2
            b = (3 / R ** 2 - 3j * kl / R - kl ** 2) / kl ** 2 / R ** 2
            rj = (r * j[None, :, :]).sum(2)
            E[at[c:c + 512]] += (g * a) @ j + ((g * b * rj)[:, :, None] * r).sum(1)
    return E


def exact(case, seed):
    if case["points"] == "clusters":
        return None      # points 0.01 from an interface: some 10^7 plane waves
    out = []
    for w in _workloads(case, seed):
        xyz = torch.from_numpy(w.xyz).to(DEVICE)
        J = _currents(case, w.J).to(torch.complex128)
        if case["call"] == "vjp":
            gJ, gx = torch.zeros_like(J), torch.zeros_like(xyz)
            if _reaction(w.d, w.k, xyz, J, (_upstream(w.N, seed), gJ, gx)) is None:
                return None
            return gJ, gx
        E = _reaction(w.d, w.k, xyz, J)
        if E is not None and case["components"] == "total":
            E += _free(w.d, w.k, xyz, J)
        out.append(E)
    return out if case["call"] == "batch" else out[0]
