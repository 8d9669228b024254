"""Device math of csrc/specfun.cuh compiled for the host (its qualifiers are empty there), against
mpmath.  CPU."""
import os
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_18491_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "specfun.cuh"
int main(int argc, char **)
{
    double x[2];
    while (argc > 1 && std::fread(x, sizeof x, 1, stdin) == 1) {
        const double r = sqrt_from_rsqrt(x[0], x[1]);
        std::fwrite(&r, sizeof r, 1, stdout);
    }
    cd z;
    while (std::fread(&z, sizeof z, 1, stdin) == 1) {
        cd S[4], M[5], h{bessel_series_holds(z) ? 1.0 : 0.0, 0.0};
        bessel_j_series<3>(z, S);
        bessel_j_seq<4>(z, 3, M);
        std::fwrite(&h, sizeof h, 1, stdout);
        std::fwrite(S, sizeof(cd), 4, stdout);
        std::fwrite(M, sizeof(cd), 4, stdout);
    }
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("specfun")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(HARNESS)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O2", "-x", "c++", "-I", CSRC, "-I", os.path.join(cuda, "include"),
                    str(src), "-o", str(exe)], check=True)
    return str(exe)


# annuli of the two areas in which the series runs: the real axis and below it (the paths of the
# integrals bend that way); the last of each ends at the limit
@pytest.mark.parametrize("lo,hi,slope", [(0.01, 1, 0), (1, 2, 0), (2, 3, 0), (3, 4, 0), (0.01, 1, 2), (1, 2, 2),
                                         (2, 3, 2), (3, 4, 2)])
def test_series_is_no_less_accurate_than_the_recurrence_where_it_runs(harness, lo, hi, slope):
    rng = np.random.default_rng(3)
    r = rng.uniform(lo, hi, 300)
    z = r * np.exp(-1j * np.arctan(slope * rng.uniform(0, 1, r.size)))
    if slope == 0:
        z = r + 0j
    out = subprocess.run([harness], input=z.tobytes(), stdout=subprocess.PIPE, check=True).stdout
    out = np.frombuffer(out, complex).reshape(-1, 9)
    runs = out[:, 0].real > 0
    assert runs.all() or not runs.any()
    if not runs.any():
        assert lo >= (2 if slope else 3)
        return
    err = np.zeros((2, z.size, 4))
    with mp.workdps(30):
        for i, v in enumerate(z):
            for n in range(4):
                b = mp.besselj(n, mp.mpc(v))
                for k in range(2):
                    err[k, i, n] = abs(mp.mpc(complex(out[i, 1 + 4 * k + n])) - b)
    rms = np.sqrt((err ** 2).mean(1))
    # of 300 errors each: an rms is known to 1 / sqrt(2 x 300) = 4%, a ratio to 6%; two of these
    assert (rms[0] < 1.12 * rms[1]).all(), rms


def test_distance_from_its_reciprocal_root(harness):
    """The near field forms R from rsqrt(R^2), which CUDA gives to an ulp: R rounded like sqrt, but
    for values next to a tie (2^-53 of an ulp's width in the correction's own rounding: rare)."""
    rng = np.random.default_rng(4)
    x = np.exp(rng.uniform(-20, 20, 20000))
    y = 1 / np.sqrt(x)
    y = np.where(rng.random(x.size) < 0.5, np.nextafter(y, 0), np.nextafter(y, np.inf))
    out = subprocess.run([harness, "r"], input=np.stack([x, y], 1).tobytes(), stdout=subprocess.PIPE, check=True).stdout
    r = np.frombuffer(out)
    assert (np.abs(x * y - np.sqrt(x)) > 0).mean() > 0.3      # without the step
    assert (r != np.sqrt(x)).mean() < 0.01
    assert (np.abs(r - np.sqrt(x)) <= np.spacing(np.sqrt(x))).all()
