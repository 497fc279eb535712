"""Layer table of the chunk kernels, checked without a GPU against 60-digit arithmetic."""
import ctypes as C
import os
import subprocess

import pytest

from test_abi_cpu import W, _spec  # noqa: F401  (W: fixture)

PROBE = r"""
#include "wri_api.cu"

// out: sigma_max, then the entries of the layer table.
extern "C" __attribute__((visibility("default"))) void table_of(const wri_grid* g, double* out) {
  std::vector<double> t;
  layer_table(*g, t);
  out[0] = axis(g->nx, *g).smax;
  std::copy(t.begin(), t.end(), out + 1);
}
"""


@pytest.fixture(scope="module")
def probe(W, tmp_path_factory):  # noqa: F811
    from paper_2410_18429_gb300 import build as B
    d = tmp_path_factory.mktemp("probe")
    src, lib = str(d / "probe.cu"), str(d / "probe.so")
    with open(src, "w") as f:
        f.write(PROBE)
    objs = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.SOURCES if s != "wri_api.cu"]
    subprocess.run([B.nvcc(), "-std=c++17", "-O3", "-Xcompiler", "-fPIC,-fvisibility=hidden", *B.ARCH, "-shared",
                    "-I", B.CSRC, "-o", lib, src, *objs], check=True, capture_output=True, text=True)
    return C.CDLL(lib)


@pytest.mark.parametrize("npml,h,omega", [(0, 10.0, 30.0), (1, 7.0, 2.0), (6, 10.0, 31.4159), (10, 26.6666666667, 50.3),
                                          (20, 50.0, 12.5), (33, 8.0, 400.0), (300, 1.25, 3.0)])
def test_entries_are_rounded_once(W, probe, npml, h, omega):  # noqa: F811
    """alpha of both half points, minus their sum, Im s and 1 / (s(half) h^2), from the profile
    s = 1 + i sigma_max (d / npml)^2 / omega: each within half a unit in the last place of the exact value for the same
    sigma_max, and 1e-6 of that for the arithmetic in two doubles.  (Complex FP64 divisions leave several.)"""
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 60
    grid = _spec(W, npml=npml, h=h, omega=omega).grid()
    out = (C.c_double * (1 + 12 * (npml + 1)))()
    probe.table_of(C.byref(grid), out)
    smax = mp.mpf(out[0])

    def stretch(d):
        return mp.mpc(1, smax * (mp.mpf(max(d, 0)) / npml) ** 2 / mp.mpf(omega)) if npml else mp.mpc(1)

    for d in range(npml + 1):
        s = stretch(d)
        half = [1 / (stretch(d + f) * mp.mpf(h) ** 2) for f in (-0.5, 0.5)]
        alpha = [v / s for v in half]
        a0 = -(alpha[0] + alpha[1])
        ref = [alpha[0].real, alpha[0].imag, alpha[1].real, alpha[1].imag, a0.real, a0.imag, s.imag, 0,
               half[0].real, half[0].imag, half[1].real, half[1].imag]
        for i, e in enumerate(ref):
            got = mp.mpf(out[1 + 12 * d + i])
            assert abs(got - e) <= (1 + mp.mpf("1e-6")) * mp.mpf(2) ** -53 * abs(e), (d, i)
