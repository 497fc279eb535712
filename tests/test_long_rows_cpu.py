"""Plans of complex64 solves on grids with long rows of x, checked without a GPU."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from test_abi_cpu import W, _spec  # noqa: F401  (W: fixture)

PROBE = r"""
#include "wri_api.cu"

// Of a solve's plan: chunk kernels or not, configuration of the boxes, work items, shared memory of a CTA of phase 1.
extern "C" __attribute__((visibility("default"))) void plan_of(const wri_group* groups, int ngroups,
                                                               const wri_solve_opts* opts, long long* out) {
  Plan P;
  plan_solve(groups, ngroups, opts, P);
  Batch b;
  b.ngroups = ngroups;
  for (int gi = 0; gi < ngroups; ++gi) b.g[gi] = P.g[gi];
  out[0] = P.lin ? 1 : 0;
  out[1] = P.tma_cfg;
  out[2] = P.nitems;
  out[3] = (long long)lin_smem(b, 4, M_P1);
}
"""


@pytest.fixture(scope="module")
def plan(W, tmp_path_factory):  # noqa: F811
    from paper_2410_18429_gb300 import build as B
    d = tmp_path_factory.mktemp("probe")
    src, lib = str(d / "probe.cu"), str(d / "probe.so")
    with open(src, "w") as f:
        f.write(PROBE)
    objs = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.SOURCES if s != "wri_api.cu"]
    subprocess.run([B.nvcc(), "-std=c++17", "-O1", "-Xcompiler", "-fPIC,-fvisibility=hidden", *B.ARCH, "-shared",
                    "-I", B.CSRC, "-o", lib, src, *objs], check=True, capture_output=True, text=True)
    probe = C.CDLL(lib)

    def run(nx, ny, nz, nsys=1, **kw):
        spec = _spec(W, nx=nx, ny=ny, nz=nz, npml=10, src=np.arange(nsys) + 5, rec_off=np.arange(nsys + 1),
                     rec_idx=np.zeros(nsys, np.int32))
        m = W._Marshal([spec])
        out = (C.c_longlong * 4)()
        probe.plan_of(m.arr, m.n, C.byref(W.make_opts(**kw)), out)
        return tuple(out)

    return run


@pytest.mark.parametrize("nx", [276, 448, 512, 628])
@pytest.mark.parametrize("ny,nsys", [(40, 1), (40, 2), (64, 1), (120, 1), (120, 2)])
def test_z_chunks_count_the_resident_ctas(plan, nx, ny, nsys):
    """An SM holds four CTAs of the chunk kernels by their registers and fewer by the stages of long rows (228 KB of
    shared memory, 1 KB of it taken per CTA): the z-chunks minimise the modelled cost for waves of that many."""
    lin, _, items, smem = plan(nx, ny, ny, nsys)
    assert lin == 1
    wave = 152 * min(4, (228 << 10) // (smem + 1024 + 128))
    columns = nsys * -(-nx * ny // 256)

    def cost(zc):
        n = columns * -(-ny // zc)
        return (-(-n // wave) + n / wave) * (zc + 6)

    best = min(cost(-(-ny // zs)) for zs in range(1, min(ny, 64) + 1))
    zc = -(-ny // (items // columns))
    assert items % columns == 0 and cost(zc) <= best * (1 + 1e-12), (items, wave)


@pytest.mark.parametrize("refined", [{}, dict(max_refine=1, refine_tol=1e-8, inner_tol=1e-2)])
def test_long_rows_run_on_the_boxes(plan, refined):
    """Below three CTAs per SM (rows of 632 nodes) the boxes are faster where they can take the batch: x extents that
    are multiples of 4, complex64."""
    assert plan(628, 40, 40, kernel=0, **refined)[0] == 1
    for nx in (632, 768, 1600):
        assert plan(nx, 40, 40, kernel=0, **refined)[:2] == (0, 9), nx
        for cfg in (18, 22, 24):
            assert plan(nx, 40, 40, kernel=2 + cfg, **refined)[:2] == (0, cfg), nx
    assert plan(630, 40, 40, kernel=0, **refined)[0] == plan(770, 40, 40, kernel=0, **refined)[0] == 1
    assert plan(768, 40, 40, kernel=0, dtype=1)[0] == 1
