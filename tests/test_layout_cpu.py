"""Device-memory layout of the host code, checked without a GPU: a probe that includes the host source
reports the byte ranges that a call touches."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from test_abi_cpu import W, _spec  # noqa: F401  (W: fixture)

PROBE = r"""
#include "wri_api.cu"

// Ends of the byte ranges that wri_gradient_noalloc writes in its static array: out[0] without the layer
// tables (z-march kernels: z tables, systems, receivers), out[1] with them (chunk kernels); out[2] and out[3]
// the sizes that it compares with its limit and with the array's for the two, out[4] the array's.
extern "C" __attribute__((visibility("default"))) void noalloc_ranges(const wri_group* groups, int ngroups,
                                                                      long long* out) {
  Plan P;
  plan_aux(groups, ngroups, P);
  size_t z = P.off_rec + sizeof(int) * (size_t)P.nnz_total;
  z = std::max(z, P.off_sys + sizeof(SysDev) * (size_t)P.nsys_total);
  size_t l = z;
  for (int gi = 0; gi < ngroups; ++gi) {
    const size_t nz = groups[gi].grid.nz, e = (size_t)kLayerTab * (groups[gi].grid.npml + 1);
    z = std::max(z, std::max(P.off_ztab[gi] + 48 * nz, P.off_ztab64[gi] + 96 * nz));
    l = std::max(l, std::max(P.off_ltab32[gi] + 4 * e, P.off_ltab64[gi] + 8 * e));
  }
  out[0] = (long long)z;
  out[1] = (long long)std::max(l, z);
  out[2] = (long long)P.aux_base;
  out[3] = (long long)P.aux_total;
  out[4] = (long long)sizeof(g_noalloc_scratch);
}

// Of a solve's plan: chunk kernels or not, iterations per iterate update, direction slots.
extern "C" __attribute__((visibility("default"))) void plan_of(const wri_group* groups, int ngroups,
                                                               const wri_solve_opts* opts, long long* out) {
  Plan P;
  plan_solve(groups, ngroups, opts, P);
  out[0] = P.lin ? 1 : 0;
  out[1] = P.xsteps;
  out[2] = P.pslots;
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
    subprocess.run([B.nvcc(), "-std=c++17", "-O1", "-Xcompiler", "-fPIC,-fvisibility=hidden", *B.ARCH, "-shared",
                    "-I", B.CSRC, "-o", lib, src, *objs], check=True, capture_output=True, text=True)
    return C.CDLL(lib)


@pytest.mark.parametrize("ngroups,npml", [(1, 10), (8, 20), (8, 226), (8, 300)])
def test_noalloc_gradient_stays_inside_its_array(W, probe, ngroups, npml):  # noqa: F811
    """The largest geometry that the limit of wri_gradient_noalloc accepts: the bytes that a call
    without layer tables touches end within the size compared with the limit, and those of a call with them
    within the size compared with the array's (npml = 300: 344 KB of tables, more than the array has for them)."""
    def ranges(nnz):
        specs = [_spec(W, nx=2 * npml + 1, ny=2 * npml + 1, nz=2 * npml + 1, npml=npml, src=np.array([0]),
                       rec_off=np.array([0, nnz]), rec_idx=np.arange(nnz, dtype=np.int32)) for _ in range(ngroups)]
        m = W._Marshal(specs)
        out = (C.c_longlong * 5)()
        probe.noalloc_ranges(m.arr, m.n, out)
        return list(out)

    limit = W.NOALLOC_SCRATCH_BYTES
    lo, hi = 1, limit // 4 // ngroups  # receivers per group
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (mid, hi) if ranges(mid)[2] <= limit else (lo, mid)
    plain, tables, base, total, size = ranges(lo)
    assert limit - 256 * ngroups < base <= limit < ranges(hi)[2]
    assert plain <= base and tables <= total and limit <= size


def test_initialised_barriers_are_fenced_before_copies_signal_them(W):  # noqa: F811
    """Every kernel that initialises mbarriers fences them for the async proxy, by the same thread, before the
    CTA's barrier (a CTA barrier alone does not order the two proxies; no run can be relied on to show it)."""
    from paper_2410_18429_gb300 import build as B
    kernels = 0
    for name in ("wri_tma.cuh", "wri_lin.cuh"):
        with open(os.path.join(B.CSRC, name)) as f:
            for part in f.read().split("__global__")[1:]:
                if "mbar_init(" in part:
                    kernels += 1
                    after = part[part.rindex("mbar_init("):]
                    assert 0 <= after.find("mbar_init_done();") < after.index("__syncthreads();"), (name, part[:120])
    assert kernels == 4


def _plan(W, probe, spec, **kw):  # noqa: F811
    m = W._Marshal([spec])
    out = (C.c_longlong * 3)()
    probe.plan_of(m.arr, m.n, C.byref(W.make_opts(**kw)), out)
    return tuple(out)


@pytest.mark.parametrize("dtype,grouped", [(0, 4), (1, 2)])
def test_iterations_per_iterate_update_of_the_chunk_configurations(W, probe, dtype, grouped):  # noqa: F811
    """18: every iteration (what the grouped configurations are compared with, bit for bit); 22: every second; 24 and
    the automatic choice: as many as there are direction slots."""
    for cfg, m in ((18, 1), (22, 2), (24, grouped)):
        lin, xsteps, slots = _plan(W, probe, _spec(W), dtype=dtype, kernel=W.KERNEL_TMA(cfg))
        assert (lin, xsteps) == (1, m) and slots == max(2, m), cfg
    assert _plan(W, probe, _spec(W), dtype=dtype, kernel=0)[:2] == (1, grouped)


def test_workspace_of_batches_that_the_boxes_cannot_take(W, probe):  # noqa: F811
    """An x extent that is not a multiple of 4: large batches have two direction slots, as on the z-march kernels, so
    that what fitted the device there fits it on the chunk kernels too (but for layer tables and the shape of the
    receiver bits); the two slots more of the others take at most 1 GiB."""
    def vectors(spec, **kw):  # complex64 vectors beyond the z-march workspace, in bytes per node and system
        n = spec.nx * spec.ny * spec.nz * len(spec.src)
        march = W.workspace_size([spec], W.make_opts(kernel=W.KERNEL_MARCH, **kw))
        return [round((W.workspace_size([spec], W.make_opts(kernel=k, **kw)) - march) / n) for k in (0, W.KERNEL_TMA(24))]

    for kw in (dict(), dict(max_refine=2, refine_tol=1e-8, inner_tol=1e-2)):
        for nx, ny, nz, slots in ((81, 80, 80, 4), (405, 408, 406, 4), (407, 410, 406, 2), (801, 400, 400, 2)):
            spec = _spec(W, nx=nx, ny=ny, nz=nz, src=np.array([0]), rec_off=np.array([0, 5]))
            assert _plan(W, probe, spec, kernel=0, **kw) == (1, slots, slots), nx
            assert vectors(spec, **kw) == [16 if slots == 4 else 0] * 2, nx
    assert _plan(W, probe, _spec(W, nx=21), dtype=1, kernel=0) == (1, 2, 2)
    assert _plan(W, probe, _spec(W, nx=400, ny=800, nz=400), kernel=0) == (1, 4, 4)
