// Launchers of the chunk kernels (wri_lin.cuh).
#include "wri_launch.h"
#include "wri_lin.cuh"

namespace wri {

// Stage layout of a batch: the two fields' regions (a chunk and nx nodes on either side, one more element
// for the 16-byte boundary at each end) and the model's.
static size_t lin_layout(const Batch& b, int rbytes, int mode, LinSet& T) {
  const bool two = mode == M_P1 || mode == M_P2;
  int nx = 0;
  T.gz = 0;
  for (int g = 0; g < b.ngroups; ++g) {
    nx = b.g[g].nx > nx ? b.g[g].nx : nx;
    T.gz = b.g[g].zc > T.gz ? b.g[g].zc : T.gz;
  }
  const int cb = 2 * rbytes;
  const int field = ((kLinChunk + 2 * nx) * cb + 16 + 127) / 128 * 128;
  const int mod = (kLinChunk * (b.g[0].m_double ? 8 : 4) + 16 + 127) / 128 * 128;
  T.off_b = field;
  T.off_m = two ? 2 * field : field;
  T.stage = T.off_m + mod;
  size_t bytes = 128 + (size_t)kLinStages * (T.stage + 16);
  if (mode == M_GRAD) bytes += (size_t)T.gz * kLinChunk * 8;
  return bytes;
}

size_t lin_smem(const Batch& b, int rbytes, int mode) {
  LinSet T;
  return lin_layout(b, rbytes, mode, T);
}

template <typename R, typename OR, int MODE, bool CONJ, int NC, int NPT, bool PAIR, bool GV, int MINB,
          bool XO = (sizeof(R) == 8)>
static cudaError_t launch_one(const Batch& b, const LinWait& w, const LinTab<MODE>& tab, cudaStream_t st) {
  LinSet T;
  T.err = w.err;
  T.wait_ns = w.wait_ns;
  T.withhold = w.withhold;
  const size_t smem = lin_layout(b, sizeof(R), MODE, T);
  auto kern = k_lin<R, OR, MODE, CONJ, NC, NPT, PAIR, GV, kLinStages, MINB, XO>;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  static thread_local size_t occ_smem = 0;  // resident CTAs at the last shared-memory size and device
  static thread_local int occ_dev = -1, occ = 0, sms = 0;
  if (occ_smem != smem || occ_dev != dev) {
    occ_dev = -1;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kLinMaxSmem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, NC + 32, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    occ_smem = smem;
    occ_dev = dev;
  }
  const long long cap = (long long)sms * occ;
  const int grid = (int)(cap < b.nitems ? cap : b.nitems);
  kern<<<grid, NC + 32, smem, st>>>(b, T, tab);
  return cudaGetLastError();
}

// planes of the batch's longest items
static int longest(const Batch& b) {
  int zc = 0;
  for (int g = 0; g < b.ngroups; ++g) zc = b.g[g].zc > zc ? b.g[g].zc : zc;
  return zc;
}

cudaError_t launch_lin(int rbytes, int obytes, int mode, bool conj, const Batch& b, const LinWait& w,
                       const double* tab, int tab_n, cudaStream_t st) {
  if (b.nitems <= 0) return cudaSuccess;
#define WRI_LIN(M, CJ, R, OR, NC, NPT, PAIR, GV, MINB) \
  return launch_one<R, OR, M, CJ, NC, NPT, PAIR, GV, MINB>(b, w, LinTab<M>(), st);
#define WRI_LIN_F32(M, CJ, GV)                                  \
  if (b.pair) WRI_LIN(M, CJ, float, float, 128, 2, true, GV, 4) \
  else WRI_LIN(M, CJ, float, float, 128, 2, false, GV, 4)
  if (mode == M_APPLY) {
    if (tab_n > kLinInlineTab) return cudaErrorInvalidValue;
    LinTab<M_APPLY> t;
    t.n = tab_n;
    for (int i = 0; i < tab_n * kLayerTab; ++i) t.v[i] = tab[i];
#define WRI_LIN_APPLY(CJ)                                                                                 \
  if (rbytes == 8) return launch_one<double, double, M_APPLY, CJ, 256, 1, false, false, 2>(b, w, t, st);          \
  if (b.pair) return launch_one<float, float, M_APPLY, CJ, 128, 2, true, false, 4>(b, w, t, st);                  \
  return launch_one<float, float, M_APPLY, CJ, 128, 2, false, false, 4>(b, w, t, st);
    if (conj) {
      WRI_LIN_APPLY(true)
    }
    WRI_LIN_APPLY(false)
#undef WRI_LIN_APPLY
  }
  if (rbytes == 4) {
    switch (mode) {
      case M_P1: WRI_LIN_F32(M_P1, false, false)
      case M_P2:
        if (b.g[0].gvec) WRI_LIN_F32(M_P2, true, true)
        WRI_LIN_F32(M_P2, true, false)
      case M_SH: WRI_LIN_F32(M_SH, true, false)
      case M_RES: WRI_LIN_F32(M_RES, false, false)
    }
  } else {
    switch (mode) {
      // long items: a kind of loop more (see the kernel's step)
      case M_P1:
        if (longest(b) < 8)
          return launch_one<double, double, M_P1, false, 256, 1, false, false, 2, false>(b, w, LinTab<M_P1>(), st);
        WRI_LIN(M_P1, false, double, double, 256, 1, false, false, 2)
      case M_P2:
        if (longest(b) < 8)
          return launch_one<double, double, M_P2, true, 256, 1, false, false, 2, false>(b, w, LinTab<M_P2>(), st);
        WRI_LIN(M_P2, true, double, double, 256, 1, false, false, 2)
      case M_SH:
        if (obytes == 4) WRI_LIN(M_SH, true, double, float, 256, 1, false, false, 2)
        WRI_LIN(M_SH, true, double, double, 256, 1, false, false, 2)
      case M_RES: WRI_LIN(M_RES, false, double, double, 256, 1, false, false, 2)
      case M_GRAD: WRI_LIN(M_GRAD, false, double, double, 256, 1, false, false, 2)
    }
  }
#undef WRI_LIN
#undef WRI_LIN_F32
  return cudaErrorInvalidValue;
}

cudaError_t launch_init_point(int rbytes, int obytes, const Batch& b, int nsys_total, cudaStream_t st) {
  if (rbytes == 4) k_init_point<float, float><<<nsys_total, 128, 0, st>>>(b, nsys_total);
  else if (obytes == 8) k_init_point<double, double><<<nsys_total, 128, 0, st>>>(b, nsys_total);
  else k_init_point<double, float><<<nsys_total, 128, 0, st>>>(b, nsys_total);
  return cudaGetLastError();
}

// One array per blockIdx.y, zeroed in 16-byte stores (8-byte ones at an unaligned start and the end).
__global__ void k_zero(const __grid_constant__ ZeroSet z) {
  unsigned char* p = (unsigned char*)z.p[blockIdx.y];
  const long long bytes = z.bytes[blockIdx.y];
  const long long head = ((uintptr_t)p & 15) ? 8 : 0, mid = (bytes - head) / 16;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
  for (long long e = t; e < mid; e += step) *(uint4*)(p + head + 16 * e) = make_uint4(0u, 0u, 0u, 0u);
  if (t == 0 && head) *(uint2*)p = make_uint2(0u, 0u);
  if (t == 0 && head + 16 * mid < bytes) *(uint2*)(p + head + 16 * mid) = make_uint2(0u, 0u);
}

cudaError_t launch_zero(const ZeroSet& z, cudaStream_t st) {
  long long most = 0;
  for (int i = 0; i < z.count; ++i) most = z.bytes[i] > most ? z.bytes[i] : most;
  if (most <= 0) return cudaSuccess;
  const long long blocks = (most / 16 + 1023) / 1024;  // 4 x 256 16-byte stores per block
  k_zero<<<dim3((unsigned)(blocks < 1 ? 1 : blocks < 152 * 8 ? blocks : 152 * 8), z.count), 256, 0, st>>>(z);
  return cudaGetLastError();
}

cudaError_t launch_point_field(int rbytes, const Batch& b, int gi, cudaStream_t st) {
  const int grid = (b.g[gi].nsys + 127) / 128;
  if (rbytes == 8) k_point_field<double><<<grid, 128, 0, st>>>(b, gi);
  else k_point_field<float><<<grid, 128, 0, st>>>(b, gi);
  return cudaGetLastError();
}

cudaError_t launch_xupdate(int rbytes, const Batch& b, cudaStream_t st) {
  if (b.xitems <= 0) return cudaSuccess;
  const int grid = (int)(b.xitems < 152 * 8 ? b.xitems : 152 * 8);
  bool wide = rbytes == 4;
  for (int g = 0; g < b.ngroups; ++g) wide = wide && b.g[g].n % 2 == 0 && (uintptr_t)b.g[g].x % 16 == 0;
  if (rbytes == 8) k_xupdate<double, 1><<<grid, 256, 0, st>>>(b);
  else if (wide) k_xupdate<float, 2><<<grid, 256, 0, st>>>(b);
  else k_xupdate<float, 1><<<grid, 256, 0, st>>>(b);
  return cudaGetLastError();
}

}  // namespace wri
