// Allocation-free variant of the fused step kernel (cavity_step_block_noalloc
// in include/cavity.h).
//
// Some callers cannot call cudaMalloc: code that runs inside another
// framework's memory pool or a pre-sized arena, where allocating from the
// driver behind that allocator's back would break its accounting or its
// out-of-memory handling.  This entry point lets such a caller run one fused
// residual + update pass over one block it already holds in device memory:
// the caller passes the input state, the output state and a 6-double output,
// and the reduction scratch the kernel needs lives in a fixed array compiled
// into the library (g_noalloc_scratch below), so no call allocates anything.
//
// The array exists once per GPU that loads the library and stays allocated
// until the process exits.  Every call shares it and it keeps the previous
// call's contents; each call overwrites all of it that it reads (descriptors
// and one partial slot per CTA), so nothing needs clearing.  Two calls whose
// work overlaps on a GPU (on different streams, or from different threads)
// race on the array and give wrong results.
//
// The paper has no counterpart: it describes no memory-management constraint.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "../../include/cavity.h"
#include "bdc_device.cuh"

using namespace bdc;

namespace {

constexpr int kTX = 32, kTY = 8, kKC = 16;  // the tile the size limit is stated in
constexpr int kDescBytes = 1280;           // BlockDev (256) + CavConst (768) + CavState (256), aligned slots
constexpr size_t kScratchBytes = kDescBytes + (size_t)CAVITY_NOALLOC_MAX_TILES * kPartStride * sizeof(double);
constexpr int kMaxDevices = 64;

static_assert(sizeof(BlockDev) <= 256 && sizeof(CavConst) <= 768 && sizeof(CavState) <= 256,
              "descriptor slots too small");

// reduction scratch and descriptors of the allocation-free entry point
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

std::mutex g_setup_mutex;
void *g_scratch_ptr[kMaxDevices] = {};

// Device address of g_noalloc_scratch on the current device, looked up once
// per device (the host-side name of the array is not a device address).
cudaError_t scratch_address(int dev, void **out) {
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_scratch_ptr[dev]) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

// Writes the three descriptors into the scratch array.  They arrive as kernel
// parameters, which the launch copies by value, so the call reads no host
// memory after it returns and makes no host-to-device copy of its own.
struct Descriptors {
  BlockDev B;
  CavConst C;
  CavState S;
};
__global__ void __launch_bounds__(128) k_noalloc_setup(const __grid_constant__ Descriptors d, BlockDev *d_block,
                                                       CavConst *d_cc, CavState *d_cs) {
  chain_trigger();  // (the step's launch waits for this one before it reads anything)
  auto copy = [](void *to, const void *from, int bytes) {
    for (int n = threadIdx.x; n < bytes / 8; n += 128)
      static_cast<unsigned long long *>(to)[n] = static_cast<const unsigned long long *>(from)[n];
  };
  static_assert(sizeof(BlockDev) % 8 == 0 && sizeof(CavConst) % 8 == 0 && sizeof(CavState) % 8 == 0, "whole words");
  copy(d_block, &d.B, sizeof(BlockDev));
  copy(d_cc, &d.C, sizeof(CavConst));
  copy(d_cs, &d.S, sizeof(CavState));
}

// RMS of the five rates and the next dt from the per-CTA partials, summed in
// the finalise's fixed order (thread-strided, then its tree); a field's square
// root or division in a thread of its own.
__global__ void __launch_bounds__(kFinThreads) k_noalloc_reduce(const double *partials, int ntiles, const CavConst *cc,
                                                                double *out6) {
  __shared__ double sv[8 * kFinThreads];
  chain_wait();
  const int tid = threadIdx.x, f = tid >> 4;
  double acc[8];
  load_slice<kFinThreads>(BcArgs{}, partials, 0, ntiles, 0, 0, 0, 0, tid, acc);
  const double t = tree_slice<kFinThreads>(acc, sv, tid);
  if ((tid & 15) != 0 || f > 5) return;
  out6[f] = f < 5 ? sqrt(t * cc->inv_nint) : cc->cfl / t;
}

// A launch that may start before the one ahead of it in the stream has ended
// (each waits for that before it reads what it wrote).
template <class K, class... A>
cudaError_t launch_after(K kernel, int grid, int block, cudaStream_t st, A... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }

}  // namespace

extern "C" CAVITY_API int cavity_step_block_noalloc(const double *q_in, double *q_out, int nx, int ny, int nz,
                                                    const cavity_params *p, double dt, double pshift,
                                                    double *out6, void *stream) {
  if (!q_in || !q_out || !out6 || !p || q_in == q_out) return CAVITY_ERR_INVALID_ARG;
  if (nx < 2 || ny < 2 || nz < 2 || !(dt >= 0.0) || !std::isfinite(pshift)) return CAVITY_ERR_INVALID_ARG;
  const long long limit_tiles = (long long)ceil_div(nx, kTX) * ceil_div(ny, kTY) * ceil_div(nz, kKC);
  if (limit_tiles > CAVITY_NOALLOC_MAX_TILES) return CAVITY_ERR_INVALID_ARG;  // beyond the fixed scratch
  cavity_params q = *p;
  if (!(q.u_ref >= 0.0)) q.u_ref = std::max(1.0, std::sqrt(q.Ra * q.Pr));
  if (std::isnan(q.t_inf)) q.t_inf = 0.5 * (q.t_hot + q.t_cold);
  if (!(q.Ra >= 0.0) || !(q.Pr > 0.0) || !(q.cfl > 0.0) || !(q.kappa > 0.0) || !(q.c4 >= 0.0) ||
      !(q.u_ref > 0.0) || !std::isfinite(q.t_inf) || (q.gravity_axis != 1 && q.gravity_axis != 2))
    return CAVITY_ERR_INVALID_ARG;

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return CAVITY_ERR_CUDA;
  void *scratch = nullptr;
  if (scratch_address(dev, &scratch) != cudaSuccess) return CAVITY_ERR_CUDA;
  unsigned char *s = (unsigned char *)scratch;
  BlockDev *d_block = (BlockDev *)s;
  CavConst *d_cc = (CavConst *)(s + 256);
  CavState *d_cs = (CavState *)(s + 1024);
  double *d_part = (double *)(s + kDescBytes);

  // dense caller layout: node (i, j, k), i in [-1, n+2], at (i+1) + (nx+4)((j+1) + (ny+4)(k+1));
  // the kernel addresses node i at XO - 1 + i, so the base is moved back by XO - 2 elements
  BlockDev B{};
  B.nx = nx; B.ny = ny; B.nz = nz;
  B.pitch = nx + 4;
  B.rows = ny + 4;
  B.plane = (long long)B.pitch * B.rows;
  B.fstride = B.plane * (nz + 4);
  for (int f = 0; f < 6; ++f) { B.wall[f] = 1; B.nbr[f] = -1; }
  // Tiles of consecutive nodes, one CTA each, of a depth that leaves the SMs
  // equal shares of the tile planes (as the handle's, assign_tiles): with
  // 16-plane tiles of 256 nodes at all sizes a 40x36x34 block was 18 CTAs and
  // 137 us a call.  Where tiles of 128 nodes would not fit the scratch, the
  // 256-node ones do (256 consecutive nodes fill no more tiles than the limit's).
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return CAVITY_ERR_CUDA;
  int nt = 128;
  const long long planes = (long long)ceil_div((long long)nx * ny, nt) * nz;
  int kc = planes <= 8LL * sms ? 1 : planes <= 16LL * sms ? 2 : planes <= 64LL * sms ? 4 : 8;
  while (kc < kKC && (long long)ceil_div((long long)nx * ny, nt) * ceil_div(nz, kc) > CAVITY_NOALLOC_MAX_TILES) kc *= 2;
  if ((long long)ceil_div((long long)nx * ny, nt) * ceil_div(nz, kc) > CAVITY_NOALLOC_MAX_TILES) {
    nt = kTX * kTY;
    kc = kKC;
  }
  B.tiles_x = ceil_div((long long)nx * ny, nt);
  B.tiles_y = 1;
  B.tiles_z = ceil_div(nz, kc);
  B.tiles_zc = B.tiles_z;  // kc-plane chunks only
  B.zsplit = nz;
  B.kc = B.kf = kc;
  B.coarse_begin = 0;
  B.fine_begin = 0;
  B.base[0] = (void *)(q_in - (XO<double>::v - 2));
  B.base[1] = (void *)(q_out - (XO<double>::v - 2));

  CavConst C{};
  const int gn[3] = {nx, ny, nz};
  set_cav_physics(C, gn, q);

  CavState S{};
  S.dt = dt;
  S.c = pshift;

  cudaStream_t st = (cudaStream_t)stream;
  k_noalloc_setup<<<1, 128, 0, st>>>(Descriptors{B, C, S}, d_block, d_cc, d_cs);
  if (cudaGetLastError() != cudaSuccess) return CAVITY_ERR_CUDA;
  StepArgs a{};  // tile_counter null: one CTA per tile
  a.blocks = d_block; a.nblocks = 1; a.cc = d_cc; a.cs = d_cs;
  const int ntiles = B.tiles_x * B.tiles_z;
  a.partials = d_part; a.parity = 0; a.mode = 0; a.ntiles = ntiles;
  a.ncoarse = ntiles;
  // walls and ghosts read as the caller filled them
  const cudaError_t e = nt == 128 ? launch_after(k_step_f64<128, false>, ntiles, nt, st, a, BcArgs{})
                                  : launch_after(k_step_f64<kTX * kTY, false>, ntiles, nt, st, a, BcArgs{});
  if (e != cudaSuccess) return CAVITY_ERR_CUDA;
  if (launch_after(k_noalloc_reduce, 1, kFinThreads, st, (const double *)d_part, ntiles, (const CavConst *)d_cc, out6) !=
      cudaSuccess)
    return CAVITY_ERR_CUDA;
  return CAVITY_OK;
}
