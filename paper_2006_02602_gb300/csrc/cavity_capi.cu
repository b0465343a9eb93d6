// C ABI of the buoyancy-driven-cavity step (include/cavity.h): host runtime
// that lays out the blocks of one or many cavities in HBM, builds the work
// lists of the kernels in bdc_device.cuh / bdc_step_f32.cuh, launches them and
// captures CUDA graphs of them to replay.  Two arithmetic forms share the
// runtime: FP64 (five FP64 arrays per buffer set) and FP32-mixed (p_hi, p_lo,
// u, v, w, T in FP32, read by the step kernel through TMA tensor maps).  A
// handle holds either one cavity split into blocks (Section 3.2
// decomposition) or a batch of single-block cavities.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cfloat>
#include <cstdlib>
#include <cstddef>
#include <climits>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/cavity.h"
#include "bdc_adjoint.cuh"
#include "bdc_device.cuh"
#include "bdc_step_f32.cuh"

using namespace bdc;

namespace {

// k_step tile of the FP64 form: 32 * ty consecutive nodes of a plane (ty = 4:
// 128 threads; three CTAs, 12 warps, per SM hide the FP64 pipe's latency
// better than one of 256); the chunk depths: assign_tiles
constexpr int kTX = 32, kTY = 4;

int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }

std::vector<int> split_sizes(int n, int parts) {  // Section 3.2: as even as possible
  std::vector<int> s(parts, n / parts);
  for (int r = 0; r < n % parts; ++r) s[r] += 1;
  return s;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// FP32 step-kernel variants compiled in: (kernel form P, tile height TY, ring
// depth R); P = 3 is k_step_f32q (two nodes per thread, the nodes behind the
// plane in registers), the one form.  The z-chunk depth is a run-time
// parameter of the tiling (the autotuner tries kF32Chunks).
#define BDC_F32_VARIANTS(X) X(3, 8, 4) X(3, 8, 5) X(3, 16, 4) X(3, 16, 5)
struct F32Shape {
  int p, ty, kc, r;
};
const int kF32Chunks[] = {16, 24, 32, 40, 48, 64, 96};
constexpr int kF32MaxChunk = 4096;

bool f32_variant_ok(int p, int ty, int kc, int r) {
  if (kc < 1 || kc > kF32MaxChunk) return false;
#define BDC_OK(P, TY, R) \
  if (p == P && ty == TY && r == R) return true;
  BDC_F32_VARIANTS(BDC_OK)
#undef BDC_OK
  return false;
}

// every (variant, chunk depth) pair the autotuner times
std::vector<F32Shape> f32_shapes() {
  std::vector<F32Shape> out;
#define BDC_SHAPE(P, TY, R) \
  for (int kc : kF32Chunks) out.push_back({P, TY, kc, R});
  BDC_F32_VARIANTS(BDC_SHAPE)
#undef BDC_SHAPE
  return out;
}

}  // namespace

// checkpoints and work arrays of the discrete adjoint (single-block cavity)
struct AdjointStore {
  int nsteps = 0, run_ckpt = 0;  // of the last forward run
  int ckpt = 0, ncp = 0;         // as allocated
  int layout = -1;             // the tiling the segment's tables were made for
  int setup = 0;               // the parameters and wall temperatures of the last forward run
  size_t set_bytes = 0;        // one buffer set of the block
  void *mem = nullptr;         // the one allocation behind the pointers below
  char *ckpt_mem = nullptr;    // ncp buffer sets: the state at steps 0, ckpt, 2 ckpt, ...
  CavState *ckpt_cs = nullptr;  // their scalars (device)
  char *seg_mem = nullptr;     // ckpt buffer sets: one recomputed segment
  BlockDev *seg_blocks = nullptr;   // ckpt block descriptors: slot s as buffer set 0, slot s + 1 as buffer set 1
  WallFace *seg_faces = nullptr;    // the block's wall faces once per slot (one walls launch per segment)
  CUtensorMap *seg_maps = nullptr;  // FP32 form: the step kernel's two maps of every slot
  char *final_mem = nullptr;   // the state after the forward run
  CavState final_cs{};
  int final_parity = 0;
  long long final_steps = 0;
  void *X = nullptr, *Q = nullptr;  // adjoint arrays: FP64 (FP64 forward) or FP32 (FP32-mixed)
  double *thetabar = nullptr, *scal = nullptr, *argpart = nullptr;
  double *gpart = nullptr;     // per-CTA node sums of the sweep (4 per CTA)
  double *dts = nullptr;       // dt of every step of a segment (device)
  unsigned int *cnt = nullptr; // finished CTAs of k_adj_sweep (zero between launches)
  int kc = 0, ctas = 0;        // the sweep's chunk depth and CTAs
  bool have_forward = false;
  double J = 0.0;
};
constexpr int kAdjParts = 2 * 152;  // argmax partials of a state

// Steps of one graph (or sequence of launches): it ends with one finalise launch for
// all of its steps, so a long run is mostly 16-step graphs (2 for calls of two or three
// steps: FP64 32^3 in calls of two 17.4 us a step, 24.6 as two graphs of one).
constexpr int kGraphs = 4;
constexpr int kGraphSteps[kGraphs] = {1, 2, 4, kGraphMax};

struct cavity {
  int dev = 0;
  bool u_ref_auto = true;  // u_ref follows Ra (default)
  AdjointStore adj;
  std::vector<cudaEvent_t> adj_ev;  // two per segment: around its reverse steps' launches
  double adj_rates_ms = 0.0;        // mean duration of one in the last reverse sweep
  int layout = 0;                   // counts assign_tiles calls
  int setup = 0;                    // counts the parameters and wall temperatures set
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int ncav = 1;
  std::vector<cavity_desc> descs;
  std::vector<cavity_params> prms;
  std::vector<CavConst> hcc;
  std::vector<char> wall_custom;  // 2 per cavity
  std::vector<double> twall;      // per cavity: hot wall then cold wall (ny*nz each) at wall_off
  bool f32 = false;               // FP32-mixed form
  size_t esize = 8;               // bytes per stored element
  int na = 5;                     // stored arrays per buffer set
  int np = 1;                     // pressure arrays
  int tx = kTX, ty = kTY, kc = 8;
  bool f32_auto = true;           // the FP32 step kernel's chunk depth by size (f32_chunk)
  int f32_r = 0;                  // ring depth of the FP32 step kernel
  int f32_p = 1;                  // nodes per thread along x of the FP32 step kernel
  int local_dt = 0;               // CAVITY_DT_LOCAL: each node at its own stable step
  long long wait_cycles = kWaitCycles;  // limit of the FP32 step kernel's bounded waits
  int withhold_plane = -1;              // timeout test: tile plane whose load is not issued
  // interior/shell split with overlapped exchange (FP64, single cavity, cut faces)
  bool overlap = false;
  std::vector<ShellFace> hshell;
  ShellFace *d_shell = nullptr;
  int n_shell = 0;                // k_shell_f64 CTAs
  cudaStream_t side = nullptr;    // the exchange's stream while the interior is stepped
  cudaEvent_t ev_shell = nullptr, ev_exch = nullptr;
  int nblocks = 0;
  std::vector<BlockDev> hb;
  std::vector<WallFace> hwall;
  std::vector<WallFace> hxwall;   // the x walls alone, with their own CTA numbers (Nusselt sums after an FP64 step)
  int n_nu = 0;                   // their CTAs
  std::vector<CutFace> hcut;
  long long xbuf_elems = 0;
  int n_step = 0, n_bc = 0, n_cut = 0;
  int nslices = kFinSlices;  // k_finalize CTAs per cavity: about 128 step partials a slice
  int form_walls = 1;  // FP64: walls formed where the step reads them (0: stored between the steps)
  int n_coarse = 0;  // FP64 step tiles of KC planes (scheduled before the fine ones)
  int part_cap = 0;  // step partials allocated (CTAs) a set
  int part_sets = kGraphMax;  // sets: steps of the longest graph (16, 4 or 1)

  BlockDev *d_blocks = nullptr;
  CavConst *d_cc = nullptr;
  CavState *d_cs = nullptr;
  WallFace *d_wall = nullptr, *d_xwall = nullptr;
  CutFace *d_cut = nullptr;
  CUtensorMap *d_maps = nullptr;
  double *d_step_part = nullptr, *d_bc_part = nullptr, *d_twall = nullptr, *d_stage = nullptr;
  double *d_fin = nullptr;  // k_finalize slice totals [kGraphMax][ncav][kFinSlices][8]
  StepResult *d_rec = nullptr;  // [kGraphMax][ncav]
  StepRecord *d_log = nullptr;  // the step log (device address of caller-owned host memory), or null
  long long log_cap = 0;
  unsigned int *d_counter = nullptr;  // the FP64 step's tile counters (kStepSlots), then BcArgs::counter
  int nsm = 0;                        // SMs of the device
  int persist_ctas = 0;               // CTAs of the persistent FP64 step kernel that fit on the GPU
  void *d_fields = nullptr, *d_xbuf = nullptr;
  size_t field_bytes = 0;
  size_t stage_elems = 0;

  int parity = 0;
  long long steps_taken = 0;
  cudaGraphExec_t graph[kGraphs][2] = {};  // kGraphSteps[q] steps from parity 0 / 1
  bool launched[kGraphs][2] = {};          // such steps have run as plain launches
  cudaStream_t capture = nullptr;          // the graphs are captured on it
  std::string err;
};

namespace {

int fail(cavity *h, int code, const std::string &msg) {
  if (h) h->err = msg;
  return code;
}

// (the error goes to the caller, not to the next call that asks for the last one)
#define CK(call)                                                                   \
  do {                                                                             \
    cudaError_t e_ = (call);                                                       \
    if (e_ != cudaSuccess) {                                                       \
      cudaGetLastError();                                                          \
      return fail(h, e_ == cudaErrorMemoryAllocation ? CAVITY_ERR_OOM : CAVITY_ERR_CUDA, \
                  std::string(#call) + ": " + cudaGetErrorString(e_));             \
    }                                                                              \
  } while (0)

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

int xo1(size_t esize) { return esize == 8 ? XO<double>::v : XO<float>::v; }

long long host_node_index(const BlockDev &B, size_t esize, int i, int j, int k) {
  return (long long)(xo1(esize) - 1 + i) + (long long)B.pitch * (j + 1) + B.plane * (k + 1);
}

void fill_consts(cavity *h, int c) {
  const int gn[3] = {h->descs[c].nx, h->descs[c].ny, h->descs[c].nz};
  set_cav_physics(h->hcc[c], gn, h->prms[c]);
}

void resolve_defaults(cavity_params *p) {
  if (!(p->u_ref >= 0.0)) p->u_ref = std::max(1.0, std::sqrt(p->Ra * p->Pr));
  if (std::isnan(p->t_inf)) p->t_inf = 0.5 * (p->t_hot + p->t_cold);
}

int check_params(const cavity_params &p) {
  if (!(p.Ra >= 0.0) || !(p.Pr > 0.0) || !(p.cfl > 0.0) || !(p.kappa > 0.0) || !(p.c4 >= 0.0) ||
      !(p.u_ref > 0.0) || !(p.kappa * p.u_ref * p.u_ref >= FLT_MIN) ||
      !(p.kappa * p.u_ref * p.u_ref < 1e300) || !std::isfinite(p.t_inf) || !std::isfinite(p.t_hot) || !std::isfinite(p.t_cold) ||
      p.t_hot == p.t_cold || (p.gravity_axis != 1 && p.gravity_axis != 2))
    return CAVITY_ERR_INVALID_ARG;
  return CAVITY_OK;
}

int check_desc(const cavity_desc &d) {
  if (d.nx < 2 || d.ny < 2 || d.nz < 2 || d.px < 1 || d.py < 1 || d.pz < 1) return CAVITY_ERR_INVALID_ARG;
  if (d.nx / d.px < 2 || d.ny / d.py < 2 || d.nz / d.pz < 2) return CAVITY_ERR_INVALID_ARG;
  if ((long long)d.nx * d.ny * d.nz > (1LL << 34)) return CAVITY_ERR_INVALID_ARG;
  if (!(d.noise_amp >= 0.0) || !std::isfinite(d.noise_amp)) return CAVITY_ERR_INVALID_ARG;
  if (d.precision != CAVITY_FP64 && d.precision != CAVITY_FP32_MIXED) return CAVITY_ERR_INVALID_ARG;
  return CAVITY_OK;
}

// ---------------------------------------------------------------------------
// layout: blocks of every cavity, wall / cut face lists, centre nodes

// Step-kernel tiles and their partial slots, block by block (a cavity's
// slots are contiguous): kc-plane chunks below the last chunk boundary, the
// planes above it in fine chunks scheduled after every block's coarse tiles.
//
// FP64: what counts is the number of tile planes (128 nodes x 1 plane) an SM
// gets.  A tile plane takes an SM about 2.1 us whatever else it runs (256^3); a
// tile's own cost (queue loads, tile look-up, reduction) is about a third of one.  So large cavities take 8-plane tiles with 2-plane ones in the
// end, small ones 4-plane and 1-plane tiles, and the fine tiles hold 8 planes
// an SM (all of a cavity of up to 38^3), enough to level what the coarse ones
// leave.  Measured per step with either, 4-plane tiles first: 32^3 11.6 and
// 14.9 us, 64^3 45 and 65, 97x65x50 51 and 64, 128^3 265 and 257, 256^3 1951 and
// 1843.
//
// FP32: tail chunks of at most kFineKC32 planes, only in blocks deeper than one
// chunk (a shallower block is one chunk: the ring's fill is paid per tile).
int f32_zsplit(int nz, int kc) { return nz <= kc ? nz : (nz - 1) / kc * kc; }
int f32_tiles_z(int nz, int kc) {
  if (nz <= kc) return 1;
  return (nz - 1) / kc + ceil_div(nz - f32_zsplit(nz, kc), std::min(kFineKC32, kc));
}

// Chunk depth of the FP32 form where neither the caller's autotuner nor the
// environment has set one.  A tile sweeps its planes one after another (1 us a
// plane alone on an SM), so a cavity whose tiles all run at once takes as long
// as its deepest tile and the tiles beside it: measured on 32^3 .. 128^3 within
// 1-2 us, a step is 7.4 + kc + (n - 1) (2.2 + 0.24 kc) us with n tiles on the
// fullest SM, and the depth is the one that makes this least.  Four tiles run at
// once on an SM; a fifth costs 8 us more (128^3: 41 us at 16 planes and four
// tiles, 49 at 12 and five) but still beats deeper ones (128^3 in 2x2x2 blocks:
// 58 us at 16 planes, 60 at 24).  Larger cavities: 24 planes up to 150 tile planes an
// SM (160^3: 66 us, 69 at 32, 71 at 16), 64 beyond (batch of 64: 230 us, 235 at
// 32; 256^3: 211 at either).  With 32 planes at all sizes: 32^3 40 us (8.4 now),
// 64^3 39 (14.5), 96x80x72 38 (19.5), 128^3 52 (41).
int f32_chunk(const cavity *h) {
  double best = 1e300;
  int kc = 0;
  long long planes = 0;
  for (const BlockDev &B : h->hb) planes += (long long)ceil_div(B.nx, h->tx) * ceil_div(B.ny, h->ty) * B.nz;
  for (int k : {1, 2, 4, 6, 8, 12, 16}) {
    long long tiles = 0;
    for (const BlockDev &B : h->hb) tiles += (long long)ceil_div(B.nx, h->tx) * ceil_div(B.ny, h->ty) * f32_tiles_z(B.nz, k);
    const int n = ceil_div(tiles, h->nsm);
    if (n > 5) continue;
    const double us = 7.4 + k + (n - 1) * (2.2 + 0.24 * k) + (n > 4 ? 8.0 : 0.0);
    if (us < best) {
      best = us;
      kc = k;
    }
  }
  return kc ? kc : planes <= 150LL * h->nsm ? 24 : 64;
}

void assign_tiles(cavity *h) {
  h->layout += 1;
  long long planes = 0;
  if (h->f32 && h->f32_auto) h->kc = f32_chunk(h);
  if (!h->f32) {
    for (const BlockDev &B : h->hb) planes += (long long)ceil_div((long long)B.nx * B.ny, h->tx * h->ty) * B.nz;
    h->kc = planes >= 64LL * h->nsm ? 8 : 4;
    h->form_walls = h->kc == 4;  // (why the line lies there: step_tile_f64)
  }
  int tile = 0, coarse = 0, fine = 0;
  for (int c = 0; c < h->ncav; ++c) h->hcc[c].tile_begin = -1;
  for (BlockDev &B : h->hb) {
    B.kc = h->kc;
    if (h->f32) {
      B.tiles_x = ceil_div(B.nx, h->tx);
      B.tiles_y = ceil_div(B.ny, h->ty);
      B.kf = std::min(kFineKC32, h->kc);
      B.zsplit = f32_zsplit(B.nz, h->kc);
      B.tiles_zc = B.nz <= h->kc ? 1 : B.zsplit / h->kc;
    } else {
      B.tiles_x = ceil_div((long long)B.nx * B.ny, h->tx * h->ty);
      B.tiles_y = 1;
      B.kf = h->kc == 8 ? 2 : 1;
      const int nfine = ceil_div(8LL * h->nsm * B.nz, planes);
      B.tiles_zc = std::max(0, B.nz - nfine) / h->kc;
      B.zsplit = B.tiles_zc * h->kc;
    }
    B.tiles_z = B.tiles_zc + ceil_div(B.nz - B.zsplit, B.kf);
    B.tile_begin = tile;
    B.coarse_begin = coarse;
    B.fine_begin = fine;
    CavConst &C = h->hcc[B.cav];
    if (C.tile_begin < 0) C.tile_begin = tile;
    tile += B.tiles_x * B.tiles_y * B.tiles_z;
    coarse += B.tiles_x * B.tiles_y * B.tiles_zc;
    fine += B.tiles_x * B.tiles_y * (B.tiles_z - B.tiles_zc);
    C.tile_end = tile;
  }
  h->n_step = tile;
  h->n_coarse = coarse;
  int most = 0;  // the most tiles of one cavity
  for (int c = 0; c < h->ncav; ++c) most = std::max(most, h->hcc[c].tile_end - h->hcc[c].tile_begin);
  h->nslices = std::max(1, std::min(kFinSlices, ceil_div(most, 128)));
  for (int c = 0; c < h->ncav; ++c) {  // contiguous slices of each cavity's step partials
    CavConst &C = h->hcc[c];
    const long long nt = C.tile_end - C.tile_begin;
    for (int g = 0; g <= kFinSlices; ++g)
      C.slice_q[g] = C.tile_begin + (int)(nt * std::min(g, h->nslices) / h->nslices);
  }
}

int build_layout(cavity *h) {
  const size_t es = h->esize;
  const int row_align = (int)(128 / es);
  h->hb.clear();
  size_t total_elems = 0;
  long long wall_off = 0;
  for (int cv = 0; cv < h->ncav; ++cv) {
    const cavity_desc &d = h->descs[cv];
    const int pg[3] = {d.px, d.py, d.pz};
    const int gn[3] = {d.nx, d.ny, d.nz};
    std::vector<int> sz[3], org[3];
    for (int a = 0; a < 3; ++a) {
      sz[a] = split_sizes(gn[a], pg[a]);
      int o = 0;
      for (int s : sz[a]) { org[a].push_back(o); o += s; }
    }
    const int first = (int)h->hb.size();
    for (int bz = 0; bz < pg[2]; ++bz)
      for (int by = 0; by < pg[1]; ++by)
        for (int bx = 0; bx < pg[0]; ++bx) {
          BlockDev B{};
          B.nx = sz[0][bx]; B.ny = sz[1][by]; B.nz = sz[2][bz];
          B.ox = org[0][bx]; B.oy = org[1][by]; B.oz = org[2][bz];
          B.pitch = ((xo1(es) + B.nx + 2 + row_align - 1) / row_align) * row_align;
          B.rows = B.ny + 4;
          B.plane = (long long)B.pitch * B.rows;
          B.fstride = ((B.plane * (B.nz + 4) + 63) / 64) * 64;
          const int c3[3] = {bx, by, bz};
          for (int f = 0; f < 6; ++f) {
            const int a = f / 2, hi = f % 2;
            int cc[3] = {c3[0], c3[1], c3[2]};
            cc[a] += hi ? 1 : -1;
            const bool inside = cc[a] >= 0 && cc[a] < pg[a];
            B.wall[f] = inside ? 0 : 1;
            B.nbr[f] = inside ? first + cc[0] + pg[0] * (cc[1] + pg[1] * cc[2]) : -1;
          }
          B.cav = cv;
          h->hb.push_back(B);
          total_elems += 2 * (size_t)h->na * (size_t)B.fstride;
        }
    CavConst &C = h->hcc[cv];
    C.wall_off = wall_off;
    wall_off += 2LL * d.ny * d.nz;
    // centre nodes in (k, j, i) lexicographic order
    std::vector<int> ax[3];
    for (int a = 0; a < 3; ++a) {
      if (gn[a] % 2 == 1) ax[a] = {(gn[a] + 1) / 2};
      else ax[a] = {gn[a] / 2, gn[a] / 2 + 1};
    }
    int m = 0;
    for (int K : ax[2])
      for (int J : ax[1])
        for (int I : ax[0]) {
          for (int id = first; id < (int)h->hb.size(); ++id) {
            const BlockDev &B = h->hb[id];
            if (I > B.ox && I <= B.ox + B.nx && J > B.oy && J <= B.oy + B.ny && K > B.oz && K <= B.oz + B.nz) {
              C.centre_blk[m] = id;
              C.centre_off[m] = host_node_index(B, es, I - B.ox, J - B.oy, K - B.oz);
            }
          }
          ++m;
        }
    C.ncentre = m;
  }
  h->nblocks = (int)h->hb.size();
  h->field_bytes = total_elems * es;
  h->twall.assign((size_t)wall_off, 0.0);
  assign_tiles(h);
  // wall faces, contiguous per cavity, and cut faces, each list with its x
  // faces first: a CTA of an x face touches one 32-byte sector per node and
  // array (its positions run along y) where the others' rows are contiguous,
  // and launched first the x faces' CTAs spread over the SMs (after a 128^3
  // FP32 step in 2 x 2 x 2 blocks the last exchange CTA ended 14-15 us after
  // the step kernel with the faces in block order, 10-12 us in this order
  // together with the finalise's reduction trees)
  h->hwall.clear();
  h->hcut.clear();
  for (int id = 0; id < h->nblocks; ++id) {
    const BlockDev &B = h->hb[id];
    const int n[3] = {B.nx, B.ny, B.nz};
    for (int f = 0; f < 6; ++f) {
      const int a = f / 2;
      const int n1 = n[a == 0 ? 1 : 0], n2 = n[a == 2 ? 1 : 2];
      if (B.wall[f]) h->hwall.push_back(WallFace{id, f, n1, n2, 0, B.cav});
      else h->hcut.push_back(CutFace{id, f, B.nbr[f], n1, n2, 0, 0});
    }
  }
  std::stable_sort(h->hwall.begin(), h->hwall.end(), [](const WallFace &x, const WallFace &y) {
    return x.cav != y.cav ? x.cav < y.cav : x.face / 2 < y.face / 2;
  });
  std::stable_sort(h->hcut.begin(), h->hcut.end(),
                   [](const CutFace &x, const CutFace &y) { return x.face / 2 < y.face / 2; });
  int bc = 0, cut = 0;
  long long xoff = 0;
  for (int c = 0; c < h->ncav; ++c) h->hcc[c].bc_begin = -1;
  for (WallFace &w : h->hwall) {
    CavConst &C = h->hcc[w.cav];
    w.cta_begin = bc;
    if (C.bc_begin < 0) C.bc_begin = C.bc_xend = bc;
    bc += ceil_div((long long)w.n1 * w.n2, kBcThreads);
    C.bc_end = bc;
    if (w.face / 2 == 0) C.bc_xend = bc;
  }
  h->hxwall.clear();
  h->n_nu = 0;
  for (int c = 0; c < h->ncav; ++c) h->hcc[c].nu_begin = -1;
  for (WallFace w : h->hwall) {
    if (w.face / 2 != 0) continue;
    CavConst &C = h->hcc[w.cav];
    w.cta_begin = h->n_nu;
    if (C.nu_begin < 0) C.nu_begin = h->n_nu;
    h->n_nu += ceil_div((long long)w.n1 * w.n2, kBcThreads);
    C.nu_end = h->n_nu;
    h->hxwall.push_back(w);
  }
  for (CutFace &c : h->hcut) {
    c.cta_begin = cut;
    c.buf_off = xoff;
    cut += ceil_div((long long)c.nb * c.nc, 256);
    xoff += (long long)(h->na + h->np) * c.nb * c.nc;
  }
  h->n_bc = bc;
  h->n_cut = cut;
  h->xbuf_elems = xoff;
  return CAVITY_OK;
}

// TMA descriptors of the FP32-mixed step kernel: two 4-D maps per block and
// buffer set over (x, y, z, array): the pressure box (40 x (TY+4) nodes of
// p_hi and p_lo) and the box of the other five arrays (40 x (TY+2) nodes)
// The pressure-box and other-box maps (out[0], out[1]) of a buffer set of
// block B's layout at `base`.
int encode_block_maps(cavity *h, const BlockDev &B, void *base, CUtensorMap out[2]) {
  void *fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  CK(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q));
  if (q != cudaDriverEntryPointSuccess || !fn) return fail(h, CAVITY_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
  EncodeTiledFn encode = (EncodeTiledFn)fn;
  for (int kind = 0; kind < 2; ++kind) {
    // columns up to node nx + 2: the row's padding lies outside the map, so a
    // box reaching past it is zero-filled, not read from HBM
    const cuuint64_t dims[4] = {(cuuint64_t)(XO<float>::v + B.nx + 2), (cuuint64_t)B.rows, (cuuint64_t)(B.nz + 4),
                                (cuuint64_t)kF32NA};
    const cuuint64_t strides[3] = {(cuuint64_t)B.pitch * 4, (cuuint64_t)B.plane * 4, (cuuint64_t)B.fstride * 4};
    const cuuint32_t box[4] = {(cuuint32_t)kF32BX, (cuuint32_t)(kind == 0 ? f32_box_yp(h->ty) : f32_box_yo(h->ty)), 1,
                               (cuuint32_t)(kind == 0 ? kF32NP : kF32NO)};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = encode(&out[kind], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(h, CAVITY_ERR_CUDA, "cuTensorMapEncodeTiled failed");
  }
  return CAVITY_OK;
}

int encode_maps(cavity *h) {
  std::vector<CUtensorMap> maps(4 * h->nblocks);
  for (int id = 0; id < h->nblocks; ++id)
    for (int s = 0; s < 2; ++s) {
      const int rc = encode_block_maps(h, h->hb[id], h->hb[id].base[s], &maps[2 * (2 * id + s)]);
      if (rc != CAVITY_OK) return rc;
    }
  if (!h->d_maps) CK(cudaMalloc(&h->d_maps, sizeof(CUtensorMap) * maps.size()));
  CK(cudaMemcpy(h->d_maps, maps.data(), sizeof(CUtensorMap) * maps.size(), cudaMemcpyHostToDevice));
  return CAVITY_OK;
}

template <int P, int TY, int R>
auto f32_kernel() {
  static_assert(P == 3, "the FP32 step kernel has one form");
  return k_step_f32q<TY, R>;
}

// dynamic shared memory of the FP32 step kernel's shape, and the largest
// shared-memory carveout (four 47 KB CTAs per SM)
cudaError_t f32_set_smem(int p, int ty, int r) {
#define BDC_ATTR(P, TY, R)                                                                                       \
  if (p == P && ty == TY && r == R) {                                                                            \
    const cudaError_t e = cudaFuncSetAttribute(f32_kernel<P, TY, R>(),                                           \
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, f32_smem_bytes(TY, R)); \
    if (e != cudaSuccess) return e;                                                                              \
    return cudaFuncSetAttribute(f32_kernel<P, TY, R>(), cudaFuncAttributePreferredSharedMemoryCarveout,         \
                                (int)cudaSharedmemCarveoutMaxShared);                                            \
  }
  BDC_F32_VARIANTS(BDC_ATTR)
#undef BDC_ATTR
  return cudaErrorInvalidValue;
}

// the FP64 step kernel of a tile of 32 * ty nodes
auto f64_kernel(int ty, bool form_walls) {
  if (ty == 4) return form_walls ? k_step_f64<kTX * 4, true> : k_step_f64<kTX * 4, false>;
  return form_walls ? k_step_f64<kTX * 8, true> : k_step_f64<kTX * 8, false>;
}

int upload_tables(cavity *h) {
  CK(cudaMemcpyAsync(h->d_blocks, h->hb.data(), sizeof(BlockDev) * h->nblocks, cudaMemcpyHostToDevice, h->stream));
  CK(cudaMemcpyAsync(h->d_cc, h->hcc.data(), sizeof(CavConst) * h->ncav, cudaMemcpyHostToDevice, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return CAVITY_OK;
}

int ensure_partials(cavity *h) {
  const int need = h->n_step + (h->overlap ? h->n_shell : 0);
  if (h->part_cap >= need) return CAVITY_OK;
  CK(cudaStreamSynchronize(h->stream));
  if (h->d_step_part) cudaFree(h->d_step_part);
  h->d_step_part = nullptr;
  h->part_cap = 0;
  // one set per step of a graph: all are reduced at its end.  Sixteen are 1.2% of a large
  // FP64 state; where they are what no longer fits, graphs are shorter.
  for (h->part_sets = kGraphMax;; h->part_sets /= 4) {
    const cudaError_t e = cudaMalloc(&h->d_step_part, h->part_sets * sizeof(double) * kPartStride * std::max(1, need));
    if (e == cudaSuccess) break;
    if (e != cudaErrorMemoryAllocation || h->part_sets == 1) CK(e);
    cudaGetLastError();
  }
  h->part_cap = std::max(1, need);
  return CAVITY_OK;
}

int alloc_device(cavity *h) {
  CK(cudaMalloc(&h->d_fields, h->field_bytes));
  CK(cudaMemsetAsync(h->d_fields, 0, h->field_bytes, h->stream));
  char *base = (char *)h->d_fields;
  for (auto &B : h->hb) {
    for (int s = 0; s < 2; ++s) {
      B.base[s] = base;
      base += (size_t)h->na * (size_t)B.fstride * h->esize;
    }
  }
  CK(cudaMalloc(&h->d_blocks, sizeof(BlockDev) * h->nblocks));
  CK(cudaMalloc(&h->d_cc, sizeof(CavConst) * h->ncav));
  CK(cudaMalloc(&h->d_cs, sizeof(CavState) * h->ncav));
  CK(cudaMemsetAsync(h->d_cs, 0, sizeof(CavState) * h->ncav, h->stream));
  CK(cudaMalloc(&h->d_wall, sizeof(WallFace) * std::max<size_t>(1, h->hwall.size())));
  CK(cudaMalloc(&h->d_xwall, sizeof(WallFace) * std::max<size_t>(1, h->hxwall.size())));
  CK(cudaMalloc(&h->d_cut, sizeof(CutFace) * std::max<size_t>(1, h->hcut.size())));
  int rc = ensure_partials(h);
  if (rc != CAVITY_OK) return rc;
  // the wall kernel's Nusselt partials, or (FP64) the x walls' of every step of a graph
  CK(cudaMalloc(&h->d_bc_part, sizeof(double) * 2 * std::max(std::max(1, h->n_bc), h->f32 ? 0 : kGraphMax * h->n_nu)));
  CK(cudaMalloc(&h->d_fin, sizeof(double) * kGraphMax * 8 * kFinSlices * h->ncav));
  CK(cudaMalloc(&h->d_rec, sizeof(StepResult) * kGraphMax * h->ncav));
  const size_t counter_bytes = sizeof(unsigned int) * (kStepSlots + (size_t)(kGraphMax + 1) * h->ncav);
  CK(cudaMalloc(&h->d_counter, counter_bytes));
  CK(cudaMemsetAsync(h->d_counter, 0, counter_bytes, h->stream));
  {
    int per_sm = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f64_kernel(h->ty, h->form_walls), kTX * h->ty, 0));
    h->persist_ctas = std::max(1, h->nsm * per_sm);
  }
  CK(cudaMalloc(&h->d_twall, sizeof(double) * std::max<size_t>(1, h->twall.size())));
  if (h->xbuf_elems > 0) CK(cudaMalloc(&h->d_xbuf, h->esize * (size_t)h->xbuf_elems));
  if (!h->hwall.empty())
    CK(cudaMemcpyAsync(h->d_wall, h->hwall.data(), sizeof(WallFace) * h->hwall.size(), cudaMemcpyHostToDevice, h->stream));
  if (!h->hxwall.empty())
    CK(cudaMemcpyAsync(h->d_xwall, h->hxwall.data(), sizeof(WallFace) * h->hxwall.size(), cudaMemcpyHostToDevice, h->stream));
  if (!h->hcut.empty())
    CK(cudaMemcpyAsync(h->d_cut, h->hcut.data(), sizeof(CutFace) * h->hcut.size(), cudaMemcpyHostToDevice, h->stream));
  if (h->f32) {
    rc = encode_maps(h);
    if (rc != CAVITY_OK) return rc;
    CK(f32_set_smem(h->f32_p, h->ty, h->f32_r));
  }
  return CAVITY_OK;
}

int upload_consts(cavity *h) {
  for (int c = 0; c < h->ncav; ++c) {
    fill_consts(h, c);
    const size_t nw = (size_t)h->descs[c].ny * h->descs[c].nz;
    double *tw = h->twall.data() + h->hcc[c].wall_off;
    if (!h->wall_custom[2 * c]) std::fill(tw, tw + nw, h->prms[c].t_hot);
    if (!h->wall_custom[2 * c + 1]) std::fill(tw + nw, tw + 2 * nw, h->prms[c].t_cold);
  }
  int rc = upload_tables(h);
  if (rc != CAVITY_OK) return rc;
  CK(cudaMemcpyAsync(h->d_twall, h->twall.data(), sizeof(double) * h->twall.size(), cudaMemcpyHostToDevice, h->stream));
  CK(cudaStreamSynchronize(h->stream));  // the host vectors may change after return
  return CAVITY_OK;
}

// ---------------------------------------------------------------------------
// kernel launches

// partials of step `s` of a graph
double *step_partials(cavity *h, int s) { return h->d_step_part + (size_t)s * h->part_cap * kPartStride; }

StepArgs step_args(cavity *h, int parity, int mode, int s) {
  StepArgs a;
  a.blocks = h->d_blocks; a.nblocks = h->nblocks; a.cc = h->d_cc; a.cs = h->d_cs;
  a.partials = step_partials(h, s); a.parity = parity; a.mode = mode;
  a.tile_counter = mode == 0 ? h->d_counter : nullptr;
  a.ntiles = h->n_step; a.local_dt = h->local_dt;
  a.ncoarse = h->n_coarse;
  a.skip_shell = 0;
  a.nnu = 0;
  a.slot = 0;
  a.chained = 0;
  a.dt_out = nullptr;
  return a;
}

StepF32Args step_f32_args(cavity *h, int parity, int s) {
  StepF32Args a;
  a.blocks = h->d_blocks; a.nblocks = h->nblocks; a.cc = h->d_cc; a.cs = h->d_cs;
  a.maps = h->d_maps; a.partials = step_partials(h, s); a.parity = parity; a.local_dt = h->local_dt;
  a.ncoarse = h->n_coarse;
  a.wait_cycles = h->wait_cycles;
  a.withhold_plane = h->withhold_plane;
  a.ghosts_late = h->n_cut > 0;
  return a;
}

BcArgs bc_args(cavity *h, int parity, int mode) {
  BcArgs a;
  a.blocks = h->d_blocks;
  a.faces = h->d_wall;
  a.nfaces = (int)h->hwall.size();
  a.cc = h->d_cc; a.cs = h->d_cs; a.ncav = h->ncav;
  a.step_partials = h->d_step_part; a.bc_partials = h->d_bc_part; a.counter = h->d_counter + kStepSlots;
  a.tile_counter = h->d_counter;
  a.t_wall = h->d_twall; a.parity = parity; a.mode = mode;
  a.shell_begin = a.shell_end = 0;
  a.log = mode == 1 || mode == 3 ? nullptr : h->d_log;  // after a step (modes 0, 4): the step log
  a.log_cap = h->log_cap;
  a.nslices = h->nslices;
  a.wall_ctas = 0;
  a.nu_only = 0;
  a.nsteps = 1;
  a.part_stride = (long long)h->part_cap * kPartStride;
  a.bc_stride = 2LL * h->n_nu;
  a.dt_out = nullptr;
  a.slot = 0;
  a.mid = h->d_fin;
  a.rec = h->d_rec;
  return a;
}

// The finalise of a graph of `nsteps` steps that leaves its state in buffer set
// `parity`, and its CTAs.  In the FP64 form the x walls' Nusselt sums have CTAs
// of their own (the FP32 step kernel leaves them in its partials): those of
// the final state here, of the others in the next step's launch.
BcArgs fin_args(cavity *h, int parity, int nsteps, int *ctas) {
  BcArgs b = bc_args(h, parity, h->f32 ? 4 : 0);
  b.nsteps = nsteps;
  *ctas = nsteps * h->ncav * h->nslices;
  if (!h->f32) {
    b.faces = h->d_xwall;
    b.nfaces = (int)h->hxwall.size();
    b.nu_only = 1;
    b.wall_ctas = h->n_nu;
    *ctas += h->n_nu;
  }
  return b;
}

ExchArgs exch_args(cavity *h, int parity) {
  ExchArgs a;
  a.blocks = h->d_blocks; a.faces = h->d_cut; a.nfaces = (int)h->hcut.size();
  a.buf = (double *)h->d_xbuf; a.parity = parity;
  return a;
}

// A launch, as a programmatic dependent of the launch before it in the same
// stream capture if `pdl` (a step, a k_between or a finalise: each waits for its
// predecessor's completion before it touches anything that one writes).
template <class K, class... A>
cudaError_t launch_chained(cavity *h, bool pdl, K kernel, int grid, dim3 block, size_t smem, A... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = h->stream;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// The persistent FP64 step kernel of the handle's tile size (32 * ty threads,
// as many CTAs as fit on the GPU at once, after the Nusselt sums' ones); without
// a tile counter one CTA per tile.
cudaError_t launch_step_f64(cavity *h, const StepArgs &a, const BcArgs &d, bool pdl) {
  const int grid = a.nnu + (a.tile_counter ? std::min(h->n_step, h->persist_ctas) : h->n_step);
  return launch_chained(h, pdl, f64_kernel(h->ty, h->form_walls), grid, dim3(kTX * h->ty), 0, a, d);
}

cudaError_t launch_step_f32(cavity *h, const StepF32Args &a, bool pdl) {
#define BDC_LAUNCH(P, TY, R)                                                                                   \
  if (h->f32_p == P && h->ty == TY && h->f32_r == R)                                                           \
    return launch_chained(h, pdl, f32_kernel<P, TY, R>(), h->n_step, dim3(kF32TX / 2, TY), f32_smem_bytes(TY, R), a);
  BDC_F32_VARIANTS(BDC_LAUNCH)
#undef BDC_LAUNCH
  return cudaErrorInvalidValue;
}

// Whether a step takes dt and the centre shift from the one before it by itself
// (an undivided FP64 cavity whose walls the step forms) instead of from a
// k_between: 32^3 11.6 us a step (12.2 with it), 16^3 9.6 (10.9).  The FP32-mixed
// step has no register left for it (126 of 128 a thread; the code costs it 7%),
// and an exchange or stored walls need the kernel in between anyway.
bool self_chained(const cavity *h) { return !h->f32 && h->ncav == 1 && h->n_cut == 0 && h->form_walls; }

void chain_step(StepArgs &a, int s) {  // step s of a sequence
  a.slot = s % kStepSlots;
  a.chained = s > 0;
  a.tile_counter += a.slot;
}

// The kernel of step `s` of a graph, reading buffer set `parity`.  From the
// second step on it is a programmatic dependent of the step or the k_between
// before it; the first gets a plain launch.
cudaError_t launch_step_kernel(cavity *h, int parity, int s) {
  if (!h->f32) {
    StepArgs a = step_args(h, parity, 0, s);
    if (self_chained(h)) chain_step(a, s);
    int ctas = 0;
    BcArgs d = fin_args(h, parity, 1, &ctas);
    if (s > 0) {
      a.nnu = h->n_nu;
      d.bc_partials += (s - 1) * d.bc_stride;
    }
    return launch_step_f64(h, a, d, s > 0);
  }
  return launch_step_f32(h, step_f32_args(h, parity, s), s > 0);
}

void launch_spectral(cavity *h) {
  const StepArgs sa = step_args(h, h->parity, 1, 0);
  if (h->f32) {
#define BDC_SPEC(P, TY, R)                                                                                       \
  if (h->f32_p == P && h->ty == TY && h->f32_r == R)                                                             \
    k_spectral<float, kF32TX, TY><<<h->n_step, dim3(kF32TX, TY), 0, h->stream>>>(sa);
    BDC_F32_VARIANTS(BDC_SPEC)
#undef BDC_SPEC
  } else {
    launch_step_f64(h, sa, BcArgs{}, false);
  }
}

// Walls of the state in buffer set `parity` stored (no sums): the steps form
// them where they read them, so the stored ones are those of the last refresh.
void launch_walls(cavity *h, int parity) {
  const BcArgs b = bc_args(h, parity, 3);
  if (h->f32) k_bc<float><<<h->n_bc, kBcThreads, 0, h->stream>>>(b);
  else k_bc<double><<<h->n_bc, kBcThreads, 0, h->stream>>>(b);
}

FinTail no_tail() {
  FinTail t{};
  t.begin = INT_MAX;
  return t;
}

// A state refresh (no step): walls with the Nusselt partials, then the
// reductions, dt among them.
void launch_refresh(cavity *h, int parity) {
  const BcArgs b = bc_args(h, parity, 1);
  const int nfin = h->ncav * h->nslices;
  if (h->f32) {
    k_bc<float><<<h->n_bc, kBcThreads, 0, h->stream>>>(b);
    k_finalize<float><<<nfin, kFinThreads, 0, h->stream>>>(b, no_tail());
  } else {
    k_bc<double><<<h->n_bc, kBcThreads, 0, h->stream>>>(b);
    k_finalize<double><<<nfin, kFinThreads, 0, h->stream>>>(b, no_tail());
  }
}

// Whether a step leaves its state's walls stored: where the next one reads them, be it
// the step kernel of a large FP64 cavity or the overlapped schedule's shell kernel.
bool stores_walls(const cavity *h) { return !h->f32 && (!h->form_walls || h->overlap); }

// The finalise of `nsteps` steps; the state in buffer set `parity` gets its
// ghost layers and stored walls in the same launch.  (blocks: other descriptors than
// the handle's, of an undivided cavity.)
cudaError_t launch_finalize(cavity *h, int parity, int nsteps, bool pdl, const BlockDev *blocks = nullptr) {
  int ctas = 0;
  BcArgs b = fin_args(h, parity, nsteps, &ctas);
  FinTail t{ctas, h->n_cut, exch_args(h, parity), bc_args(h, parity, 3)};
  if (blocks) b.blocks = t.walls.blocks = blocks;
  ctas += h->n_cut + (stores_walls(h) ? h->n_bc : 0);
  if (h->f32) return launch_chained(h, pdl, k_finalize<float>, ctas, dim3(kFinThreads), 0, b, t);
  return launch_chained(h, pdl, k_finalize<double>, ctas, dim3(kFinThreads), 0, b, t);
}

// What the step after the one that left its state in buffer set `parity` waits
// for (dt, the centre shift, ghost layers, stored walls).
cudaError_t launch_between(cavity *h, int parity, bool pdl) {
  const ExchArgs x = exch_args(h, parity);
  const BcArgs b = bc_args(h, parity, 3);
  const int grid = h->ncav + h->n_cut + (stores_walls(h) ? h->n_bc : 0);
  if (h->f32) return launch_chained(h, pdl, k_between<float>, grid, dim3(kBetweenThreads), 0, x, b, h->n_cut);
  return launch_chained(h, pdl, k_between<double>, grid, dim3(kBetweenThreads), 0, x, b, h->n_cut);
}

void launch_pack(cavity *h, int parity, cudaStream_t s = nullptr) {
  if (!s) s = h->stream;
  if (h->f32) k_pack<float><<<h->n_cut, 256, 0, s>>>(exch_args(h, parity));
  else k_pack<double><<<h->n_cut, 256, 0, s>>>(exch_args(h, parity));
}

void launch_unpack(cavity *h, int parity, cudaStream_t s = nullptr) {
  if (!s) s = h->stream;
  if (h->f32) k_unpack<float><<<h->n_cut, 256, 0, s>>>(exch_args(h, parity));
  else k_unpack<double><<<h->n_cut, 256, 0, s>>>(exch_args(h, parity));
}

int launch_exchange(cavity *h, int parity) {
  if (h->n_cut == 0) return CAVITY_OK;
  launch_pack(h, parity);
  CK(cudaGetLastError());
  launch_unpack(h, parity);
  CK(cudaGetLastError());
  return CAVITY_OK;
}

// second stream and the fork/join events (created once): of the overlapped step, of the
// step log's records
cudaError_t ensure_side(cavity *h) {
  cudaError_t e = cudaSuccess;
  if (!h->side) e = cudaStreamCreateWithFlags(&h->side, cudaStreamNonBlocking);
  if (e == cudaSuccess && !h->ev_shell) e = cudaEventCreateWithFlags(&h->ev_shell, cudaEventDisableTiming);
  if (e == cudaSuccess && !h->ev_exch) e = cudaEventCreateWithFlags(&h->ev_exch, cudaEventDisableTiming);
  return e;
}

// The overlapped step (FP64, cut faces): shell nodes first, then the
// exchange of the new ghost layers on the side stream while the persistent
// kernel steps the remaining nodes; walls and the finalise after both.
int launch_step_overlapped(cavity *h, int parity) {
  const ShellArgs sa{h->d_blocks, h->d_shell, (int)h->hshell.size(), h->d_cc, h->d_cs, h->d_step_part,
                     (long long)h->n_step, parity, h->local_dt};
  k_shell_f64<<<h->n_shell, kShellThreads, 0, h->stream>>>(sa);
  CK(cudaGetLastError());
  CK(cudaEventRecord(h->ev_shell, h->stream));
  CK(cudaStreamWaitEvent(h->side, h->ev_shell, 0));
  launch_pack(h, parity ^ 1, h->side);
  launch_unpack(h, parity ^ 1, h->side);
  CK(cudaGetLastError());
  CK(cudaEventRecord(h->ev_exch, h->side));
  StepArgs st = step_args(h, parity, 0, 0);
  st.skip_shell = 1;
  CK(launch_step_f64(h, st, BcArgs{}, false));
  CK(cudaStreamWaitEvent(h->stream, h->ev_exch, 0));
  // the finalise with the walls (and their Nusselt partials) in the same launch
  BcArgs ba = bc_args(h, parity ^ 1, 0);
  ba.wall_ctas = h->n_bc;
  ba.shell_begin = h->n_step;
  ba.shell_end = (long long)h->n_step + h->n_shell;
  k_finalize<double><<<h->ncav * h->nslices + h->n_bc, kFinThreads, 0, h->stream>>>(ba, no_tail());
  CK(cudaGetLastError());
  return CAVITY_OK;
}

// The step log's record of step `s` of a sequence, on the side stream, after the step launched last.
int launch_record(cavity *h, int parity, int s) {
  int ctas = 0;
  BcArgs b = fin_args(h, parity, 1, &ctas);
  b.step_partials = step_partials(h, s);
  b.bc_partials += s * b.bc_stride;
  CK(cudaEventRecord(h->ev_shell, h->stream));
  CK(cudaStreamWaitEvent(h->side, h->ev_shell, 0));
  k_step_record<<<h->ncav, kFinThreads, 0, h->side>>>(b, s);
  CK(cudaGetLastError());
  return CAVITY_OK;
}

// nsteps explicit steps from buffer set `parity` (launched, or captured into a
// graph): the steps one after another, then one finalise launch for all of them.
// With a step log the records of all but the last two (the finalise's) are written
// beside the steps.
int launch_steps(cavity *h, int parity, int nsteps) {
  const bool records = h->d_log && nsteps > 2;
  for (int s = 0; s < nsteps; ++s, parity ^= 1) {
    if (h->overlap) {
      const int rc = launch_step_overlapped(h, parity);
      if (rc != CAVITY_OK) return rc;
      continue;
    }
    CK(launch_step_kernel(h, parity, s));
    if (records && s >= 1 && s <= nsteps - 2) {
      const int rc = launch_record(h, parity, s - 1);
      if (rc != CAVITY_OK) return rc;
    }
    if (s == nsteps - 1) {
      if (records) {  // the finalise moves on the time, which the records start from
        CK(cudaEventRecord(h->ev_exch, h->side));
        CK(cudaStreamWaitEvent(h->stream, h->ev_exch, 0));
      }
      CK(launch_finalize(h, parity ^ 1, nsteps, !records));
    } else if (!self_chained(h)) {
      CK(launch_between(h, parity ^ 1, true));
    }
  }
  return CAVITY_OK;
}

// walls, ghosts, dt and Nusselt of the state in the current buffer set (no step)
int refresh_state(cavity *h) {
  launch_spectral(h);
  CK(cudaGetLastError());
  launch_refresh(h, h->parity);
  CK(cudaGetLastError());
  return launch_exchange(h, h->parity);
}

void drop_graphs(cavity *h) {
  for (int q = 0; q < kGraphs; ++q)
    for (int par = 0; par < 2; ++par) {
      if (h->graph[q][par]) cudaGraphExecDestroy(h->graph[q][par]);
      h->graph[q][par] = nullptr;
      h->launched[q][par] = false;
    }
}

// While it lives, this thread may make calls that allocate although one of its
// (or, in global mode, anyone's) streams is being captured.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// The graph of kGraphSteps[q] steps from buffer set `par` (every setter that
// changes a launch drops them), captured on a stream of the handle's own.  A caller
// may be capturing another stream meanwhile: instantiating would be refused then,
// and would end that capture.
int ensure_graph(cavity *h, int q, int par) {
  if (h->graph[q][par]) return CAVITY_OK;
  RelaxedCapture relaxed;
  if (h->overlap) CK(ensure_side(h));
  if (!h->capture) CK(cudaStreamCreateWithFlags(&h->capture, cudaStreamNonBlocking));
  cudaGraph_t g = nullptr;
  CK(cudaStreamBeginCapture(h->capture, cudaStreamCaptureModeRelaxed));
  std::swap(h->stream, h->capture);
  const int rc = launch_steps(h, par, kGraphSteps[q]);
  std::swap(h->stream, h->capture);
  const cudaError_t e = cudaStreamEndCapture(h->capture, &g);
  if (rc != CAVITY_OK) { if (g) cudaGraphDestroy(g); return rc; }
  CK(e);
  const cudaError_t e2 = cudaGraphInstantiate(&h->graph[q][par], g, 0);
  cudaGraphDestroy(g);
  CK(e2);
  CK(cudaGraphUpload(h->graph[q][par], h->stream));  // (its first launch would)
  return CAVITY_OK;
}

// kGraphSteps[q] steps from buffer set `par`: the first two times as the launches
// themselves, from then on as a graph, which the second time builds behind its own
// launches.  So the GPU never waits for a graph to be built, as it did when the call
// that first needed one built it: a first call of 20 steps took FP32-mixed 32^3 329 us
// of device time (189 now, 178 once the graphs are there), 256^3 4379 (4240, 4230), FP64
// 32^3 339 (244, 238).  Steps asked for once build none.
int run_piece(cavity *h, int q, int par) {
  if (h->graph[q][par]) {
    CK(cudaGraphLaunch(h->graph[q][par], h->stream));
    return CAVITY_OK;
  }
  cudaStreamCaptureStatus capturing;
  CK(cudaStreamIsCapturing(h->stream, &capturing));
  if (capturing != cudaStreamCaptureStatusNone)  // as a graph's launch is: its steps would run at every replay
    return fail(h, CAVITY_ERR_CUDA, "the handle's stream is being captured");
  const int rc = launch_steps(h, par, kGraphSteps[q]);
  if (rc != CAVITY_OK) return rc;
  if (h->launched[q][par]) ensure_graph(h, q, par);  // (without one, the next time launches again)
  h->launched[q][par] = true;
  return CAVITY_OK;
}

// The graphs a call of nsteps steps from the present buffer set replays, before it is timed.
int build_graphs(cavity *h, int nsteps) {
  int par = h->parity;
  for (int q = kGraphs - 1; q >= 0; --q)
    for (; kGraphSteps[q] <= h->part_sets && nsteps >= kGraphSteps[q]; nsteps -= kGraphSteps[q]) {
      const int rc = ensure_graph(h, q, par);
      if (rc != CAVITY_OK) return rc;
      par ^= kGraphSteps[q] & 1;
    }
  return CAVITY_OK;
}

int run_steps(cavity *h, int nsteps) {
  for (int q = kGraphs - 1; q >= 0; --q)
    for (; kGraphSteps[q] <= h->part_sets && nsteps >= kGraphSteps[q]; nsteps -= kGraphSteps[q]) {
      const int rc = run_piece(h, q, h->parity);
      if (rc != CAVITY_OK) return rc;
      h->parity ^= kGraphSteps[q] & 1;
      h->steps_taken += kGraphSteps[q];
    }
  return CAVITY_OK;
}

// change the FP32 step kernel's tile shape: work lists, maps, graphs
int retile(cavity *h, int p, int ty, int kc, int r) {
  CK(cudaStreamSynchronize(h->stream));
  h->f32_p = p;
  h->ty = ty;
  h->kc = kc;
  h->f32_r = r;
  h->f32_auto = false;
  assign_tiles(h);
  int rc = ensure_partials(h);
  if (rc == CAVITY_OK) rc = upload_tables(h);
  if (rc == CAVITY_OK) rc = encode_maps(h);
  if (rc != CAVITY_OK) return rc;
  CK(f32_set_smem(p, ty, r));
  drop_graphs(h);
  return CAVITY_OK;
}

int init_state(cavity *h) {
  CK(cudaMemsetAsync(h->d_fields, 0, h->field_bytes, h->stream));
  CK(cudaMemsetAsync(h->d_cs, 0, sizeof(CavState) * h->ncav, h->stream));
  h->parity = 0;
  h->steps_taken = 0;
  for (int id = 0; id < h->nblocks; ++id) {
    const BlockDev &B = h->hb[id];
    const cavity_desc &d = h->descs[B.cav];
    const cavity_params &p = h->prms[B.cav];
    InitArgs a{h->d_blocks, h->d_cc, id, 0, d.seed, d.noise_amp, p.t_hot, p.t_cold};
    const long long n = (long long)B.nx * B.ny * B.nz;
    if (h->f32) k_init<float><<<ceil_div(n, 256), 256, 0, h->stream>>>(a);
    else k_init<double><<<ceil_div(n, 256), 256, 0, h->stream>>>(a);
    CK(cudaGetLastError());
  }
  return refresh_state(h);
}

// device staging buffer of at least n doubles for host transfers (grown on demand)
int ensure_stage(cavity *h, size_t n) {
  if (h->d_stage && h->stage_elems >= n) return CAVITY_OK;
  CK(cudaStreamSynchronize(h->stream));
  if (h->d_stage) {
    cudaFree(h->d_stage);
    h->d_stage = nullptr;
    h->stage_elems = 0;
  }
  CK(cudaMalloc(&h->d_stage, n * sizeof(double)));
  h->stage_elems = n;
  return CAVITY_OK;
}

int popcount5(int m) {
  int c = 0;
  for (int f = 0; f < kNF; ++f) c += (m >> f) & 1;
  return c;
}

int read_states(cavity *h, std::vector<CavState> &st) {
  st.resize(h->ncav);
  CK(cudaMemcpyAsync(st.data(), h->d_cs, sizeof(CavState) * h->ncav, cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return CAVITY_OK;
}

int read_state(cavity *h, int cav, CavState *st) {
  CK(cudaMemcpyAsync(st, h->d_cs + cav, sizeof(CavState), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return CAVITY_OK;
}

int state_status(const CavState &st) {
  if (st.flags & 2) return CAVITY_ERR_TIMEOUT;
  if (st.flags & 1) return CAVITY_ERR_NONFINITE;
  return CAVITY_OK;
}

int all_status(cavity *h) {
  std::vector<CavState> st;
  int rc = read_states(h, st);
  if (rc != CAVITY_OK) return rc;
  int worst = CAVITY_OK;
  for (const CavState &s : st) {
    const int r = state_status(s);
    if (r == CAVITY_ERR_TIMEOUT) return r;
    if (r != CAVITY_OK) worst = r;
  }
  return worst;
}

int get_fields_cav(cavity *h, int cav, int mask, double *host, size_t count) {
  if (!host || mask <= 0 || mask > CAVITY_FIELD_ALL || cav < 0 || cav >= h->ncav) return CAVITY_ERR_INVALID_ARG;
  const cavity_desc &d = h->descs[cav];
  const size_t N = (size_t)d.nx * d.ny * d.nz;
  if (count != (size_t)popcount5(mask) * N) return fail(h, CAVITY_ERR_INVALID_ARG, "count mismatch");
  DeviceGuard g(h->dev);
  int rc = ensure_stage(h, count);
  if (rc != CAVITY_OK) return rc;
  CavState st;
  rc = read_state(h, cav, &st);
  if (rc != CAVITY_OK) return rc;
  for (int id = 0; id < h->nblocks; ++id) {
    const BlockDev &B = h->hb[id];
    if (B.cav != cav) continue;
    MoveArgs a{h->d_blocks, id, h->parity, mask, {d.nx, d.ny, d.nz}, h->d_stage, st.c};
    const int grid = ceil_div((long long)B.nx * B.ny * B.nz, 256);
    if (h->f32) k_gather<float><<<grid, 256, 0, h->stream>>>(a);
    else k_gather<double><<<grid, 256, 0, h->stream>>>(a);
    CK(cudaGetLastError());
  }
  CK(cudaMemcpyAsync(host, h->d_stage, count * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return CAVITY_OK;
}

// The reverse sweep's chunk depth and CTAs: 32 x kAdjTY columns; the depth that
// makes (waves + 0.25) x (depth + 2.5) least, waves the mean of the exact and the
// rounded-up number, at least 1.5 in all: a chunk sweeps four planes of z terms
// beside its own (2.5 planes' work), and the last CTAs run half alone.  What it picks
// against a sweep over the depths, us a reverse step: 128^3 FP32 110.0 at 15 planes (110.5 at 10,
// 108.5 at 14, 117.7 at 8, 123 at 19, 126 at 32), 64^3 FP32 32.8 at 2 (28.3 at 4), 97x65x50 FP32 42.2 at
// 4 (37.8 at 7), FP64 390 (359 at 3); FP64 32^3 46.0 at 1 (71.7 at 2), 48^3 124.8 at 4 (136 at 2):
// the best but for up to 16% at sizes whose last wave is nearly empty.
int adj_tiling(cavity *h, int *kc, int *ctas) {
  const cavity_desc &d = h->descs[0];
  int per_sm = 1;
  if (h->f32) {
    constexpr int smem = (int)adj_smem_bytes<float, kAdjTY>();
    CK(cudaFuncSetAttribute(k_adj_sweep<float, kAdjTY>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_adj_sweep<float, kAdjTY>, 32 * kAdjTY, smem));
  } else {
    constexpr int smem = (int)adj_smem_bytes<double, kAdjTY>();
    CK(cudaFuncSetAttribute(k_adj_sweep<double, kAdjTY>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_adj_sweep<double, kAdjTY>, 32 * kAdjTY, smem));
  }
  const long long xy = (long long)ceil_div(d.nx, 32) * ceil_div(d.ny, kAdjTY);
  const int slots = h->nsm * std::max(per_sm, 1);
  double best = 1e300;
  for (int k = 1; k <= d.nz; ++k) {
    const long long tiles = xy * ceil_div(d.nz, k);
    const double cost = std::max(1.5, 0.5 * ((double)tiles / slots + ceil_div(tiles, slots)) + 0.25) * (k + 2.5);
    if (cost < best) {
      best = cost;
      *kc = k;
      *ctas = (int)tiles;
    }
  }
  return CAVITY_OK;
}

// Per segment slot: its block descriptor (slot s read, slot s + 1 written), its
// wall faces (one walls launch covers the segment) and, in the FP32 form, its
// tensor maps; made again when the tiling has changed.
int adj_tables(cavity *h) {
  AdjointStore &A = h->adj;
  const int ckpt = A.ckpt;
  if (A.layout != h->layout) {
    std::vector<BlockDev> sb(ckpt, h->hb[0]);
    std::vector<WallFace> sf;
    for (int s = 0; s < ckpt; ++s) {
      sb[s].base[0] = A.seg_mem + (size_t)s * A.set_bytes;
      sb[s].base[1] = A.seg_mem + (size_t)std::min(s + 1, ckpt - 1) * A.set_bytes;
      for (WallFace f : h->hwall) {
        f.block = s;
        f.cta_begin += s * h->n_bc;
        sf.push_back(f);
      }
    }
    CK(cudaMemcpyAsync(A.seg_blocks, sb.data(), sizeof(BlockDev) * sb.size(), cudaMemcpyHostToDevice, h->stream));
    CK(cudaMemcpyAsync(A.seg_faces, sf.data(), sizeof(WallFace) * sf.size(), cudaMemcpyHostToDevice, h->stream));
    std::vector<CUtensorMap> sm;
    if (h->f32) {
      sm.resize(2 * (size_t)ckpt);
      for (int s = 0; s < ckpt; ++s) {
        const int rc = encode_block_maps(h, h->hb[0], A.seg_mem + (size_t)s * A.set_bytes, &sm[2 * s]);
        if (rc != CAVITY_OK) return rc;
      }
      CK(cudaMemcpyAsync(A.seg_maps, sm.data(), sizeof(CUtensorMap) * sm.size(), cudaMemcpyHostToDevice, h->stream));
    }
    CK(cudaStreamSynchronize(h->stream));  // the host vectors end here
    A.layout = h->layout;
  }
  return CAVITY_OK;
}

// The constant walls (u = v = w = 0, the isothermal T) in every slot: the forward run's,
// which the reverse sweep recomputes with whatever the handle has been given since.
int adj_walls(cavity *h) {
  AdjointStore &A = h->adj;
  const int ckpt = A.ckpt;
  BcArgs ba = bc_args(h, 0, 5);
  ba.blocks = A.seg_blocks;
  ba.faces = A.seg_faces;
  ba.nfaces = (int)h->hwall.size() * ckpt;
  if (h->f32) k_bc<float><<<h->n_bc * ckpt, kBcThreads, 0, h->stream>>>(ba);
  else k_bc<double><<<h->n_bc * ckpt, kBcThreads, 0, h->stream>>>(ba);
  CK(cudaGetLastError());
  return CAVITY_OK;
}

// A recomputed step: slot s to slot s + 1 (nothing is finalised, but for a step log)
cudaError_t launch_recompute(cavity *h, int s, bool pdl) {
  const AdjointStore &A = h->adj;
  if (!h->f32) {
    StepArgs a = step_args(h, 0, 0, 0);
    if (self_chained(h) && !h->d_log) chain_step(a, s);
    a.dt_out = A.dts + s;
    a.blocks = A.seg_blocks + s;
    return launch_step_f64(h, a, BcArgs{}, pdl);
  }
  StepF32Args a = step_f32_args(h, 0, 0);
  a.blocks = A.seg_blocks + s;
  a.maps = A.seg_maps + 2 * s;
  return launch_step_f32(h, a, pdl);
}

// dt, the centre shift (and stored walls) of slot s for the recomputed step after it,
// or for the reverse step from the segment's last state
cudaError_t launch_recompute_between(cavity *h, int s) {
  const AdjointStore &A = h->adj;
  ExchArgs x = exch_args(h, 0);
  BcArgs b = bc_args(h, 0, 3);
  x.blocks = b.blocks = A.seg_blocks + s;
  b.dt_out = A.dts + s;
  b.slot = self_chained(h) ? (s - 1) % kStepSlots : 0;
  const int grid = 1 + (stores_walls(h) ? h->n_bc : 0);
  if (h->f32) return launch_chained(h, true, k_between<float>, grid, dim3(kBetweenThreads), 0, x, b, 0);
  return launch_chained(h, true, k_between<double>, grid, dim3(kBetweenThreads), 0, x, b, 0);
}

void free_adjoint(AdjointStore &A) {
  if (A.mem) cudaFree(A.mem);
  A = AdjointStore{};
}

void release(cavity *h) {
  DeviceGuard g(h->dev);
  if (h->stream) cudaStreamSynchronize(h->stream);
  drop_graphs(h);
  void *ptrs[] = {h->d_fields, h->d_blocks, h->d_cc, h->d_cs, h->d_wall, h->d_cut, h->d_step_part,
                  h->d_bc_part, h->d_counter, h->d_twall, h->d_xbuf, h->d_stage, h->d_maps, h->d_fin, h->d_rec, h->d_shell, h->d_xwall};
  for (void *p : ptrs)
    if (p) cudaFree(p);
  AdjointStore &A = h->adj;
  free_adjoint(A);
  if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
  if (h->side) cudaStreamDestroy(h->side);
  if (h->capture) cudaStreamDestroy(h->capture);
  if (h->ev_shell) cudaEventDestroy(h->ev_shell);
  if (h->ev_exch) cudaEventDestroy(h->ev_exch);
  for (cudaEvent_t e : h->adj_ev) cudaEventDestroy(e);
  h->adj_ev.clear();
}

int create_common(const cavity_desc *descs, const cavity_params *params, int n, cavity_t **out) {
  if (!out) return CAVITY_ERR_INVALID_ARG;
  *out = nullptr;
  if (!descs || n < 1) return CAVITY_ERR_INVALID_ARG;
  for (int c = 0; c < n; ++c) {
    if (check_desc(descs[c]) != CAVITY_OK) return CAVITY_ERR_INVALID_ARG;
    if (n > 1 && (descs[c].px != 1 || descs[c].py != 1 || descs[c].pz != 1)) return CAVITY_ERR_INVALID_ARG;
    if (descs[c].precision != descs[0].precision) return CAVITY_ERR_INVALID_ARG;
    if (params) {
      cavity_params q = params[c];
      resolve_defaults(&q);
      if (check_params(q) != CAVITY_OK) return CAVITY_ERR_INVALID_ARG;
    }
  }
  const cavity_desc &d0 = descs[0];
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || d0.device < 0 || d0.device >= ndev) return CAVITY_ERR_CUDA;
  cavity *h = new (std::nothrow) cavity();
  if (!h) return CAVITY_ERR_OOM;
  h->ncav = n;
  h->descs.assign(descs, descs + n);
  h->prms.resize(n);
  for (int c = 0; c < n; ++c) {
    if (params) {
      h->prms[c] = params[c];
      resolve_defaults(&h->prms[c]);
    } else {
      cavity_default_params(&h->prms[c]);
    }
  }
  h->hcc.assign(n, CavConst{});
  h->wall_custom.assign(2 * n, 0);
  h->dev = d0.device;
  h->f32 = d0.precision == CAVITY_FP32_MIXED;
  h->esize = h->f32 ? 4 : 8;
  h->na = h->f32 ? Store<float>::NA : Store<double>::NA;
  h->np = h->f32 ? Store<float>::NP : Store<double>::NP;
  if (!h->f32) {
    // tile-height override for tuning sweeps: BDC_F64_TY=4 or 8
    if (const char *env = std::getenv("BDC_F64_TY")) {
      const int ty = std::atoi(env);
      if (ty == 4 || ty == 8) h->ty = ty;
    }
  }
  if (h->f32) {
    h->tx = kF32TX;
    h->ty = kF32TY;
    h->f32_r = kF32R;
    h->f32_p = 3;
    // shape override for tuning sweeps: BDC_F32_TILE="TY,KC,R[,P]" (a compiled shape)
    if (const char *env = std::getenv("BDC_F32_TILE")) {
      int ty = 0, kc = 0, r = 0, p = 3;
      const int got = std::sscanf(env, "%d,%d,%d,%d", &ty, &kc, &r, &p);
      if (got >= 3 && f32_variant_ok(p, ty, kc, r)) {
        h->ty = ty;
        h->kc = kc;
        h->f32_r = r;
        h->f32_p = p;
        h->f32_auto = false;
      }
    }
  }
  int rc = CAVITY_OK;
  {
    DeviceGuard g(h->dev);
    if (d0.stream) {
      h->stream = (cudaStream_t)d0.stream;
    } else {
      if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) rc = CAVITY_ERR_CUDA;
      h->own_stream = true;
    }
    if (rc == CAVITY_OK && cudaDeviceGetAttribute(&h->nsm, cudaDevAttrMultiProcessorCount, h->dev) != cudaSuccess)
      rc = CAVITY_ERR_CUDA;
    if (rc == CAVITY_OK) rc = build_layout(h);
    if (rc == CAVITY_OK) rc = alloc_device(h);
    if (rc == CAVITY_OK) rc = upload_consts(h);
    if (rc == CAVITY_OK) rc = init_state(h);
    if (rc == CAVITY_OK && cudaStreamSynchronize(h->stream) != cudaSuccess) rc = CAVITY_ERR_CUDA;
  }
  if (rc != CAVITY_OK) {
    release(h);
    delete h;
    return rc;
  }
  *out = h;
  return CAVITY_OK;
}

}  // namespace

// ===========================================================================
// cavity_check_sqrt: relative difference of sqrt_newton from CUDA's sqrt
__global__ void k_check_sqrt(const double *x, long long n, double *rel) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double r = sqrt(x[i]), s = sqrt_newton(x[i]);
  rel[i] = s == r ? 0.0 : fabs(s - r) / r;
}

// cavity_check_div3: whether div3 equals CUDA's correctly rounded x / 3
__global__ void k_check_div3(const double *x, long long n, unsigned char *diff) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  diff[i] = div3(x[i]) != x[i] / 3.0;
}

// FP64 FMA throughput of the GPU: every thread runs kDfmaChains independent
// chains x <- x a + b (a = 1 - 2^-20, b = 2^-20: the values stay near 1, no
// overflow or subnormals), unrolled so that the FP64 pipe always has an
// independent FMA to issue; the sum is compared with a value it never takes,
// so no chain can be removed.  FLOPs = 2 per FMA.
constexpr int kDfmaChains = 8, kDfmaUnroll = 4, kDfmaThreads = 256;
__global__ void __launch_bounds__(kDfmaThreads) k_dfma_peak(double *sink, int iters, double a, double b) {
  double x[kDfmaChains];
#pragma unroll
  for (int c = 0; c < kDfmaChains; ++c) x[c] = 1.0 + 1e-3 * (threadIdx.x + c);
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int r = 0; r < kDfmaUnroll; ++r)
#pragma unroll
      for (int c = 0; c < kDfmaChains; ++c) x[c] = fma(x[c], a, b);
  }
  double s = 0.0;
#pragma unroll
  for (int c = 0; c < kDfmaChains; ++c) s += x[c];
  if (s == -1.0) sink[blockIdx.x] = s;
}

extern "C" {

int cavity_default_params(cavity_params *p) {
  if (!p) return CAVITY_ERR_INVALID_ARG;
  p->Ra = 1e5; p->Pr = 0.71; p->cfl = 0.5; p->kappa = 0.1; p->c4 = 1.0 / 32.0;
  p->u_ref = -1.0; p->t_inf = NAN; p->t_hot = 1.0; p->t_cold = 0.0; p->gravity_axis = 2;
  resolve_defaults(p);
  return CAVITY_OK;
}

int cavity_create(const cavity_desc *desc, cavity_t **out) { return create_common(desc, nullptr, 1, out); }

int cavity_create_batch(const cavity_desc *descs, const cavity_params *params, int n, cavity_t **out) {
  return create_common(descs, params, n, out);
}

int cavity_batch_size(cavity_t *h) { return h ? h->ncav : CAVITY_ERR_INVALID_ARG; }

int cavity_set_params(cavity_t *h, const cavity_params *p) {
  if (!h || !p) return CAVITY_ERR_INVALID_ARG;
  cavity_params q = *p;
  const bool auto_uref = !(q.u_ref >= 0.0);
  resolve_defaults(&q);
  if (check_params(q) != CAVITY_OK) return fail(h, CAVITY_ERR_INVALID_ARG, "invalid parameters");
  DeviceGuard g(h->dev);
  CK(cudaStreamSynchronize(h->stream));
  h->u_ref_auto = auto_uref;
  for (auto &pc : h->prms) pc = q;
  h->setup += 1;
  int rc = upload_consts(h);
  if (rc != CAVITY_OK) return rc;
  if (h->steps_taken == 0) return init_state(h);
  return refresh_state(h);
}

int cavity_set_wall_temperature(cavity_t *h, int wall, const double *host, size_t n) {
  if (!h || !host || (wall != 0 && wall != 1)) return CAVITY_ERR_INVALID_ARG;
  const size_t nw = (size_t)h->descs[0].ny * h->descs[0].nz;
  if (n != nw) return fail(h, CAVITY_ERR_INVALID_ARG, "wall temperature count must be ny*nz");
  for (size_t q = 0; q < n; ++q)
    if (!std::isfinite(host[q])) return fail(h, CAVITY_ERR_INVALID_ARG, "non-finite wall temperature");
  DeviceGuard g(h->dev);
  CK(cudaStreamSynchronize(h->stream));
  std::copy(host, host + n, h->twall.begin() + h->hcc[0].wall_off + (wall ? nw : 0));
  h->wall_custom[wall] = 1;
  h->setup += 1;
  int rc = upload_consts(h);
  if (rc != CAVITY_OK) return rc;
  return refresh_state(h);
}

int cavity_step(cavity_t *h, int nsteps) {
  if (!h || nsteps < 0) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(h->dev);
  return run_steps(h, nsteps);
}

int cavity_batch_state(cavity_t *h, int cav, double out[10]) {
  if (!h || !out || cav < 0 || cav >= h->ncav) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(h->dev);
  CavState st;
  int rc = read_state(h, cav, &st);
  if (rc != CAVITY_OK) return rc;
  out[0] = (double)st.step;
  out[1] = st.t;
  out[2] = st.dt;
  for (int f = 0; f < 5; ++f) out[3 + f] = st.res[f];
  out[8] = st.nu_hot;
  out[9] = st.nu_cold;
  return state_status(st);
}

int cavity_batch_get_fields(cavity_t *h, int cav, int mask, double *host, size_t count) {
  if (!h) return CAVITY_ERR_INVALID_ARG;
  return get_fields_cav(h, cav, mask, host, count);
}

static_assert(sizeof(StepRecord) == sizeof(cavity_step_record), "step record layout");
static_assert(offsetof(StepRecord, flags) == offsetof(cavity_step_record, flags), "step record layout");

int cavity_set_step_log(cavity_t *h, cavity_step_record *host, long long capacity) {
  if (!h) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(h->dev);
  StepRecord *dev = nullptr;
  if (host) {
    if (capacity < 1) return fail(h, CAVITY_ERR_INVALID_ARG, "step log: capacity < 1");
    cudaPointerAttributes pa;
    if (cudaPointerGetAttributes(&pa, host) != cudaSuccess || pa.type != cudaMemoryTypeHost || !pa.devicePointer) {
      cudaGetLastError();
      return fail(h, CAVITY_ERR_INVALID_ARG, "step log: not page-locked host memory the device can address");
    }
    dev = (StepRecord *)pa.devicePointer;
  }
  CK(cudaStreamSynchronize(h->stream));
  if (host) CK(ensure_side(h));  // the records' stream
  h->d_log = dev;
  h->log_cap = host ? capacity : 0;
  drop_graphs(h);  // the finalise launches in the graphs carry the log
  return CAVITY_OK;
}

int cavity_step_log_alloc(long long records, cavity_step_record **out) {
  if (!out || records < 1 || records > (1LL << 32)) return CAVITY_ERR_INVALID_ARG;
  *out = nullptr;
  void *p = nullptr;
  const size_t bytes = (size_t)records * sizeof(cavity_step_record);
  if (cudaHostAlloc(&p, bytes, cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess) {
    cudaGetLastError();
    return CAVITY_ERR_OOM;
  }
  std::memset(p, 0, bytes);
  *out = (cavity_step_record *)p;
  return CAVITY_OK;
}

int cavity_step_log_free(cavity_step_record *p) {
  if (p && cudaFreeHost(p) != cudaSuccess) return CAVITY_ERR_CUDA;
  return CAVITY_OK;
}

int cavity_residual(cavity_t *h, double out[5]) {
  if (!h || !out) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(h->dev);
  CavState st;
  int rc = read_state(h, 0, &st);
  if (rc != CAVITY_OK) return rc;
  for (int f = 0; f < 5; ++f) out[f] = st.res[f];
  return state_status(st);
}

int cavity_nusselt(cavity_t *h, double *hot, double *cold) {
  if (!h) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(h->dev);
  CavState st;
  int rc = read_state(h, 0, &st);
  if (rc != CAVITY_OK) return rc;
  if (hot) *hot = st.nu_hot;
  if (cold) *cold = st.nu_cold;
  return state_status(st);
}

int cavity_get_time(cavity_t *h, long long *step, double *t, double *dt) {
  if (!h) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(h->dev);
  CavState st;
  int rc = read_state(h, 0, &st);
  if (rc != CAVITY_OK) return rc;
  if (step) *step = st.step;
  if (t) *t = st.t;
  if (dt) *dt = st.dt;
  return state_status(st);
}

int cavity_get_fields(cavity_t *h, int mask, double *host, size_t count) {
  if (!h) return CAVITY_ERR_INVALID_ARG;
  return get_fields_cav(h, 0, mask, host, count);
}

int cavity_get_fields_box(cavity_t *h, int mask, int i0, int j0, int k0, int ni, int nj, int nk, double *host,
                          size_t count) {
  if (!h || !host || mask <= 0 || mask > CAVITY_FIELD_ALL) return CAVITY_ERR_INVALID_ARG;
  const cavity_desc &d = h->descs[0];
  if (ni < 1 || nj < 1 || nk < 1 || i0 < 1 || j0 < 1 || k0 < 1 || i0 + ni - 1 > d.nx || j0 + nj - 1 > d.ny ||
      k0 + nk - 1 > d.nz)
    return fail(h, CAVITY_ERR_INVALID_ARG, "box outside the interior");
  const size_t n = (size_t)ni * nj * nk;
  if (count != (size_t)popcount5(mask) * n) return fail(h, CAVITY_ERR_INVALID_ARG, "count mismatch");
  DeviceGuard g(h->dev);
  int rc = ensure_stage(h, count);
  if (rc != CAVITY_OK) return rc;
  CavState st;
  rc = read_state(h, 0, &st);
  if (rc != CAVITY_OK) return rc;
  int nb0 = 0;  // blocks of cavity 0
  while (nb0 < h->nblocks && h->hb[nb0].cav == 0) ++nb0;
  BoxArgs a{h->d_blocks, nb0, h->parity, mask, i0, j0, k0, ni, nj, nk, h->d_stage, st.c};
  if (h->f32) k_gather_box<float><<<ceil_div((long long)n, 256), 256, 0, h->stream>>>(a);
  else k_gather_box<double><<<ceil_div((long long)n, 256), 256, 0, h->stream>>>(a);
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(host, h->d_stage, count * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return CAVITY_OK;
}

int cavity_set_fields(cavity_t *h, int mask, const double *host, size_t count) {
  if (!h || !host || mask <= 0 || mask > CAVITY_FIELD_ALL) return CAVITY_ERR_INVALID_ARG;
  const cavity_desc &d = h->descs[0];
  const size_t N = (size_t)d.nx * d.ny * d.nz;
  if (count != (size_t)popcount5(mask) * N) return fail(h, CAVITY_ERR_INVALID_ARG, "count mismatch");
  DeviceGuard g(h->dev);
  int rc = ensure_stage(h, count);
  if (rc != CAVITY_OK) return rc;
  CavState st;
  rc = read_state(h, 0, &st);
  if (rc != CAVITY_OK) return rc;
  // fold the pending centre shift into the stored p, then c = 0
  for (int id = 0; id < h->nblocks; ++id) {
    const BlockDev &B = h->hb[id];
    if (B.cav != 0) continue;
    if (st.c != 0.0 && !(mask & CAVITY_FIELD_P)) {
      const int grid = ceil_div((long long)(B.nx + 4) * (B.ny + 4) * (B.nz + 4), 256);
      if (h->f32) k_shift_p<float><<<grid, 256, 0, h->stream>>>(h->d_blocks, id, h->parity, st.c);
      else k_shift_p<double><<<grid, 256, 0, h->stream>>>(h->d_blocks, id, h->parity, st.c);
      CK(cudaGetLastError());
    }
  }
  CK(cudaMemsetAsync(&h->d_cs[0].c, 0, sizeof(double), h->stream));
  CK(cudaMemcpyAsync(h->d_stage, host, count * sizeof(double), cudaMemcpyHostToDevice, h->stream));
  for (int id = 0; id < h->nblocks; ++id) {
    const BlockDev &B = h->hb[id];
    if (B.cav != 0) continue;
    MoveArgs a{h->d_blocks, id, h->parity, mask, {d.nx, d.ny, d.nz}, h->d_stage, 0.0};
    const int grid = ceil_div((long long)B.nx * B.ny * B.nz, 256);
    if (h->f32) k_scatter<float><<<grid, 256, 0, h->stream>>>(a);
    else k_scatter<double><<<grid, 256, 0, h->stream>>>(a);
    CK(cudaGetLastError());
  }
  rc = refresh_state(h);
  if (rc != CAVITY_OK) return rc;
  CK(cudaStreamSynchronize(h->stream));
  return CAVITY_OK;
}

int cavity_num_blocks(cavity_t *h) { return h ? h->nblocks : CAVITY_ERR_INVALID_ARG; }

int cavity_get_block_array(cavity_t *h, int block, int field, double *host, size_t count, int dims[6]) {
  if (!h || block < 0 || block >= h->nblocks || field < 0 || field >= h->na) return CAVITY_ERR_INVALID_ARG;
  const BlockDev &B = h->hb[block];
  const size_t n = (size_t)(B.nx + 4) * (B.ny + 4) * (B.nz + 4);
  if (dims) { dims[0] = B.nx; dims[1] = B.ny; dims[2] = B.nz; dims[3] = B.ox; dims[4] = B.oy; dims[5] = B.oz; }
  if (!host) return count == 0 ? CAVITY_OK : CAVITY_ERR_INVALID_ARG;
  if (count != n) return fail(h, CAVITY_ERR_INVALID_ARG, "count mismatch");
  DeviceGuard g(h->dev);
  int rc = ensure_stage(h, count);
  if (rc != CAVITY_OK) return rc;
  if (!h->f32) launch_walls(h, h->parity);  // (the FP32-mixed form returns them as last refreshed)
  if (h->f32) k_copy_block<float><<<ceil_div((long long)n, 256), 256, 0, h->stream>>>(h->d_blocks, block, h->parity, field, h->d_stage);
  else k_copy_block<double><<<ceil_div((long long)n, 256), 256, 0, h->stream>>>(h->d_blocks, block, h->parity, field, h->d_stage);
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(host, h->d_stage, n * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return CAVITY_OK;
}

int cavity_get_face_buffer(cavity_t *h, int block, int face, double *host, size_t count) {
  if (!h || !host || block < 0 || block >= h->nblocks || face < 0 || face > 5) return CAVITY_ERR_INVALID_ARG;
  for (const CutFace &c : h->hcut) {
    if (c.src != block || c.face != face) continue;
    const size_t n = (size_t)(h->na + h->np) * c.nb * c.nc;
    if (count != n) return fail(h, CAVITY_ERR_INVALID_ARG, "count mismatch");
    DeviceGuard g(h->dev);
    // the step's exchange writes the ghost layers directly: pack the current
    // state's faces (the values every exchange of this state sends)
    launch_pack(h, h->parity);
    CK(cudaGetLastError());
    if (h->f32) {
      std::vector<float> tmp(n);
      CK(cudaMemcpyAsync(tmp.data(), (float *)h->d_xbuf + c.buf_off, n * sizeof(float), cudaMemcpyDeviceToHost,
                         h->stream));
      CK(cudaStreamSynchronize(h->stream));
      for (size_t q = 0; q < n; ++q) host[q] = (double)tmp[q];
    } else {
      CK(cudaMemcpyAsync(host, (double *)h->d_xbuf + c.buf_off, n * sizeof(double), cudaMemcpyDeviceToHost,
                         h->stream));
      CK(cudaStreamSynchronize(h->stream));
    }
    return CAVITY_OK;
  }
  return fail(h, CAVITY_ERR_INVALID_ARG, "face is a wall");
}

int cavity_exchange(cavity_t *h) {
  if (!h) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(h->dev);
  return launch_exchange(h, h->parity);
}

int cavity_autotune(cavity_t *h, int steps, double out[5]) {
  if (!h || steps < 1) return CAVITY_ERR_INVALID_ARG;
  if (!h->f32) return fail(h, CAVITY_ERR_UNSUPPORTED, "the FP64 form has one tile shape");
  DeviceGuard g(h->dev);
  CK(cudaStreamSynchronize(h->stream));
  if (std::getenv("BDC_F32_TILE")) {  // a pinned shape (set at creation): no trials
    if (out) {
      out[0] = h->ty;
      out[1] = h->kc;
      out[2] = h->f32_r;
      out[3] = h->f32_p;
      out[4] = 0.0;
    }
    return CAVITY_OK;
  }
  // save the state (fields, per-cavity scalars, ping-pong parity, step count)
  void *backup = nullptr;
  CK(cudaMalloc(&backup, h->field_bytes));
  std::vector<CavState> st0;
  int rc = read_states(h, st0);
  const int par0 = h->parity;
  const long long steps0 = h->steps_taken;
  auto restore = [&]() -> int {
    CK(cudaMemcpyAsync(h->d_fields, backup, h->field_bytes, cudaMemcpyDeviceToDevice, h->stream));
    CK(cudaMemcpyAsync(h->d_cs, st0.data(), sizeof(CavState) * h->ncav, cudaMemcpyHostToDevice, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    h->parity = par0;
    h->steps_taken = steps0;
    return CAVITY_OK;
  };
  if (rc == CAVITY_OK && cudaMemcpyAsync(backup, h->d_fields, h->field_bytes, cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess)
    rc = fail(h, CAVITY_ERR_CUDA, "state backup failed");
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (rc == CAVITY_OK && (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess))
    rc = fail(h, CAVITY_ERR_CUDA, "event creation failed");
  // one trial of a shape: `steps` graph-replayed steps after a warm-up, from the saved
  // state (their graphs built before: that takes longer than a small cavity's steps)
  auto trial = [&](const F32Shape &s, double &us) -> int {
    int r = retile(h, s.p, s.ty, s.kc, s.r);
    if (r == CAVITY_OK) r = build_graphs(h, steps);
    if (r == CAVITY_OK) r = cavity_step(h, 2);  // warm-up
    if (r != CAVITY_OK) return r;
    cudaEventRecord(e0, h->stream);
    r = cavity_step(h, steps);
    cudaEventRecord(e1, h->stream);
    if (cudaEventSynchronize(e1) != cudaSuccess) r = fail(h, CAVITY_ERR_CUDA, "trial failed");
    if (r != CAVITY_OK) return r;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    us = 1e3 * ms / steps;
    return restore();
  };
  // every shape once, then the four fastest again (each keeps its better
  // time): one trial's noise between close shapes no longer decides
  std::vector<F32Shape> shapes = f32_shapes();
  const size_t listed = shapes.size();
  // and the shape held on entry, where the list has it not: the depth that follows
  // the size goes down to one plane (32^3 8.4 us a step, 23.4 at the list's 16)
  const F32Shape held = {h->f32_p, h->ty, h->kc, h->f32_r};
  const bool in_list = std::any_of(shapes.begin(), shapes.end(), [&](const F32Shape &s) {
    return s.p == held.p && s.ty == held.ty && s.kc == held.kc && s.r == held.r;
  });
  if (!in_list) shapes.push_back(held);
  std::vector<double> t(shapes.size(), 1e300);
  for (size_t q = 0; q < shapes.size() && rc == CAVITY_OK; ++q) rc = trial(shapes[q], t[q]);
  std::vector<size_t> order(shapes.size());
  for (size_t q = 0; q < order.size(); ++q) order[q] = q;
  std::stable_sort(order.begin(), order.end(), [&](size_t x, size_t y) { return t[x] < t[y]; });
  for (size_t q = 0; q < std::min<size_t>(4, order.size()) && rc == CAVITY_OK; ++q) {
    double us = 1e300;
    rc = trial(shapes[order[q]], us);
    t[order[q]] = std::min(t[order[q]], us);
  }
  double best_us = 1e300;
  F32Shape best = held;
  for (size_t q = 0; q < listed; ++q)
    if (t[q] < best_us) {
      best_us = t[q];
      best = shapes[q];
    }
  const F32Shape keep = !in_list && t[listed] <= best_us ? held : best;
  if (rc == CAVITY_OK) rc = retile(h, keep.p, keep.ty, keep.kc, keep.r);
  if (rc == CAVITY_OK) rc = restore();
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaFree(backup);
  if (rc == CAVITY_OK && out) {
    out[0] = best.ty;
    out[1] = best.kc;
    out[2] = best.r;
    out[3] = best.p;
    out[4] = best_us;
  }
  return rc;
}

int cavity_adjoint_forward(cavity_t *h, int nsteps, int ckpt, double *J) {
  if (!h || nsteps < 1 || ckpt < 1) return CAVITY_ERR_INVALID_ARG;
  if (h->local_dt) return fail(h, CAVITY_ERR_UNSUPPORTED, "adjoint: global time stepping only");
  if ((long long)(h->descs[0].nx + 4) * (h->descs[0].ny + 4) * (h->descs[0].nz + 4) >= (1LL << 31))
    return fail(h, CAVITY_ERR_UNSUPPORTED, "adjoint: fewer than 2^31 nodes with the two-node halo");
  if (h->ncav != 1 || h->nblocks != 1) return fail(h, CAVITY_ERR_UNSUPPORTED, "adjoint: single-block cavity only");
  DeviceGuard g(h->dev);
  AdjointStore &A = h->adj;
  const BlockDev &B = h->hb[0];
  const cavity_desc &d = h->descs[0];
  const size_t set_bytes = (size_t)h->na * (size_t)B.fstride * h->esize;
  const int ncp = (nsteps + ckpt - 1) / ckpt;
  CK(cudaStreamSynchronize(h->stream));
  if (A.set_bytes != set_bytes || A.ncp < ncp || A.ckpt < ckpt) {
    free_adjoint(A);
    const size_t abytes = h->esize * 5 * (size_t)B.fstride;
    const int rt = adj_tiling(h, &A.kc, &A.ctas);
    if (rt != CAVITY_OK) return rt;
    // one allocation for all: fifteen of them cost a gradient 350 us (32^3 FP64 4750
    // -> 4400) to 1.4 ms (128^3 FP32, 2.8 GB: 47.9 -> 46.5 ms) more to make and release
    const struct { void **p; size_t bytes; } parts[] = {
        {(void **)&A.ckpt_mem, set_bytes * ncp},
        {(void **)&A.seg_mem, set_bytes * ckpt},
        {(void **)&A.final_mem, set_bytes},
        {(void **)&A.X, abytes},
        {(void **)&A.Q, abytes},
        {(void **)&A.ckpt_cs, sizeof(CavState) * ncp},
        {(void **)&A.thetabar, sizeof(double) * d.ny * d.nz},
        {(void **)&A.scal, sizeof(double) * kScCount},
        {(void **)&A.argpart, sizeof(double) * 2 * kAdjParts * ckpt},  // one set per segment slot
        {(void **)&A.cnt, sizeof(unsigned int)},
        {(void **)&A.gpart, sizeof(double) * 4 * A.ctas},
        {(void **)&A.dts, sizeof(double) * (ckpt + 1)},
        {(void **)&A.seg_blocks, sizeof(BlockDev) * ckpt},
        {(void **)&A.seg_faces, sizeof(WallFace) * h->hwall.size() * ckpt},
        {(void **)&A.seg_maps, h->f32 ? sizeof(CUtensorMap) * 2 * (size_t)ckpt : 0}};
    size_t total = 0;
    for (const auto &q : parts) total += (q.bytes + 511) / 512 * 512;
    CK(cudaMalloc(&A.mem, total));
    total = 0;
    for (const auto &q : parts) {
      *q.p = (char *)A.mem + total;
      total += (q.bytes + 511) / 512 * 512;
    }
    // (a slot's velocity walls stay zero, and nothing a step reads is unset)
    CK(cudaMemsetAsync(A.seg_mem, 0, set_bytes * ckpt, h->stream));
    CK(cudaMemsetAsync(A.cnt, 0, sizeof(unsigned int), h->stream));
    A.set_bytes = set_bytes;
    A.ckpt = ckpt;
    A.ncp = ncp;
  }
  A.have_forward = false;
  int rc = adj_tables(h);
  if (rc == CAVITY_OK) rc = adj_walls(h);
  if (rc != CAVITY_OK) return rc;
  A.nsteps = nsteps;
  A.run_ckpt = ckpt;
  A.setup = h->setup;
  CK(cudaMemsetAsync(&h->d_cs[0].nu_sum, 0, sizeof(double), h->stream));
  for (int n = 0; n < nsteps; n += ckpt) {
    const int c = n / ckpt;
    CK(cudaMemcpyAsync(A.ckpt_mem + (size_t)c * set_bytes, h->hb[0].base[h->parity], set_bytes,
                       cudaMemcpyDeviceToDevice, h->stream));
    CK(cudaMemcpyAsync(A.ckpt_cs + c, h->d_cs, sizeof(CavState), cudaMemcpyDeviceToDevice, h->stream));
    rc = run_steps(h, std::min(ckpt, nsteps - n));
    if (rc != CAVITY_OK) return rc;
  }
  CK(cudaMemcpyAsync(A.final_mem, h->hb[0].base[h->parity], set_bytes, cudaMemcpyDeviceToDevice, h->stream));
  CK(cudaMemcpyAsync(&A.final_cs, h->d_cs, sizeof(CavState), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  A.final_parity = h->parity;
  A.final_steps = h->steps_taken;
  A.J = A.final_cs.nu_sum / nsteps;
  A.have_forward = true;
  if (J) *J = A.J;
  return state_status(A.final_cs);
}

int cavity_adjoint_backward(cavity_t *h, double *grad_wall, size_t n, double *grad_ra) {
  if (!h) return CAVITY_ERR_INVALID_ARG;
  AdjointStore &A = h->adj;
  if (!A.have_forward) return fail(h, CAVITY_ERR_INVALID_ARG, "adjoint: no forward run recorded");
  const cavity_desc &d = h->descs[0];
  if (grad_wall && n != (size_t)d.ny * d.nz) return fail(h, CAVITY_ERR_INVALID_ARG, "grad_wall count must be ny*nz");
  DeviceGuard g(h->dev);
  const cavity_params &p = h->prms[0];
  int rc = adj_tables(h);
  if (rc != CAVITY_OK) return rc;
  AdjArgs a{};
  a.B = h->hb[0];
  a.C = h->hcc[0];
  a.scal = A.scal;
  a.thetabar = A.thetabar;
  a.nparts = kAdjParts;
  a.gpart = A.gpart;
  a.cnt = A.cnt;
  a.kc = A.kc;
  a.tiles_x = ceil_div(d.nx, 32);
  a.tiles_y = ceil_div(d.ny, kAdjTY);
  a.coef = 1.0 / ((double)A.nsteps * d.ny * d.nz * 2.0 * a.C.h[0] * (p.t_hot - p.t_cold));
  a.dfloor = (h->u_ref_auto && p.Ra * p.Pr > 1.0) ? p.kappa * p.Pr : 0.0;
  void *X = A.X, *Q = A.Q;
  const size_t abytes = h->esize * 5 * (size_t)a.B.fstride;
  CK(cudaMemsetAsync(X, 0, abytes, h->stream));
  CK(cudaMemsetAsync(Q, 0, abytes, h->stream));
  CK(cudaMemsetAsync(A.scal, 0, sizeof(double) * kScCount, h->stream));
  a.Q = X;
  if (h->f32) k_adj_start<float><<<ceil_div((long long)d.ny * d.nz, 256), 256, 0, h->stream>>>(a);
  else k_adj_start<double><<<ceil_div((long long)d.ny * d.nz, 256), 256, 0, h->stream>>>(a);
  CK(cudaGetLastError());
  const int ck = A.run_ckpt, nseg = (A.nsteps + ck - 1) / ck;
  while (h->adj_ev.size() < 2 * (size_t)nseg) {
    cudaEvent_t e = nullptr;
    CK(cudaEventCreate(&e));
    h->adj_ev.push_back(e);
  }
  auto slot = [&](int s) { return (void *)(A.seg_mem + (size_t)s * A.set_bytes); };
  auto sweep = [&]() -> int {
    for (int c = nseg - 1; c >= 0; --c) {
      const int s0 = c * ck, len = std::min(ck, A.nsteps - s0);
      // recompute the segment from its checkpoint (copied to slot 0), each step
      // reading slot s and writing slot s + 1
      CK(cudaMemcpyAsync(slot(0), A.ckpt_mem + (size_t)c * A.set_bytes, A.set_bytes, cudaMemcpyDeviceToDevice,
                         h->stream));
      CK(cudaMemcpyAsync(h->d_cs, A.ckpt_cs + c, sizeof(CavState), cudaMemcpyDeviceToDevice, h->stream));
      CK(cudaMemcpyAsync(A.dts, &h->d_cs->dt, sizeof(double), cudaMemcpyDeviceToDevice, h->stream));
      for (int s = 0; s + 1 < len; ++s) {
        CK(launch_recompute(h, s, s > 0 && !h->d_log));
        if (h->d_log) {  // its record is written again: a finalise after every step
          CK(launch_finalize(h, 0, 1, true, A.seg_blocks + s + 1));
          CK(cudaMemcpyAsync(A.dts + s + 1, &h->d_cs->dt, sizeof(double), cudaMemcpyDeviceToDevice, h->stream));
        } else if (!self_chained(h) || s + 2 == len) {
          CK(launch_recompute_between(h, s + 1));
        }
      }
      // the walls (formed by the step where it reads them) of every stored state
      BcArgs ba = bc_args(h, 0, 3);
      ba.blocks = A.seg_blocks;
      ba.faces = A.seg_faces;
      ba.nfaces = (int)h->hwall.size() * len;
      if (h->f32) k_bc<float><<<h->n_bc * len, kBcThreads, 0, h->stream>>>(ba);
      else k_bc<double><<<h->n_bc * len, kBcThreads, 0, h->stream>>>(ba);
      CK(cudaGetLastError());
      constexpr int kGridY = 65535;  // a longer segment's states take more than one launch
      for (int s = 0; s < len; s += kGridY) {
        const dim3 parts(kAdjParts, std::min(kGridY, len - s));
        double *out = A.argpart + 2 * (size_t)kAdjParts * s;
        if (h->f32) k_adj_argmax_seg<float><<<parts, 256, 0, h->stream>>>(A.seg_blocks + s, h->hcc[0], out);
        else k_adj_argmax_seg<double><<<parts, 256, 0, h->stream>>>(A.seg_blocks + s, h->hcc[0], out);
        CK(cudaGetLastError());
      }
      // reverse sweep over the segment
      CK(cudaEventRecord(h->adj_ev[2 * c], h->stream));
      for (int s = len - 1; s >= 0; --s) {
        a.B.base[0] = slot(s);
        a.dt = A.dts + s;
        a.argpart = A.argpart + 2 * (size_t)kAdjParts * s;
        a.objective = s0 + s > 0;
        a.X = X;
        a.Q = Q;
        const bool pdl = s < len - 1;
        if (h->f32)
          CK(launch_chained(h, pdl, k_adj_sweep<float, kAdjTY>, A.ctas, dim3(32 * kAdjTY), adj_smem_bytes<float, kAdjTY>(), a));
        else
          CK(launch_chained(h, pdl, k_adj_sweep<double, kAdjTY>, A.ctas, dim3(32 * kAdjTY), adj_smem_bytes<double, kAdjTY>(), a));
        std::swap(X, Q);
      }
      CK(cudaEventRecord(h->adj_ev[2 * c + 1], h->stream));
    }
    return CAVITY_OK;
  };
  rc = sweep();
  // the state after the forward run, also where the sweep failed on the way
  CK(cudaMemcpyAsync(h->hb[0].base[A.final_parity], A.final_mem, A.set_bytes, cudaMemcpyDeviceToDevice, h->stream));
  CK(cudaMemcpyAsync(h->d_cs, &A.final_cs, sizeof(CavState), cudaMemcpyHostToDevice, h->stream));
  h->parity = A.final_parity;
  h->steps_taken = A.final_steps;
  double ra = 0.0;
  CK(cudaMemcpyAsync(&ra, A.scal + kScRa, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  if (grad_wall)
    CK(cudaMemcpyAsync(grad_wall, A.thetabar, sizeof(double) * n, cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  // (set since: its walls and its dt by what holds now, as after the setter)
  if (A.setup != h->setup) {
    const int r2 = refresh_state(h);
    if (rc == CAVITY_OK) rc = r2;
  }
  if (rc != CAVITY_OK) return rc;
  if (grad_ra) *grad_ra = ra;
  double tot = 0.0;
  for (int c = 0; c < nseg; ++c) {
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, h->adj_ev[2 * c], h->adj_ev[2 * c + 1]));
    tot += ms;
  }
  h->adj_rates_ms = tot / A.nsteps;
  return CAVITY_OK;
}

int cavity_adjoint_kernel_ms(cavity_t *h, double *ms) {
  if (!h || !ms) return CAVITY_ERR_INVALID_ARG;
  if (h->adj_rates_ms <= 0.0) return fail(h, CAVITY_ERR_INVALID_ARG, "adjoint: no reverse sweep timed yet");
  *ms = h->adj_rates_ms;
  return CAVITY_OK;
}

int cavity_set_overlap(cavity_t *h, int on) {
  if (!h) return CAVITY_ERR_INVALID_ARG;
  if (on && (h->f32 || h->ncav != 1))
    return fail(h, CAVITY_ERR_UNSUPPORTED, "overlap: FP64 single-cavity handles only");
  DeviceGuard g(h->dev);
  CK(cudaStreamSynchronize(h->stream));
  h->overlap = on && h->n_cut > 0;  // nothing to overlap without cut faces
  if (h->overlap && h->hshell.empty()) {
    int cta = 0;
    for (int id = 0; id < h->nblocks; ++id) {
      const BlockDev &B = h->hb[id];
      const int n[3] = {B.nx, B.ny, B.nz};
      for (int f = 0; f < 6; ++f) {
        if (B.wall[f]) continue;
        const int a = f / 2;
        const int n1 = n[a == 0 ? 1 : 0], n2 = n[a == 2 ? 1 : 2];
        h->hshell.push_back(ShellFace{id, f, n1, n2, cta});
        cta += ceil_div(2LL * n1 * n2, kShellThreads);
      }
    }
    h->n_shell = cta;
    CK(cudaMalloc(&h->d_shell, sizeof(ShellFace) * h->hshell.size()));
    CK(cudaMemcpy(h->d_shell, h->hshell.data(), sizeof(ShellFace) * h->hshell.size(), cudaMemcpyHostToDevice));
    CK(ensure_side(h));
  }
  if (h->overlap) launch_walls(h, h->parity);  // this schedule's shell kernel reads the stored walls
  const int rc = ensure_partials(h);
  drop_graphs(h);
  return rc;
}

int cavity_set_time_stepping(cavity_t *h, int mode) {
  if (!h || (mode != CAVITY_DT_GLOBAL && mode != CAVITY_DT_LOCAL)) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(h->dev);
  CK(cudaStreamSynchronize(h->stream));
  h->local_dt = mode == CAVITY_DT_LOCAL;
  drop_graphs(h);  // the kernels' arguments are part of the captured graphs
  return CAVITY_OK;
}

int cavity_time_kernels(cavity_t *h, int nsteps, double ms[4]) {
  if (!h || !ms || nsteps < 1) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(h->dev);
  cudaEvent_t ev[5];
  for (auto &e : ev) CK(cudaEventCreate(&e));
  double acc[4] = {0, 0, 0, 0};
  int rc = CAVITY_OK;
  for (int s = 0; s < nsteps && rc == CAVITY_OK; ++s) {
    const int par = h->parity;
    cudaEventRecord(ev[0], h->stream);
    cudaError_t e = launch_step_kernel(h, par, 0);
    cudaEventRecord(ev[1], h->stream);
    if (e == cudaSuccess) e = launch_finalize(h, par ^ 1, 1, false);
    cudaEventRecord(ev[2], h->stream);
    cudaEventRecord(ev[3], h->stream);
    cudaEventRecord(ev[4], h->stream);
    const cudaError_t es = cudaEventSynchronize(ev[4]);
    if (e == cudaSuccess) e = es;
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) { rc = fail(h, CAVITY_ERR_CUDA, cudaGetErrorString(e)); break; }
    for (int q = 0; q < 4; ++q) {
      float t = 0.f;
      cudaEventElapsedTime(&t, ev[q], ev[q + 1]);
      acc[q] += t;
    }
    h->parity ^= 1;
    h->steps_taken += 1;
  }
  for (auto &e : ev) cudaEventDestroy(e);
  for (int q = 0; q < 4; ++q) ms[q] = acc[q] / nsteps;
  ms[2] = ms[3] = 0.0;
  return rc;
}

int cavity_check_div3(const double *x, long long n, long long *n_diff) {
  if (!x || !n_diff || n < 1 || n > (1ll << 26)) return CAVITY_ERR_INVALID_ARG;
  for (long long i = 0; i < n; ++i)
    if (!(std::fabs(x[i]) >= 4.0 * DBL_MIN && std::fabs(x[i]) <= DBL_MAX)) return CAVITY_ERR_INVALID_ARG;
  double *d = nullptr;
  const size_t bytes = (size_t)n * sizeof(double);
  cudaError_t e = cudaMalloc(&d, bytes + (size_t)n);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? CAVITY_ERR_OOM : CAVITY_ERR_CUDA;
  std::vector<unsigned char> diff((size_t)n);
  e = cudaMemcpy(d, x, bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_check_div3<<<(unsigned)((n + 255) / 256), 256>>>(d, n, (unsigned char *)(d + n));
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(diff.data(), d + n, (size_t)n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (e != cudaSuccess) return CAVITY_ERR_CUDA;
  long long nd = 0;
  for (unsigned char c : diff) nd += c != 0;
  *n_diff = nd;
  return CAVITY_OK;
}

int cavity_check_sqrt(const double *x, long long n, double *max_rel, long long *n_diff) {
  if (!x || !max_rel || !n_diff || n < 1 || n > (1ll << 26)) return CAVITY_ERR_INVALID_ARG;
  for (long long i = 0; i < n; ++i)
    if (!(x[i] >= DBL_MIN && x[i] <= DBL_MAX)) return CAVITY_ERR_INVALID_ARG;
  double *d = nullptr;
  const size_t bytes = (size_t)n * sizeof(double);
  cudaError_t e = cudaMalloc(&d, 2 * bytes);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? CAVITY_ERR_OOM : CAVITY_ERR_CUDA;
  std::vector<double> rel((size_t)n);
  e = cudaMemcpy(d, x, bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_check_sqrt<<<(unsigned)((n + 255) / 256), 256>>>(d, n, d + n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(rel.data(), d + n, bytes, cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (e != cudaSuccess) return CAVITY_ERR_CUDA;
  double m = 0.0;
  long long nd = 0;
  for (double r : rel) {
    m = std::max(m, r);
    nd += r != 0.0;
  }
  *max_rel = m;
  *n_diff = nd;
  return CAVITY_OK;
}

int cavity_test_wait_timeout(cavity_t *h, long long wait_cycles, int withhold_plane) {
  if (!h) return CAVITY_ERR_INVALID_ARG;
  if (!h->f32) return fail(h, CAVITY_ERR_UNSUPPORTED, "bounded waits exist in the FP32-mixed step only");
  if (wait_cycles < 1000 || wait_cycles > kWaitCycles || withhold_plane < -1)
    return fail(h, CAVITY_ERR_INVALID_ARG, "wait limit outside [1000, 4e9] cycles or plane < -1");
  DeviceGuard g(h->dev);
  CK(cudaStreamSynchronize(h->stream));
  h->wait_cycles = wait_cycles;
  h->withhold_plane = withhold_plane;
  drop_graphs(h);
  return CAVITY_OK;
}

int cavity_measure_fp64_peak(int device, double *tflops) {
  if (!tflops) return CAVITY_ERR_INVALID_ARG;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(device);
  cavity *h = nullptr;  // no handle: CK reports the code only
  int sms = 0, per_sm = 0;
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_dfma_peak, kDfmaThreads, 0));
  const int grid = sms * std::max(per_sm, 1);
  const int iters = 4096;
  double *sink = nullptr;
  cudaStream_t st = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  int rc = CAVITY_OK;
  float best = 0.f;
  if (cudaMalloc(&sink, sizeof(double) * grid) != cudaSuccess) return CAVITY_ERR_OOM;
  if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    rc = CAVITY_ERR_CUDA;
  } else {
    const double a = 1.0 - 1.0 / 1048576.0, b = 1.0 / 1048576.0;
    k_dfma_peak<<<grid, kDfmaThreads, 0, st>>>(sink, iters / 8, a, b);  // warm-up
    for (int rep = 0; rep < 3 && rc == CAVITY_OK; ++rep) {
      cudaEventRecord(e0, st);
      k_dfma_peak<<<grid, kDfmaThreads, 0, st>>>(sink, iters, a, b);
      cudaEventRecord(e1, st);
      float ms = 0.f;
      if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
        rc = CAVITY_ERR_CUDA;
        break;
      }
      if (best == 0.f || ms < best) best = ms;
    }
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (st) cudaStreamDestroy(st);
  cudaFree(sink);
  if (rc != CAVITY_OK) return rc;
  const double flops = 2.0 * kDfmaChains * kDfmaUnroll * (double)iters * grid * kDfmaThreads;
  *tflops = flops / (best * 1e-3) / 1e12;
  return CAVITY_OK;
}

int cavity_sync(cavity_t *h) {
  if (!h) return CAVITY_ERR_INVALID_ARG;
  DeviceGuard g(h->dev);
  return all_status(h);
}

int cavity_destroy(cavity_t *h) {
  if (!h) return CAVITY_OK;
  release(h);
  delete h;
  return CAVITY_OK;
}

const char *cavity_strerror(int code) {
  switch (code) {
    case CAVITY_OK: return "ok";
    case CAVITY_ERR_INVALID_ARG: return "invalid argument";
    case CAVITY_ERR_OOM: return "out of memory";
    case CAVITY_ERR_CUDA: return "CUDA runtime error";
    case CAVITY_ERR_NONFINITE: return "non-finite residual or spectral radius";
    case CAVITY_ERR_TIMEOUT: return "device-side wait timed out";
    case CAVITY_ERR_UNSUPPORTED: return "unsupported request";
    default: return "unknown status";
  }
}

const char *cavity_last_error(cavity_t *h) { return h ? h->err.c_str() : ""; }

}  // extern "C"
