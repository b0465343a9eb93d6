// Device-side data structures and kernels of the buoyancy-driven-cavity step
// (Xue & Roy, arXiv 2006.02602).  Shared by the C-ABI translation unit only.
//
// Per step, on the handle's stream (sequences of 1, 2, 4 and 16 steps per
// buffer parity, launched or as CUDA graphs, each kernel a programmatic dependent
// of the one before):
//   k_step      fused residual (Eqs. 1-3) + explicit Euler update of every
//               interior node of every block, walls (Section 2) formed where
//               they are read; FP64 residual sums as per-CTA partials, the
//               spectral-radius maximum of the new state as an atomic maximum;
//   k_between   what the next step waits for (undivided small FP64 cavities
//               see to it in the step itself): dt from that maximum, the centre
//               shift, and with cut faces the ghost layers of the new state
//               from the neighbours' layers (Section 4.5, Listings 1-2, V3: p
//               at depth 2, u, v, w, T at depth 1);
//   k_finalize  once a sequence, for all of its steps (the last one's exchange and
//               stored walls in the same launch): the partials reduced in a
//               fixed order: residual norms, Nusselt numbers, time, non-finite
//               flag, the step log's last two records;
//   k_step_record  with a step log, beside the steps after it: a step's record.
// On a state refresh: k_bc (walls stored), k_pack / k_unpack.
//
// Storage: each block holds two buffer sets (ping-pong); a set is NF
// consecutive padded arrays, x fastest.  Local node (i, j, k), i in
// [-1, n+2], sits at element (XO1 - 1 + i) + pitch (j + 1) + plane (k + 1)
// so that node 1 of every row starts on a 32-byte boundary.
#pragma once

#include <cfloat>
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

namespace bdc {

constexpr int kNF = 5;           // p, u, v, w, T
constexpr int kMaxCentre = 8;    // 2^3 centre nodes at most
constexpr int kPartStride = 8;   // doubles per step partial: 5 sums, sr max, pad
constexpr int kBcThreads = 128;  // wall positions per k_bc CTA (one per thread)
constexpr int kFinSlices = 16;   // k_finalize CTAs per cavity at most

struct BlockDev {
  int nx, ny, nz;        // interior nodes of the block
  int ox, oy, oz;        // global node index = o + local index
  int pitch;             // elements per row
  int rows;              // ny + 4
  long long plane;       // pitch * rows
  long long fstride;     // elements per field array
  int wall[6];           // face on a cavity wall (-x, +x, -y, +y, -z, +z)
  int nbr[6];            // neighbour block across a cut face, -1 on walls
  int cav;               // cavity this block belongs to
  int tiles_x, tiles_y, tiles_z;
  int tile_begin;        // first partial slot (k_step tile) of this block
  // z chunking of the step kernels: chunks 0 .. tiles_zc-1 of kc planes cover
  // planes 1 .. zsplit, the other tiles_z - tiles_zc chunks split planes
  // zsplit+1 .. nz into chunks of kf planes.  Scheduling index c runs over
  // every block's coarse tiles first (coarse_begin + local) and the fine ones
  // last (ncoarse + fine_begin + local): the persistent FP64 grid's counter
  // and the FP32 grids' block order both end on short tiles.  Partial slots
  // stay block-major (tile_begin + local tile index), so a cavity's are
  // contiguous.
  int tiles_zc, zsplit, coarse_begin, fine_begin;
  int kc, kf;
  void *base[2];         // buffer sets (field f at base + f * fstride)
};
constexpr int kFineKC32 = 8;  // the largest kf of the FP32 form

struct CavConst {
  double h[3], ih[3], ih2[3], ihh[3];
  double nu, alpha, gs, t_inf, b2min, c4, cfl, diffsr, inv_dT;
  double inv_nint, inv_nwall;
  // folded coefficients of the FP64 rates: c4 / (2 h_d) (the dissipation
  // weight of |V_d| + sqrt(V_d^2 + 4 beta^2)), nu / h_d^2, alpha / h_d^2,
  // 2 nu sum 1/h_d^2, 2 alpha sum 1/h_d^2, gs T_inf
  double dsc[3], nuhh[3], alhh[3], nu2s, al2s, gst;
  // FP32 copies (rounded to nearest, as a device conversion would) of the
  // constants the FP32 kernels and estimates use, so that no kernel spends
  // FP64-pipe conversions on them: 1/h, 1/(2h), nu/h^2, alpha/h^2, c4/2, gs,
  // T_inf, beta_min^2, the diffusive spectral term, cfl, c4
  float fih[3], fh2[3], fnh[3], fah[3];
  float fc4h, fgs, ftinf, fb2min, fdiffsr, fcfl;
  float fc4;
  // the spectral bound at rest, S0 = beta_min (1/h_x + 1/h_y + 1/h_z) + the
  // diffusive term (FP64), and 2 beta_min (FP32): the FP64 step's dt filter
  // works on S - S0
  double s0;
  float f2b0;
  int gaxis;
  int gn[3];
  int ncentre;
  int centre_blk[kMaxCentre];
  long long centre_off[kMaxCentre];  // element offset of the node in its field array
  int tile_begin, tile_end;          // k_step CTAs of this cavity
  int slice_q[kFinSlices + 1];       // k_finalize slice g reduces the step partials slice_q[g] .. slice_q[g+1]-1
  double wscale[2];                  // FP32 step's sums of 3 T_w - 4 T_1 + T_2 -> hot, cold wall fluxes: +-h_x^-1 / (2 dT)
  int bc_begin, bc_end;              // k_bc CTAs of this cavity (all wall faces)
  int bc_xend;                       // the x walls' CTAs (the Nusselt partials) come first: bc_begin .. bc_xend-1
  int nu_begin, nu_end;              // CTAs of this cavity in the list of its x walls alone
  long long wall_off;                // offset of this cavity's wall temperatures
};

// The grid- and parameter-derived members of CavConst (everything but the
// cavity's tile/wall ranges and centre nodes), from the interior node counts
// and resolved parameters.  One definition for every entry point.
inline void set_cav_physics(CavConst &C, const int gn[3], const cavity_params &p) {
  double sih = 0.0;
  for (int d = 0; d < 3; ++d) {
    const double np1 = (double)gn[d] + 1.0;
    C.gn[d] = gn[d];
    C.h[d] = 1.0 / np1;
    C.ih[d] = np1;
    C.ih2[d] = 0.5 * np1;
    C.ihh[d] = np1 * np1;
    sih += C.ihh[d];
  }
  C.nu = p.Pr;
  C.alpha = 1.0;
  C.gs = p.Ra * p.Pr;
  C.t_inf = p.t_inf;
  C.b2min = p.kappa * p.u_ref * p.u_ref;
  C.c4 = p.c4;
  C.cfl = p.cfl;
  C.diffsr = 2.0 * (C.nu > C.alpha ? C.nu : C.alpha) * sih;
  C.inv_dT = 1.0 / (p.t_hot - p.t_cold);
  C.inv_nint = 1.0 / ((double)gn[0] * gn[1] * gn[2]);
  C.inv_nwall = 1.0 / ((double)gn[1] * gn[2]);
  C.wscale[0] = 0.5 * C.ih[0] * C.inv_dT;
  C.wscale[1] = -0.5 * C.ih[0] * C.inv_dT;
  for (int d = 0; d < 3; ++d) {
    C.dsc[d] = 0.5 * C.c4 * C.ih[d];
    C.nuhh[d] = C.nu * C.ihh[d];
    C.alhh[d] = C.alpha * C.ihh[d];
  }
  C.nu2s = 2.0 * C.nu * sih;
  C.al2s = 2.0 * C.alpha * sih;
  C.gst = C.gs * C.t_inf;
  for (int d = 0; d < 3; ++d) {
    C.fih[d] = (float)C.ih[d];
    C.fh2[d] = (float)C.ih2[d];
    C.fnh[d] = (float)(C.nu * C.ihh[d]);
    C.fah[d] = (float)(C.alpha * C.ihh[d]);
  }
  C.fc4 = (float)C.c4;
  {
    const double b0 = std::sqrt(C.b2min);
    C.s0 = b0 * (C.ih[0] + C.ih[1] + C.ih[2]) + C.diffsr;
    C.f2b0 = (float)(2.0 * b0);
  }
  C.fc4h = (float)(0.5 * C.c4);
  C.fgs = (float)C.gs;
  C.ftinf = (float)C.t_inf;
  C.fb2min = (float)C.b2min;
  C.fdiffsr = (float)C.diffsr;
  C.fcfl = (float)C.cfl;
  C.gaxis = p.gravity_axis;
}

// Steps of an undivided FP64 cavity follow one another without a kernel between
// them: step s takes dt from the maximum step s - 1 left in its slot, writes its
// own, and clears the one after, which step s - 2 wrote and step s - 1 read.
// Other steps use slot 0.
constexpr int kStepSlots = 3;

struct CavState {
  double dt;         // dt of the next step
  double c;          // pending centre-pressure shift of the stored p (after dt: step_tile_f64 reads the pair)
  double t;          // simulated time
  long long step;    // steps taken
  double res[5];     // RMS dq/dt of the last step
  double nu_hot, nu_cold;
  int flags;         // bit 0: non-finite residual or spectral radius
  int pad;
  // for the step in flight (zero before it), in the step's slot (kStepSlots):
  // the largest spectral bound of its new state, and the FP64 step's largest
  // published dt-filter floor (float_key ^ 0x80000000, 0 = none)
  double smax[kStepSlots];
  unsigned int sfl[kStepSlots], pad2;
  double dt0;        // dt as the last finalise left it (dt itself moves on within a graph)
  double nu_sum;     // sum of nu_hot over the steps (the adjoint's forward run zeroes it)
  // the step log's running values between two finalises (k_step_record's own)
  double log_t, log_dt;
  long long log_bad;
};

struct StepRecord {   // one step's record in the host-memory step log (the C ABI's cavity_step_record)
  long long step;
  double t, dt;
  double res[5];
  double nu_hot, nu_cold;
  long long flags;
};

struct WallFace {     // one wall face of one block, processed by k_bc
  int block, face;
  int n1, n2;         // face interior extents (faster, slower face axis)
  int cta_begin;      // first k_bc CTA
  int cav;
};

struct ShellFace {    // the two layers next to one cut face, processed by k_shell_f64
  int block, face;
  int n1, n2;         // face interior extents (faster, slower face axis)
  int cta_begin;
};

struct CutFace {      // one cut face of one block, processed by k_pack / k_unpack
  int src, face, dst;
  int nb, nc;         // face extents (faster, slower face axis)
  int cta_begin;
  long long buf_off;  // element offset into the exchange buffer
};

// ---------------------------------------------------------------------------
// storage traits

template <class S> struct XO;
template <> struct XO<double> { static constexpr int v = 4; };
template <> struct XO<float> { static constexpr int v = 8; };  // node 1 starts a 32-byte sector

template <class S>
__device__ __forceinline__ long long node_index(const BlockDev &B, int i, int j, int k) {
  return (long long)(XO<S>::v - 1 + i) + (long long)B.pitch * (j + 1) + B.plane * (k + 1);
}

// Arrays of one buffer set.  FP64 form: p, u, v, w, T.  FP32-mixed form:
// p_hi, p_lo, u, v, w, T_hi, T_lo (p = p_hi + p_lo and T = T_hi + T_lo,
// unevaluated FP32 pairs: their time-step accumulation is compensated).
// NP = arrays of p; the transported fields u, v, w, T start at array NP.
template <class S> struct Store;
template <> struct Store<double> { static constexpr int NA = 5, NP = 1; };
template <> struct Store<float> { static constexpr int NA = 7, NP = 2; };

template <class S>
__device__ __forceinline__ double load_p(const S *base, long long fs, long long o);
template <>
__device__ __forceinline__ double load_p<double>(const double *base, long long, long long o) { return base[o]; }
template <>
__device__ __forceinline__ double load_p<float>(const float *base, long long fs, long long o) {
  return (double)base[o] + (double)base[fs + o];
}
template <class S>
__device__ __forceinline__ void store_p(S *base, long long fs, long long o, double v);
template <>
__device__ __forceinline__ void store_p<double>(double *base, long long, long long o, double v) { base[o] = v; }
template <>
__device__ __forceinline__ void store_p<float>(float *base, long long fs, long long o, double v) {
  const float hi = (float)v;
  base[o] = hi;
  base[fs + o] = (float)(v - (double)hi);
}

// temperature: array NP + 3 (FP64), or the pair NP + 3 (hi), NP + 4 (lo) (FP32-mixed)
template <class S>
__device__ __forceinline__ double load_T(const S *base, long long fs, long long o) {
  return load_p<S>(base + (Store<S>::NP + 3) * fs, fs, o);
}
template <class S>
__device__ __forceinline__ void store_T(S *base, long long fs, long long o, double v) {
  store_p<S>(base + (Store<S>::NP + 3) * fs, fs, o, v);
}

// ---------------------------------------------------------------------------
// deterministic block reductions (fixed shuffle tree, fixed warp order)

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// ---------------------------------------------------------------------------
// Square root of a positive, normal, finite FP64 value without the FP64 pipe.
// GB300 issues an FP64 warp instruction every 16 cycles an SM (two lanes a
// clock), FP32 and integer ones up to four a cycle.  With q = 4^k m, m in [1, 4):
//   y ~ 1/sqrt(m) (rsqrt.approx.ftz.f32), s_0 = sh + sl by one Newton step on
//   the FP32 pair of m's leading 46 bits: relative error below 2^-43;
//   r = m - s_0^2, exact, as a 64-bit integer (s_0 has 46 fraction bits);
//   s = s_0 + r y / 2, the correction (below 2^9 units in the last place)
//   formed in FP32 and added to s_0's significand as an integer.
// The result is within one unit in the last place of the correctly rounded
// root (cavity_check_sqrt measures this against CUDA's sqrt; the clamps keep
// s_0 in [1, 2], where a unit of its last place is 2^-52; one root in 1300 is
// not the correctly rounded one, with r from an FP64 fused multiply-add one in
// 90).  Arguments that are NaN or infinite give a finite value:
// the rates reach NaN or infinity through beta^2 and the weights.
__device__ __forceinline__ double sqrt_newton(double q) {
  const int hi = __double2hiint(q);
  const unsigned lo = (unsigned)__double2loint(q);
  const int odd = ~(hi >> 20) & 1;  // the unbiased exponent is odd
  const int mhi = (hi & 0xfffff) | ((1023 + odd) << 20);
  const float qh = __int_as_float((int)(__funnelshift_l(lo, (unsigned)hi, 3) & 0x7fffffu) | ((127 + odd) << 23));
  // the significand's next 23 bits, as an integer in FP32
  const float ql = __fsub_rn(__uint_as_float(0x4b000000u | ((lo & 0x1fffffffu) >> 6)), 8388608.f);
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(qh));
  const float hy = 0.5f * y;
  const float sh = fminf(fmaxf(__fmul_rn(qh, y), 1.f), 1.99999988f);
  const float res = __fmaf_rn(ql, __int_as_float((127 - 46 + odd) << 23), __fmaf_rn(-sh, sh, qh));
  const int n = __float2int_rn(__fmul_rn(__fmul_rn(res, hy), 0x1p46f));
  long long s0 = ((long long)__float_as_int(sh) << 29) + (896ll << 52) + ((long long)n << 6);
  s0 = max(min(s0, 0x4000000000000000ll), 0x3ff0000000000000ll);
  // m - s0^2, below 2^-39, in units of 2^-92 (s0 is a multiple of 2^-46), modulo 2^64
  const unsigned long long t = (unsigned long long)(s0 - (1022ll << 52)) >> 6;
  const long long r = (long long)(((1ull << 52 | (unsigned long long)(mhi & 0xfffff) << 32 | lo) << (40 + odd)) - t * t);
  const float rf = __fsub_rn(__int_as_float(0x4b400000 + (int)(r >> 32)), 12582912.f);
  const int n2 = __float2int_rn(__fmul_rn(rf, __fmul_rn(hy, 0x1p-8f)));
  return __longlong_as_double(s0 + n2 + ((long long)((hi - mhi) >> 1) << 32));
}

// 4 x for a positive normal x (the exponent raised by two; infinite or NaN
// past FP64's range), and the larger of two non-negative values (their bit
// patterns order like the values, a NaN above all): integer operations
// instead of FP64-pipe slots.
__device__ __forceinline__ double times4(double x) {
  return __hiloint2double(min(__double2hiint(x) + (2 << 20), 0x7ff00000), __double2loint(x));
}
__device__ __forceinline__ double max_nonneg(double a, double b) {
  return __double_as_longlong(a) > __double_as_longlong(b) ? a : b;
}

// ---------------------------------------------------------------------------
// Per-node rates, Eqs. 1-3, FP64.  Star values: c, x-, x+, y-, y+, z-, z+.
// Rearranged for few FP64 operations (GB300's FP64 pipe is the bound):
//  - beta^2 eps_d / h_d^4 = c4 lambda_d / h_d, so the continuity rate needs no
//    division, and c4 lambda_d / h_d = (|V_d| + sqrt(V_d^2 + 4 beta^2)) c4/(2 h_d);
//  - the central advection and the diffusion of one transported field share
//    the neighbour weights: -a_d (q_+ - q_-) + k (q_+ + q_- - 2 q_c) / h_d^2
//    = (k/h_d^2 - a_d) q_+ + (k/h_d^2 + a_d) q_- - 2 k q_c / h_d^2, with
//    a_d = V_d / (2 h_d); u, v, w share one set of weights (k = nu), T has its
//    own (k = alpha): seven FMAs per field instead of sixteen operations;
//  - the dissipation, the advection weights, the square roots and the whole of
//    T's transport in 64-bit integers: 41 FP64 operations a node are left here and
//    11 in the update and the residual sums; the kernel executes 58 (95 before) of
//    its 1911 instructions a node on the FP64 pipe, the others in issue slots that
//    it leaves empty (ncu, 128^3 in 2x2x2 blocks).
//    256^3 2445 -> 1825 us a step, 128^3 in 2x2x2 blocks 341 -> 260, 64^3 58 -> 45.6.
//    About here the two pipes balance: u, v and w in integers too make it slower
//    (256^3 2256, spills), and so does an FP64 div V or T the other way (1870,
//    1908 with T's weights alone in FP64).

struct NodeF64 {
  double p[13];  // c, x-, x+, y-, y+, z-, z+, x-2, x+2, y-2, y+2, z-2, z+2
  double u[7], v[7], w[7], T[7];
};

// FP64 values in 64-bit fixed point.  to_fixed<K> takes a value to units of
// 2^-(52+K) of 2^(E - 1023), E the largest exponent field of the values to be
// summed; from_fixed<K> rounds a sum in those units to the nearest FP64 value.
// The sum itself is exact: its error is a unit a term and one rounding, where
// FP64 operations round each by 2^-53.  About 12 and 18 integer instructions.
// A term 2^64 below the largest, and a result below 2^-959, count as zero; a
// term that is NaN, infinite or 2^1020 and above makes the result NaN (E = 2047;
// a velocity that is NaN or infinite reaches every rate through beta^2, div V
// and the momentum sums in FP64).
__device__ __forceinline__ unsigned fixed_exp(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
// v >> n, zero from n = 64 on
__device__ __forceinline__ unsigned long long shr(unsigned long long v, unsigned n) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
template <int K> __device__ __forceinline__ long long to_fixed(double v, int E) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned sh = (unsigned)E - ((hi >> 20) & 0x7ffu);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = ((unsigned long long)__funnelshift_l(lo, mh, K) << 32) | (lo << K);
  const long long sg = (long long)((int)hi >> 31);
  return ((long long)shr(m, sh) ^ sg) - sg;
}
template <int K> __device__ __forceinline__ double from_fixed(long long S, int E) {
  const long long sg = S >> 63;
  const unsigned long long A = (unsigned long long)((S ^ sg) - sg);
  const int lz = __clzll((long long)A);
  const unsigned long long N = (A << ((lz - 1) & 63)) + 512;  // |S| < 2^63: the leading bit at 62, rounded at 10
  const unsigned long long r = ((unsigned long long)(unsigned)(E + 10 - K - lz) << 52) + (N >> 10);
  const unsigned long long bad = E >= 2043 ? 0x7ff8ull << 48 : 0;
  const unsigned long long v = A == 0 || E < 64 ? 0 : r | ((unsigned long long)sg & (1ull << 63));
  return __longlong_as_double((long long)(v | bad));
}

// The dissipation sum_d e_d (p_++ - 4 p_+ + 6 p_0 - 4 p_- + p_--)_d with
// e_d = (|V_d| + sqrt(V_d^2 + 4 beta^2)) c4 / (2 h_d).  The weights e_d below 2^62
// in units of 2^(e - 2105), the fourth differences below 2^63 (the star's
// coefficients add up to 16) in units of 2^(E - 1081).
struct Weight3 {
  long long m[3];
  int e;
};
__device__ __forceinline__ void dissipation_weights(const CavConst &C, double b2, const double V[3], Weight3 &x) {
  const double f4 = times4(b2);
  int e[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double s = sqrt_newton(fma(V[d], V[d], f4)), a = fabs(V[d]);
    const int E = (int)(max(fixed_exp(s), fixed_exp(a)) >> 20);
    const unsigned long long b = (unsigned long long)__double_as_longlong(C.dsc[d]) << 11 | 1ull << 63;
    x.m[d] = (long long)__umul64hi((unsigned long long)(to_fixed<8>(a, E) + to_fixed<8>(s, E)), b);
    e[d] = E + (__double2hiint(C.dsc[d]) >> 20);
  }
  x.e = max(max(e[0], e[1]), e[2]);
#pragma unroll
  for (int d = 0; d < 3; ++d) x.m[d] = (long long)shr((unsigned long long)x.m[d], (unsigned)(x.e - e[d]));
}
__device__ __forceinline__ double dissipation(const double p[13], const Weight3 &x) {
  unsigned e = 0;
#pragma unroll
  for (int q = 0; q < 13; ++q) e = max(e, fixed_exp(p[q]));
  const int E = (int)(e >> 20);
  const long long c6 = 6 * to_fixed<6>(p[0], E);
  long long D[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    D[d] = (to_fixed<6>(p[7 + 2 * d], E) + to_fixed<6>(p[8 + 2 * d], E)) -
           4 * (to_fixed<6>(p[1 + 2 * d], E) + to_fixed<6>(p[2 + 2 * d], E)) + c6;
  }
  // the differences shifted up together, so that the products keep their bits
  const int sh = __clzll((D[0] ^ (D[0] >> 63)) | (D[1] ^ (D[1] >> 63)) | (D[2] ^ (D[2] >> 63)) | 1) - 1;
  long long S = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d) S += __mul64hi(x.m[d], D[d] << sh);
  return from_fixed<9>(S, E >= 2043 ? 2047 : E + x.e - sh - 2038);
}

// a_d = V_d / (2 h_d), unrounded: the upper 64 bits of the mantissas' product, the
// exponent field it has with their product in [2, 4), and its sign.
struct Advect {
  unsigned long long m;
  int e;
  long long sg;
};
__device__ __forceinline__ Advect advect(double v, double ih2) {
  const unsigned long long one = 1ull << 63;
  const unsigned long long a = (unsigned long long)__double_as_longlong(v) << 11 | one;
  const unsigned long long b = (unsigned long long)__double_as_longlong(ih2) << 11 | one;
  return {__umul64hi(a, b), (int)(fixed_exp(v) >> 20) + (__double2hiint(ih2) >> 20) - 1022,
          (long long)(__double2hiint(v) >> 31)};
}

// The neighbour weights D + a (minus side) and D - a (plus side), D = k / h_d^2,
// rounded once each.
__device__ __forceinline__ void weights(double D, const Advect &a, double &minus, double &plus) {
  const int E = max(__double2hiint(D) >> 20, a.e);
  const long long x = to_fixed<9>(D, E);
  const long long t = (long long)shr(a.m >> 2, (unsigned)(E - a.e)), y = (t ^ a.sg) - a.sg;
  minus = from_fixed<9>(x + y, E);
  plus = from_fixed<9>(x - y, E);
}

// Advection and diffusion of one field as the sum over the six neighbours of
// weight times (q_neighbour - q_centre): the weights D +- a (below 2^61 in units of
// 2^(e - 1082)) and the differences (below 2^60 in units of 2^(E - 1081)) are exact
// but for their last unit.  Both are split into signed 32-bit halves: the sums H
// of the high products (below 2^59: a direction's two weights add up to 2^61) and
// L of the mixed ones (below 6 2^60) hold the result; the product of the low
// halves, at most a quarter of H's unit, is left out.  Against 128-bit values the
// error is 0.16 to 0.6 of the seven FMAs' (random stars, smooth and rough).
struct Weight6 {
  int h[6], l[6];
  int e;
};
__device__ __forceinline__ void split(long long v, int &h, int &l) {
  l = (int)v;
  h = (int)((v - l) >> 32);
}
__device__ __forceinline__ void transport_weights(const double D[3], const Advect a[3], Weight6 &w) {
  w.e = max(max(max(a[0].e, a[1].e), a[2].e), max(max(__double2hiint(D[0]), __double2hiint(D[1])), __double2hiint(D[2])) >> 20);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const long long x = to_fixed<7>(D[d], w.e);
    const long long t = (long long)shr(a[d].m >> 4, (unsigned)(w.e - a[d].e)), y = (t ^ a[d].sg) - a[d].sg;
    split(x + y, w.h[2 * d], w.l[2 * d]);
    split(x - y, w.h[2 * d + 1], w.l[2 * d + 1]);
  }
}
__device__ __forceinline__ double transport(const double q[7], const Weight6 &w) {
  unsigned e = 0;
#pragma unroll
  for (int i = 0; i < 7; ++i) e = max(e, fixed_exp(q[i]));
  const int E = (int)(e >> 20);
  const long long c = to_fixed<6>(q[0], E);
  long long H = 0, L = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    int dh, dl;
    split(to_fixed<6>(q[1 + i], E) - c, dh, dl);
    H += (long long)w.h[i] * dh;
    L += (long long)w.h[i] * dl;
    L += (long long)w.l[i] * dh;
  }
  // H in units of 2^(w.e + E - 2099), L of 2^-32 of that
  return from_fixed<9>((H << 4) + (L >> 28), E >= 2043 ? 2047 : w.e + E - 1019);
}

// The part of the rates that reads the velocities alone (and the centre T):
// beta^2, the dissipation weights, div V and the momentum rates without the
// pressure gradient.
struct VelF64 {
  double b2, divV, ru, rv, rw;
  Weight3 e;
  Advect a[3];
};

#define BDC_TRANSPORT(q, xm, xp, ym, yp, zm, zp, centre) \
  fma(xp, q[2], fma(xm, q[1], fma(yp, q[4], fma(ym, q[3], fma(zp, q[6], fma(zm, q[5], centre))))))

__device__ __forceinline__ void rates_vel_f64(const CavConst &C, const NodeF64 &n, VelF64 &x) {
  const double u0 = n.u[0], v0 = n.v[0], w0 = n.w[0];
  const double b2 = max_nonneg(fma(u0, u0, fma(v0, v0, w0 * w0)), C.b2min);
  x.b2 = b2;
  const double V[3] = {u0, v0, w0};
  dissipation_weights(C, b2, V, x.e);
  x.divV = fma(n.u[2] - n.u[1], C.ih2[0], fma(n.v[4] - n.v[3], C.ih2[1], (n.w[6] - n.w[5]) * C.ih2[2]));
  // neighbour weights: m = minus side, p = plus side
  x.a[0] = advect(u0, C.ih2[0]);
  x.a[1] = advect(v0, C.ih2[1]);
  x.a[2] = advect(w0, C.ih2[2]);
  double nxm, nxp, nym, nyp, nzm, nzp;
  weights(C.nuhh[0], x.a[0], nxm, nxp);
  weights(C.nuhh[1], x.a[1], nym, nyp);
  weights(C.nuhh[2], x.a[2], nzm, nzp);
  // the buoyancy force (Eq. 2) enters the gravity-axis momentum rate with its centre term
  const double buoy = fma(C.gs, n.T[0], -C.gst);
  const double bv = C.gaxis == 1 ? buoy : 0.0, bw = C.gaxis == 2 ? buoy : 0.0;
  x.ru = BDC_TRANSPORT(n.u, nxm, nxp, nym, nyp, nzm, nzp, -C.nu2s * u0);
  x.rv = BDC_TRANSPORT(n.v, nxm, nxp, nym, nyp, nzm, nzp, fma(-C.nu2s, v0, bv));
  x.rw = BDC_TRANSPORT(n.w, nxm, nxp, nym, nyp, nzm, nzp, fma(-C.nu2s, w0, bw));
}

__device__ __forceinline__ void rates_pt_f64(const CavConst &C, const NodeF64 &n, const VelF64 &x, double r[5]) {
  r[0] = fma(-x.b2, x.divV, -dissipation(n.p, x.e));
  r[1] = fma(-(n.p[2] - n.p[1]), C.ih2[0], x.ru);
  r[2] = fma(-(n.p[4] - n.p[3]), C.ih2[1], x.rv);
  r[3] = fma(-(n.p[6] - n.p[5]), C.ih2[2], x.rw);
  const double D[3] = {C.alhh[0], C.alhh[1], C.alhh[2]};
  Weight6 w;
  transport_weights(D, x.a, w);
  r[4] = transport(n.T, w);
}
#undef BDC_TRANSPORT

// spectral-radius bound of one node's state (the dt denominator); square
// roots within one unit in the last place (sqrt_newton), so dt is the
// correctly rounded formula's to a few ulp
__device__ __forceinline__ double spectral_f64(const CavConst &C, double u, double v, double w) {
  // (every product-sum an explicit FMA: the same bits in every kernel)
  const double b2 = max_nonneg(fma(u, u, fma(v, v, w * w)), C.b2min);
  const double f4 = times4(b2);
  const double sx = fabs(u) + sqrt_newton(fma(u, u, f4));
  const double sy = fabs(v) + sqrt_newton(fma(v, v, f4));
  const double sz = fabs(w) + sqrt_newton(fma(w, w, f4));
  return fma(0.5, fma(sx, C.ih[0], fma(sy, C.ih[1], sz * C.ih[2])), C.diffsr);
}

// Rates (from their velocity part x on) and explicit update of one node: the new p, u, v, w, T in q (p with
// the pending centre shift taken off), the rates in r.  One function for
// k_step_f64 and k_shell_f64, so a node gives the same bits in either.
__device__ __forceinline__ void update_node_f64(const CavConst &C, const NodeF64 &n, const VelF64 &x, double dt,
                                                double cshift, int local_dt, double q[5], double r[5]) {
  rates_pt_f64(C, n, x, r);
  const double dtn = local_dt ? C.cfl / spectral_f64(C, n.u[0], n.v[0], n.w[0]) : dt;
  q[0] = fma(dtn, r[0], n.p[0] - cshift);
  q[1] = fma(dtn, r[1], n.u[0]);
  q[2] = fma(dtn, r[2], n.v[0]);
  q[3] = fma(dtn, r[3], n.w[0]);
  q[4] = fma(dtn, r[4], n.T[0]);
}

// FP32 estimate of spectral_f64 (the same formula: relative error below
// 1e-6; beta_min^2 = kappa u_ref^2 is at least FP32's smallest normal, so the
// estimate is finite).  The FP64 adjoint's argmax skips a node whose estimate,
// raised by 1e-5, stays below a value the exact FP64 maximum already reached
// (the FP64 step filters on spectral_dev_f32 below instead).
__device__ __forceinline__ float spectral_est_f32(const CavConst &C, float uf, float vf, float wf) {
  const float b2 = fmaxf(__fmaf_rn(uf, uf, __fmaf_rn(vf, vf, __fmul_rn(wf, wf))), C.fb2min);
  const float f4 = __fmul_rn(4.f, b2);
  const float qx = __fmaf_rn(uf, uf, f4), qy = __fmaf_rn(vf, vf, f4), qz = __fmaf_rn(wf, wf, f4);
  float rx, ry, rz;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rx) : "f"(qx));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ry) : "f"(qy));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rz) : "f"(qz));
  const float sx = __fmaf_rn(qx, rx, fabsf(uf)), sy = __fmaf_rn(qy, ry, fabsf(vf)), sz = __fmaf_rn(qz, rz, fabsf(wf));
  return __fmaf_rn(0.5f, __fmaf_rn(sx, C.fih[0], __fmaf_rn(sy, C.fih[1], __fmul_rn(sz, C.fih[2]))), C.fdiffsr);
}
// |x| as FP32, rounded toward zero, from the FP64 bit pattern by integer
// operations (a conversion instruction would take slots of GB300's narrow
// FP64 pipe): the exponent rebiased from 1023 to 127, the significand cut to
// 23 bits.  Relative error below 2^-23 in FP32's normal range; exponents
// below it give a value below 2^-125, above it (and inf/NaN) a finite value
// of FP32's largest exponent.
__device__ __forceinline__ float abs_f32_trunc(double x) {
  const unsigned lo = (unsigned)__double2loint(x), hi = (unsigned)__double2hiint(x);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const unsigned m = __funnelshift_l(lo, hi, 3) & 0x7fffffu;  // significand bits 51..29
  const int ec = min(max(e, 896), 1150);
  return __uint_as_float(((unsigned)(ec - 896) << 23) | m);
}
__device__ __forceinline__ float spectral_est_f32(const CavConst &C, double u, double v, double w) {
  return spectral_est_f32(C, abs_f32_trunc(u), abs_f32_trunc(v), abs_f32_trunc(w));
}

// FP32 estimate of D = S - S0, the spectral bound less its value at rest,
// from |u|, |v|, |w| >= 0.  With beta^2 = max(|V|^2, beta_min^2),
// sqrt(V_d^2 + 4 beta^2) - 2 beta_min = (V_d^2 + 4 (beta^2 - beta_min^2)) /
// (sqrt(V_d^2 + 4 beta^2) + 2 beta_min): every term is non-negative, so D
// comes out with a relative error of a few 1e-7 however small it is next to
// S0 (an estimate of S itself has its error on the scale of S0, which near
// rest exceeds the spread of S over the nodes).
__device__ __forceinline__ float spectral_dev_f32(const CavConst &C, float uf, float vf, float wf) {
  const float vv = __fmaf_rn(uf, uf, __fmaf_rn(vf, vf, __fmul_rn(wf, wf)));
  const float f4 = __fmul_rn(4.f, fmaxf(vv, C.fb2min));
  const float d4 = __fmul_rn(4.f, fmaxf(__fsub_rn(vv, C.fb2min), 0.f));  // 4 (beta^2 - beta_min^2)
  const float V[3] = {uf, vf, wf};
  float acc = 0.f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float q = __fmaf_rn(V[d], V[d], f4);
    float r, rd;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(q));
    const float den = __fmaf_rn(q, r, C.f2b0);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rd) : "f"(den));
    const float term = __fmaf_rn(__fmaf_rn(V[d], V[d], d4), rd, V[d]);
    acc = __fmaf_rn(term, C.fih[d], acc);
  }
  return __fmul_rn(0.5f, acc);
}

// Order-preserving map of a float (either sign) to a signed int, so that a
// warp can take a float maximum with __reduce_max_sync, and its inverse.
__device__ __forceinline__ int float_key(float f) {
  const int b = __float_as_int(f);
  return b >= 0 ? b : b ^ 0x7fffffff;
}
__device__ __forceinline__ float key_float(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff); }

// ---------------------------------------------------------------------------
// k_step, FP64: a tile is NT consecutive nodes of a block's (x, y) plane, x
// fastest (node e = (i - 1) + nx (j - 1)), over a chunk of planes; one thread
// per (i, j) column sweeps the chunk in k.  The z-neighbours live in register
// queues (5 deep for p, 3 deep for u, v, w, T); x/y neighbours come through L1.
//
// Why these tiles: the FP64 pipe (two lanes a clock per SM) takes a warp
// instruction's 16 cycles whether its lanes hold a node or not, and one warp a
// scheduler already keeps it 70% busy.  So what counts is that every lane of
// every warp holds a node -- consecutive nodes do, whatever nx is, where a
// 32-wide tile leaves 24% of the lanes of a 97-wide and 38% of a 40-wide block
// idle -- and that the SMs get equal numbers of planes (the chunk depth:
// assign_tiles in cavity_capi.cu).

struct StepArgs {
  const BlockDev *blocks;
  int nblocks;
  const CavConst *cc;
  CavState *cs;
  double *partials;  // [tile][kPartStride]
  int parity;        // read base[parity], write base[parity ^ 1]
  int mode;          // 0 = step, 1 = spectral radius of the current state only
  unsigned int *tile_counter;  // persistent CTAs fetch tiles from it (zero before a step); null: one CTA per tile
  int ntiles;
  int local_dt;                // 1: each node at dt_n = cfl / S_n of its state (pseudo time)
  int skip_shell;              // 1: leave the nodes within two layers of a cut face to k_shell_f64
  int ncoarse;                 // coarse tiles of all blocks (scheduling indices below it)
  int nnu;                     // the first CTAs: the x walls' Nusselt sums of the state read here
  int slot;                    // of this step's maximum, dt-filter floor and tile counter
  int chained;                 // 1: dt and the centre shift from the step before (no kernel in between)
  double *dt_out;              // chained: dt goes here, too (null: nowhere)
};

// p of one stored node through L2
template <class S>
__device__ __forceinline__ double load_p_l2(const S *base, long long fs, long long o);
template <>
__device__ __forceinline__ double load_p_l2<double>(const double *base, long long, long long o) {
  return __ldcg(base + o);
}
template <>
__device__ __forceinline__ double load_p_l2<float>(const float *base, long long fs, long long o) {
  return (double)__ldcg(base + o) + (double)__ldcg(base + fs + o);
}

// The mean of p over the centre nodes (their count is 1, 2, 4 or 8: the scaling
// is exact), summed in lexicographic (k, j, i) order; absent nodes are zeros.
__device__ __forceinline__ double centre_mean(int n, const double *v) {
  double csum = 0.0;
  for (int m = 0; m < kMaxCentre; ++m) csum += v[m];
  return csum * (n == 8 ? 0.125 : n == 4 ? 0.25 : n == 2 ? 0.5 : 1.0);
}

__device__ __forceinline__ void step_max(double *slot, double smax) {
  // positive values order like their bit patterns
  atomicMax((unsigned long long *)slot, (unsigned long long)__double_as_longlong(smax));
}

// A programmatic dependent: every earlier kernel of the chain has finished
// and its memory is visible.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The kernel after this one may start when every CTA has said so (or ended): a
// step's CTAs do at the end of their sweeps, so that the next step's are not
// placed beside them on whichever SMs have room (an uneven spread: 128^3
// FP32-mixed 71 us a step against 52).
__device__ __forceinline__ void chain_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// whether local node (i, j, k) of B lies within two layers of one of B's cut
// faces with index below `faces` (all six: faces = 6)
__device__ __forceinline__ bool in_shell(const BlockDev &B, int i, int j, int k, int faces) {
  const int x[3] = {i, j, k}, n[3] = {B.nx, B.ny, B.nz};
  for (int f = 0; f < faces; ++f) {
    if (B.wall[f]) continue;
    const int a = f >> 1;
    if ((f & 1) ? x[a] >= n[a] - 1 : x[a] <= 2) return true;
  }
  return false;
}

__device__ __forceinline__ int find_block(const BlockDev *blocks, int nblocks, int cta) {
  int lo = 0, hi = nblocks - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (blocks[mid].tile_begin <= cta) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The tile of scheduling index c: its block, x/y tile, plane range and
// partial slot (coarse and fine chunks as described at BlockDev).
struct TileRef {
  int b, tx, ty, k0, k1, slot;
};

__device__ __forceinline__ TileRef tile_ref(const BlockDev *blocks, int nblocks, int ncoarse, int c) {
  const bool coarse = c < ncoarse;
  const int u = coarse ? c : c - ncoarse;
  // the last block whose first tile of this class is at or before u (blocks
  // without tiles of the class share their successor's start and are passed)
  int lo = 0, hi = nblocks - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    const int begin = coarse ? blocks[mid].coarse_begin : blocks[mid].fine_begin;
    if (begin <= u) lo = mid; else hi = mid - 1;
  }
  const BlockDev &B = blocks[lo];
  const int l = u - (coarse ? B.coarse_begin : B.fine_begin);
  TileRef T;
  T.b = lo;
  T.tx = l % B.tiles_x;
  T.ty = (l / B.tiles_x) % B.tiles_y;
  const int zl = l / (B.tiles_x * B.tiles_y);
  T.k0 = coarse ? zl * B.kc + 1 : B.zsplit + zl * B.kf + 1;
  T.k1 = coarse ? min(T.k0 + B.kc - 1, B.zsplit) : min(T.k0 + B.kf - 1, B.nz);
  const int tz = coarse ? zl : B.tiles_zc + zl;
  T.slot = B.tile_begin + T.tx + B.tiles_x * (T.ty + B.tiles_y * tz);
  return T;
}

// x / 3 correctly rounded in three FP64 operations (a rounded reciprocal, then
// one residual correction through fused multiply-adds: Markstein, IBM J. Res.
// Dev. 34 (1990)), where a full division is a long dependent FP64 sequence on
// GB300's narrow FP64 pipe.
__device__ __forceinline__ double div3(double x) {
  constexpr double y = 1.0 / 3.0;
  const double q = x * y;
  return fma(fma(-q, 3.0, x), y, q);
}

// the adiabatic wall's T from the two interior nodes next to it
__device__ __forceinline__ double adiabatic_T(double T1, double T2) { return div3(fma(4.0, T1, -T2)); }

// wfloor: a warp-uniform FP32 value of D = S - S0 at or below the one of an
// exact spectral value of this step that some lane of the warp -- or, through
// the cavity's published floor, of any CTA -- has already recorded, lowered
// by 1e-13 of that value (more than the FP64 rounding of S, of S0 and of
// their difference); -inf before the first.  A node whose estimate of D,
// raised by 1e-5 (over 10x its error), stays at or below wfloor cannot raise
// the maximum, so only the others are evaluated in FP64 and the maximum --
// hence dt -- is exactly the FP64 one.  Carried across the warp's tiles of
// one cavity (`fcav`: the cavity it belongs to; a tile of another cavity,
// in a batch, starts again from -inf).
//
// Walls (Section 2) are formed where they are read (FORM), from the two
// interior layers next to each wall, by the formulas k_bc stores them with: two
// FP64 operations in the warps that hold a node next to an x wall, a few in the
// first and last planes.  u = v = w = 0 and the isothermal T never change and
// stay stored.  Large cavities read stored walls, which k_between writes: the
// line is at 64 tile planes an SM: 128^3 263 us a step with walls formed, 257
// stored, 256^3 1890 and 1843; 64^3 45 either way, 32^3 11.6 and 13.1.
template <int NT, bool FORM>
__device__ __forceinline__ void step_tile_f64(const StepArgs &a, int cta, const double *dc, float &wfloor, int &fcav) {
  const TileRef tile = tile_ref(a.blocks, a.nblocks, a.ncoarse, cta);
  const BlockDev &B = a.blocks[tile.b];
  const CavConst &C = a.cc[B.cav];
  CavState &st = a.cs[B.cav];
  if (B.cav != fcav) {
    wfloor = -INFINITY;
    fcav = B.cav;
  }
  // the cavity's floor as published by every CTA so far this step (a value
  // at or below an exact spectral value some warp recorded): warps far from
  // the maximum start near it too
  if (a.mode == 0) {
    const unsigned u = *(volatile const unsigned *)&st.sfl[a.slot];
    if (u != 0u) wfloor = fmaxf(wfloor, key_float((int)(u ^ 0x80000000u)));
  }
  float published = wfloor;
  const int tid = threadIdx.x, e = tile.tx * NT + tid;
  const int j = e / B.nx + 1, i = e - (j - 1) * B.nx + 1;
  const int k0 = tile.k0;
  const int k1 = tile.k1;
  const bool active = j <= B.ny;
  if (!FORM || !dc) dc = &st.dt;
  const double dt = dc[0], cshift = dc[1];

  const double *__restrict__ src = (const double *)B.base[a.parity];
  double *__restrict__ dst = (double *)B.base[a.parity ^ 1];
  const long long fs = B.fstride;
  const double *__restrict__ P = src;
  const double *__restrict__ U = src + fs;
  const double *__restrict__ V = src + 2 * fs;
  const double *__restrict__ W = src + 3 * fs;
  const double *__restrict__ TT = src + 4 * fs;
  const long long pl = B.plane, pt = B.pitch;

  // the node's place next to the x and y walls: bits 1, 2 the first and second
  // node from x = 0, 4, 8 from the other x wall, 16 .. 128 the y walls
  int edge = 0;
  if (B.wall[0]) edge |= i == 1 ? 1 : i == 2 ? 2 : 0;
  if (B.wall[1]) edge |= i == B.nx ? 4 : i == B.nx - 1 ? 8 : 0;
  if (B.wall[2]) edge |= j == 1 ? 16 : j == 2 ? 32 : 0;
  if (B.wall[3]) edge |= j == B.ny ? 64 : j == B.ny - 1 ? 128 : 0;
  const int zlow = B.wall[4] ? 2 : 0, zhigh = B.wall[5] ? B.nz - 1 : B.nz + 1;  // planes next to the z walls
  double s0 = 0, s1 = 0, s2 = 0, s3 = 0, s4 = 0, smax = 0;
  if (active) {
    const bool edge_x = FORM && __any_sync(__activemask(), edge & 15);
    const bool edge_y = FORM && __any_sync(__activemask(), edge & 240);
    long long o = node_index<double>(B, i, j, k0);
    // z queues: p at k-2..k+1, the others at k-1..k
    double pq0 = P[o - 2 * pl], pq1 = P[o - pl], pq2 = P[o], pq3 = P[o + pl];
    double uq0 = U[o - pl], uq1 = U[o];
    double vq0 = V[o - pl], vq1 = V[o];
    double wq0 = W[o - pl], wq1 = W[o];
    double Tq0 = TT[o - pl], Tq1 = TT[o];
    for (int k = k0; k <= k1; ++k, o += pl) {
      NodeF64 n;
      const double pq4 = P[o + 2 * pl];
      const double uq2 = U[o + pl], vq2 = V[o + pl], wq2 = W[o + pl], Tq2 = TT[o + pl];
      if (a.mode == 0 && a.skip_shell && in_shell(B, i, j, k, 6)) {
        // computed by k_shell_f64 (interior/shell split)
      } else if (a.mode == 0) {
        n.p[0] = pq2; n.p[5] = pq1; n.p[6] = pq3; n.p[11] = pq0; n.p[12] = pq4;
        n.p[1] = P[o - 1]; n.p[2] = P[o + 1];
        n.p[7] = P[o - 2]; n.p[8] = P[o + 2];
        n.p[3] = P[o - pt]; n.p[4] = P[o + pt];
        n.p[9] = P[o - 2 * pt]; n.p[10] = P[o + 2 * pt];
#define BDC_LOAD7(arr, F, q0, q1, q2)                                           \
  arr[0] = q1; arr[5] = q0; arr[6] = q2;                                        \
  arr[1] = F[o - 1]; arr[2] = F[o + 1];                         \
  arr[3] = F[o - pt]; arr[4] = F[o + pt];
        BDC_LOAD7(n.T, TT, Tq0, Tq1, Tq2)
        BDC_LOAD7(n.u, U, uq0, uq1, uq2)
        BDC_LOAD7(n.v, V, vq0, vq1, vq2)
        BDC_LOAD7(n.w, W, wq0, wq1, wq2)
#undef BDC_LOAD7
        // the velocities' part first: it needs no wall value, and its arrays are
        // gone when the walls change p and T in place (168 registers; all
        // loads and the walls first took 218)
        VelF64 x;
        rates_vel_f64(C, n, x);
        // walls: branches a warp skips as a whole (inlined as predicated code,
        // their FP64 operations cost every warp 15%)
        if (FORM) {
          if (edge_x) {
            if (edge & 3) {  // x = 0: w = 2 p1 - p2, g = 2 w - p1
              if (edge & 1) n.p[1] = fma(2.0, pq2, -n.p[2]);
              n.p[7] = fma(2.0, n.p[1], -pq2);
            }
            if (edge & 12) {
              if (edge & 4) n.p[2] = fma(2.0, pq2, -n.p[1]);
              n.p[8] = fma(2.0, n.p[2], -pq2);
            }
          }
          if (edge_y) {
            if (edge & 48) {
              if (edge & 16) {
                n.p[3] = fma(2.0, pq2, -n.p[4]);
                n.T[3] = adiabatic_T(Tq1, n.T[4]);
              }
              n.p[9] = fma(2.0, n.p[3], -pq2);
            }
            if (edge & 192) {
              if (edge & 64) {
                n.p[4] = fma(2.0, pq2, -n.p[3]);
                n.T[4] = adiabatic_T(Tq1, n.T[3]);
              }
              n.p[10] = fma(2.0, n.p[4], -pq2);
            }
          }
          if (k <= zlow) {
            if (k == 1) {
              n.p[5] = fma(2.0, pq2, -pq3);
              n.T[5] = adiabatic_T(Tq1, Tq2);
            }
            n.p[11] = fma(2.0, n.p[5], -pq2);
          }
          if (k >= zhigh) {
            if (k == zhigh + 1) {
              n.p[6] = fma(2.0, pq2, -pq1);
              n.T[6] = adiabatic_T(Tq1, Tq0);
            }
            n.p[12] = fma(2.0, n.p[6], -pq2);
          }
        }
        double r[5], qn[5];
        update_node_f64(C, n, x, dt, cshift, a.local_dt, qn, r);
        const double un = qn[1], vn = qn[2], wn = qn[3];
        for (int f = 0; f < 5; ++f) dst[o + f * fs] = qn[f];
        s0 += r[0] * r[0]; s1 += r[1] * r[1]; s2 += r[2] * r[2]; s3 += r[3] * r[3]; s4 += r[4] * r[4];
        float best = -INFINITY;
        const float dest = spectral_dev_f32(C, abs_f32_trunc(un), abs_f32_trunc(vn), abs_f32_trunc(wn));
        if (__fmul_rn(dest, 1.00001f) > wfloor) {
          const double e = spectral_f64(C, un, vn, wn);
          smax = fmax(smax, e);
          best = __double2float_rd((e - C.s0) - 1e-13 * e);
        }
        // share over the lanes sweeping this tile (all active lanes run the same k range)
        const unsigned am = __activemask();
        wfloor = fmaxf(wfloor, key_float(__reduce_max_sync(am, float_key(best))));
        if (wfloor > published) {  // publish a rise for the other warps
          if ((int)(threadIdx.x & 31) == __ffs(am) - 1)
            atomicMax(&st.sfl[a.slot], (unsigned)float_key(wfloor) ^ 0x80000000u);
          published = wfloor;
        }
      } else {
        smax = fmax(smax, spectral_f64(C, uq1, vq1, wq1));
      }
      pq0 = pq1; pq1 = pq2; pq2 = pq3; pq3 = pq4;
      uq0 = uq1; uq1 = uq2; vq0 = vq1; vq1 = vq2; wq0 = wq1; wq1 = wq2; Tq0 = Tq1; Tq1 = Tq2;
    }
  }
  // CTA reduction of the six partials, in a fixed order and with few FP64
  // warp instructions (25 warp adds for the five sums of 128 threads, where a
  // shuffle tree in every warp takes 100): field f by the 16 threads 16 f ..
  // 16 f + 15, each NT / 16 values, then a butterfly; the maximum (of positive
  // values) on the bit patterns.
  __shared__ double red[5][NT];
  __shared__ unsigned long long redm[NT / 32];
  const int lane = tid & 31, wid = tid >> 5;
  red[0][tid] = s0; red[1][tid] = s1; red[2][tid] = s2; red[3][tid] = s3; red[4][tid] = s4;
  {
    const unsigned mh = (unsigned)__double2hiint(smax), ml = (unsigned)__double2loint(smax);
    const unsigned wh = __reduce_max_sync(0xffffffffu, mh);
    const unsigned wl = __reduce_max_sync(0xffffffffu, mh == wh ? ml : 0u);
    if (lane == 0) redm[wid] = ((unsigned long long)wh << 32) | wl;
  }
  __syncthreads();
  if (wid < 3) {
    const int f = tid >> 4, s = tid & 15;
    double v = 0.0;
    if (f < 5) {
      const double *p = &red[f][s];
#pragma unroll
      for (int q = 0; q < NT / 16; ++q) v = q == 0 ? p[0] : v + p[16 * q];
    }
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (f == 5) {
      unsigned long long m = redm[0];
      for (int q = 1; q < NT / 32; ++q) m = redm[q] > m ? redm[q] : m;
      v = __longlong_as_double((long long)m);
      if (s == 0 && a.mode == 0) step_max(&st.smax[a.slot], v);
    }
    if (s == 0) a.partials[(long long)tile.slot * kPartStride + f] = v;
  }
}

// ---------------------------------------------------------------------------
// k_shell_f64: the nodes within two layers of a cut face (the interior/shell
// split of Section 4.7).  They are stepped first, so that the exchange of the
// new ghost layers can run on a second stream while k_step_f64 (skip_shell)
// steps the rest.  One thread per (layer, face position) of each cut face;
// a node near an edge belongs to the first cut face (in face order) within
// two layers of it.  Partials: one slot per CTA after the tiles' slots.

struct ShellArgs {
  const BlockDev *blocks;
  const ShellFace *faces;
  int nfaces;
  const CavConst *cc;
  const CavState *cs;
  double *partials;       // slot part_off + cta
  long long part_off;
  int parity;
  int local_dt;
};

constexpr int kShellThreads = 256;

static __global__ void __launch_bounds__(kShellThreads) k_shell_f64(ShellArgs a) {
  const int cta = blockIdx.x, tid = threadIdx.x;
  int lo = 0, hi = a.nfaces - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.faces[mid].cta_begin <= cta) lo = mid; else hi = mid - 1;
  }
  const ShellFace &F = a.faces[lo];
  const BlockDev &B = a.blocks[F.block];
  const CavConst &C = a.cc[B.cav];
  double s[5] = {0, 0, 0, 0, 0}, smax = 0.0;
  const long long per_layer = (long long)F.n1 * F.n2;
  const long long e = (long long)(cta - F.cta_begin) * kShellThreads + tid;
  if (e < 2 * per_layer) {
    const int d = (int)(e / per_layer) + 1;
    const long long r2 = e % per_layer;
    const int ax = F.face >> 1, hi_face = F.face & 1;
    const int n[3] = {B.nx, B.ny, B.nz};
    int x[3];
    x[ax] = hi_face ? n[ax] + 1 - d : d;
    x[ax == 0 ? 1 : 0] = (int)(r2 % F.n1) + 1;
    x[ax == 2 ? 1 : 2] = (int)(r2 / F.n1) + 1;
    if (!in_shell(B, x[0], x[1], x[2], F.face)) {  // not claimed by an earlier cut face
      const double *src = (const double *)B.base[a.parity];
      double *dst = (double *)B.base[a.parity ^ 1];
      const long long fs = B.fstride, pt = B.pitch, pl = B.plane;
      const long long o = node_index<double>(B, x[0], x[1], x[2]);
      NodeF64 nd;
      const long long po[13] = {0, -1, 1, -pt, pt, -pl, pl, -2, 2, -2 * pt, 2 * pt, -2 * pl, 2 * pl};
      for (int q = 0; q < 13; ++q) nd.p[q] = __ldg(src + o + po[q]);
      for (int q = 0; q < 7; ++q) {
        nd.u[q] = __ldg(src + fs + o + po[q]);
        nd.v[q] = __ldg(src + 2 * fs + o + po[q]);
        nd.w[q] = __ldg(src + 3 * fs + o + po[q]);
        nd.T[q] = __ldg(src + 4 * fs + o + po[q]);
      }
      const CavState &st = a.cs[B.cav];
      double r[5], qn[5];
      VelF64 x;
      rates_vel_f64(C, nd, x);
      update_node_f64(C, nd, x, st.dt, st.c, a.local_dt, qn, r);
      for (int f = 0; f < 5; ++f) {
        dst[o + f * fs] = qn[f];
        s[f] = r[f] * r[f];
      }
      smax = spectral_f64(C, qn[1], qn[2], qn[3]);
    }
  }
  __shared__ double red[kShellThreads / 32][6];
  const int lane = tid & 31, wid = tid >> 5;
  for (int f = 0; f < 5; ++f) s[f] = warp_sum(s[f]);
  smax = warp_max(smax);
  if (lane == 0) {
    for (int f = 0; f < 5; ++f) red[wid][f] = s[f];
    red[wid][5] = smax;
  }
  __syncthreads();
  if (tid < 6) {
    double acc = red[0][tid];
    for (int q = 1; q < kShellThreads / 32; ++q) acc = (tid == 5) ? fmax(acc, red[q][tid]) : acc + red[q][tid];
    a.partials[(a.part_off + cta) * kPartStride + tid] = acc;
  }
}

// ---------------------------------------------------------------------------
// k_bc (wall conditions + Nusselt partials) and k_finalize (reduction of the
// partials, state advance).

// k_pack / k_unpack / k_exchange (below)
struct ExchArgs {
  const BlockDev *blocks;
  const CutFace *faces;
  int nfaces;
  double *buf;   // FP64 storage: values; FP32 storage: reinterpreted as float
  int parity;
};

constexpr int kGraphMax = 16;  // steps of the longest graph

struct StepResult {  // one step's outcome of one cavity, from that step's last finalise CTA
  double res[5], dt, nu[2];
  int bad;
};

struct BcArgs {
  const BlockDev *blocks;
  const WallFace *faces;
  int nfaces;
  const CavConst *cc;
  CavState *cs;
  int ncav;
  const double *step_partials;
  double *bc_partials;        // [k_bc cta][2]
  unsigned int *counter;      // [nsteps][ncav] CTAs done, then [ncav] steps done (zero between launches)
  const double *t_wall;       // hot walls then cold walls, per cavity at wall_off
  unsigned int *tile_counter; // the FP64 step's tile counters (kStepSlots): reset here
  long long shell_begin, shell_end;  // k_shell_f64 partial slots of this step (single cavity; empty if equal)
  int parity;                 // buffer set holding the new state
  int nslices;                // finalise CTAs per cavity (1 .. kFinSlices)
  int wall_ctas;              // after an FP64 step: CTAs of the finalise that take the x walls' Nusselt sums
                              //   (nu_only), or all walls (the overlapped schedule)
  int nu_only;                // 1: wall_ctas read the new state's T next to the x walls (faces: the x walls
                              //   alone) and write no walls
  int nsteps;                 // steps of the graph (1 .. kGraphMax), their partials part_stride, bc_stride apart
  long long part_stride, bc_stride;
  double *mid;                // [nsteps][ncav][kFinSlices][8] slice totals
  StepResult *rec;            // [nsteps][ncav]
  double *dt_out;             // k_between: the next step's dt goes here, too (null: nowhere)
  int slot;                   // k_between: the slot of the step before it
  StepRecord *log;            // after a step: the step log (host memory), or null
  long long log_cap;          // its records per cavity
  int mode;                   // 0 after a step, 1 after init / set_fields,
                              // 3 walls only (k_bc), no reductions, 5 the same with
                              //   the constant walls in both buffer sets,
                              // 4 after an FP32 step (k_finalize only): Nusselt
                              //   sums in the step partials
};

// the outward wall heat flux over the temperature difference at an x-wall node
__device__ __forceinline__ double wall_flux(const CavConst &C, double tw, double T1, double T2) {
  return (3.0 * tw - 4.0 * T1 + T2) * (0.5 * C.ih[0]) * C.inv_dT;
}

// Walls of one face node.  u = v = w = 0 and the isothermal T never change
// between steps: they are written (into both buffer sets) only when `other`
// is given (state refresh); p's wall and ghost values and the adiabatic T are
// written, and T next to the x walls goes into the Nusselt sums.
template <class S>
__device__ __forceinline__ void apply_wall(const BlockDev &B, const CavConst &C, S *base, int face,
                                           int c1, int c2, const double *t_wall, double &nu_h,
                                           double &nu_c, S *other = nullptr) {
  // wall node: coordinate w on the face axis, c1 on the face's faster axis (y
  // for x faces, else x), c2 on the slower one (z, except y for z faces)
  const int axis = face >> 1, high = face & 1;
  const int na = axis == 0 ? B.nx : (axis == 1 ? B.ny : B.nz);
  const int w = high ? na + 1 : 0;
  const int s = high ? -1 : 1;
  const long long W = node_index<S>(B, axis == 0 ? w : c1, axis == 0 ? c1 : (axis == 1 ? w : c2), axis == 2 ? w : c2);
  const long long step = axis == 0 ? 1 : (axis == 1 ? (long long)B.pitch : B.plane);
  const long long N1 = W + s * step, N2 = W + 2 * s * step, G = W - s * step;
  const long long fs = B.fstride;
  constexpr int NP = Store<S>::NP;
  // every load before the first store (the stores go to the wall and ghost
  // nodes, the loads read interior ones, but the compiler cannot tell)
  const double p1 = load_p<S>(base, fs, N1), p2 = load_p<S>(base, fs, N2);
  const double T1 = load_T<S>(base, fs, N1), T2 = load_T<S>(base, fs, N2);
  double tw = 0.0;
  if (axis == 0) {
    const int J = B.oy + c1, K = B.oz + c2;
    const long long widx = (long long)(J - 1) + (long long)C.gn[1] * (K - 1);
    tw = t_wall[C.wall_off + (high ? (long long)C.gn[1] * C.gn[2] : 0) + widx];
  }
  if (other) {
    base[NP * fs + W] = S(0); base[(NP + 1) * fs + W] = S(0); base[(NP + 2) * fs + W] = S(0);
    other[NP * fs + W] = S(0); other[(NP + 1) * fs + W] = S(0); other[(NP + 2) * fs + W] = S(0);
  }
  const double pw = 2.0 * p1 - p2;
  store_p<S>(base, fs, W, pw);
  store_p<S>(base, fs, G, 2.0 * pw - p1);
  if (axis == 0) {
    if (other) {
      store_T<S>(base, fs, W, tw);
      store_T<S>(other, fs, W, tw);
    }
    const double flux = wall_flux(C, tw, T1, T2);
    if (high) nu_c += -flux; else nu_h += flux;
  } else {
    store_T<S>(base, fs, W, adiabatic_T(T1, T2));
  }
}

// ---------------------------------------------------------------------------
// Finalise: one cavity's per-CTA partials reduced in a fixed order and its
// state advanced (residual RMS, spectral maximum -> next dt, Nusselt numbers,
// time, step count, centre pressure).  GB300's FP64 pipe does about two
// lanes per clock per SM, and one dependent FP64 add costs tens of cycles,
// so the FP64 sums are spread over up to kFinSlices CTAs per cavity
// (BcArgs::nslices, contiguous slices of the partials, about 128 partials a
// slice) and every sum is a shallow fixed tree: within a CTA the eight
// fields are transposed through shared memory and summed by 16 threads each
// (an 8-term tree, then four butterfly levels), and the last CTA of a cavity
// combines the slice totals by the same butterfly.  Nusselt sums: the x-wall
// CTAs' or the wall kernel's partials (modes 0, 1) or the step partials' slots
// 6 and 7, sums of 3 T_w - 4 T_1 + T_2 (mode 4, FP32 step).
//
// Where it runs: nothing of it is needed to start the next step (dt comes from
// the atomic maximum, the centre shift from the state itself), so it runs once
// at the end of a graph, for all of the graph's steps at once, each from its own
// set of partials; the last step's last CTA then goes through the steps in
// order (time, step log, flags).  As a kernel between the steps it took 7-9 us
// of every step (FP32-mixed 256^3), 12 with the FP64 walls and 16-19 with a
// decomposed cavity's exchange.  (In the first CTAs of the next step's launch
// instead, its call cost the FP32 step kernel spills and 7% of its time.)
constexpr int kFinThreads = 128;

__device__ __forceinline__ double fin_comb(int f, double x, double y) { return f == 5 ? fmax(x, y) : x + y; }

// Field f of the NT values in sv[f * NT ..] summed (f == 5: maximum) by the
// 16 threads t = 16 f .. 16 f + 15 of the CTA: thread s of the group takes
// values s, s + 16, .. s + 112 in a 3-level tree, then a butterfly over the
// group; every thread of the group ends with the same total.
template <int NT>
__device__ __forceinline__ double fin_tree(const double *sv, int f, int s) {
  static_assert(NT == 128, "eight fields x 16 threads, eight values a thread");
  const double *p = sv + f * NT + s;
  const double a0 = fin_comb(f, p[0], p[16]), a1 = fin_comb(f, p[32], p[48]);
  const double a2 = fin_comb(f, p[64], p[80]), a3 = fin_comb(f, p[96], p[112]);
  double v = fin_comb(f, fin_comb(f, a0, a1), fin_comb(f, a2, a3));
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) v = fin_comb(f, v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// One slice of a cavity's partials, thread tid's in thread-strided order.
template <int NT>
__device__ __forceinline__ void load_slice(const BcArgs &a, const double *step_partials, long long q0, long long q1,
                                           long long b0, long long b1, long long s0, long long s1, int tid,
                                           double acc[8]) {
  for (int f = 0; f < 8; ++f) acc[f] = 0.0;  // the spectral radius is positive: 0 is its identity too
  long long q = q0 + tid;
  if (q < q1) {  // the first partial is taken as it is, not added to zero
    const double2 *pp = reinterpret_cast<const double2 *>(step_partials + q * kPartStride);
    const double2 x0 = pp[0], x1 = pp[1], x2 = pp[2], x3 = pp[3];
    acc[0] = x0.x; acc[1] = x0.y; acc[2] = x1.x; acc[3] = x1.y; acc[4] = x2.x; acc[5] = x2.y;
    if (a.mode == 4) { acc[6] = x3.x; acc[7] = x3.y; }
    q += NT;
  }
#pragma unroll 4
  for (; q < q1; q += NT) {
    const double *pp = step_partials + q * kPartStride;
    for (int f = 0; f < 5; ++f) acc[f] += pp[f];
    acc[5] = fmax(acc[5], pp[5]);
    if (a.mode == 4) {
      acc[6] += pp[6];
      acc[7] += pp[7];
    }
  }
  for (long long r = s0 + tid; r < s1; r += NT) {  // shell-kernel partials
    const double *pp = step_partials + r * kPartStride;
    for (int f = 0; f < 5; ++f) acc[f] += pp[f];
    acc[5] = fmax(acc[5], pp[5]);
  }
  for (long long r = b0 + tid; r < b1; r += NT) {
    acc[6] += a.bc_partials[2 * r];
    acc[7] += a.bc_partials[2 * r + 1];
  }
}

// The CTA tree of the threads' slice sums: field f's total ends in threads
// 16 f .. 16 f + 15.
template <int NT>
__device__ __forceinline__ double tree_slice(const double acc[8], double *sv, int tid) {
#pragma unroll
  for (int f = 0; f < 8; ++f) sv[f * NT + tid] = acc[f];
  __syncthreads();
  return fin_tree<NT>(sv, tid >> 4, tid & 15);
}

template <class S, int NT>
__device__ __forceinline__ void exchange_cta(const ExchArgs &a, int cta);
template <class S>
__device__ __forceinline__ int bc_cta(const BcArgs &a, int cta, bool reduce);

// The x walls' Nusselt partial of one CTA: kBcThreads positions of one face
// (its first threads; sh: a double per warp).  Returns the face's cavity.
template <class S>
__device__ __forceinline__ int nu_cta(const BcArgs &a, int cta, double *sh) {
  const int tid = threadIdx.x;
  int fi = 0;
  for (int base = 0; base < a.nfaces; base += 32) {
    const int l = base + (tid & 31);
    const unsigned m = __ballot_sync(0xffffffffu, l < a.nfaces && a.faces[l].cta_begin <= cta);
    if (m) fi = base + 31 - __clz(m);
  }
  const WallFace &F = a.faces[fi];
  const BlockDev &B = a.blocks[F.block];
  const CavConst &C = a.cc[F.cav];
  const int high = F.face & 1, e = (cta - F.cta_begin) * kBcThreads + tid;
  double flux = 0.0;
  if (tid < kBcThreads && e < F.n1 * F.n2) {
    const int j = e % F.n1 + 1, k = e / F.n1 + 1;
    const S *q = (const S *)B.base[a.parity];
    const long long N1 = node_index<S>(B, high ? B.nx : 1, j, k), N2 = high ? N1 - 1 : N1 + 1;
    const double T1 = load_T<S>(q, B.fstride, N1), T2 = load_T<S>(q, B.fstride, N2);
    const long long widx = (long long)(B.oy + j - 1) + (long long)C.gn[1] * (B.oz + k - 1);
    flux = wall_flux(C, a.t_wall[C.wall_off + (high ? (long long)C.gn[1] * C.gn[2] : 0) + widx], T1, T2);
    if (high) flux = -flux;
  }
  const double v = warp_sum(flux);
  if ((tid & 31) == 0) sh[tid >> 5] = v;
  __syncthreads();
  if (tid == 0) {
    double t = 0;
    for (int q = 0; q < kBcThreads / 32; ++q) t += sh[q];
    a.bc_partials[2LL * cta] = high ? 0.0 : t;
    a.bc_partials[2LL * cta + 1] = high ? t : 0.0;
  }
  return F.cav;
}

// The totals of a step, field f's in thread 16 f: the slices' totals (shm, [slice][field])
// combined by the field's 16 threads (slice s in thread 16 f + s, a butterfly over the
// first nsl), then in fields 6 and 7 the tree of the wall CTAs' Nusselt partials w0 ..
// w1 - 1, thread-strided (rows 6 and 7 of sv, which nobody may be reading any more).
template <int NT>
__device__ __forceinline__ double step_totals(const double *bc_partials, int w0, int w1, int nsl, const double *shm,
                                              double *sv, int tid) {
  const int f = tid >> 4, s = tid & 15;
  if (w1 > w0) {
    double h = 0.0, c = 0.0;
    for (int q = w0 + tid; q < w1; q += NT) {
      h += bc_partials[2LL * q];
      c += bc_partials[2LL * q + 1];
    }
    sv[6 * NT + tid] = h;
    sv[7 * NT + tid] = c;
  }
  __syncthreads();
  double t = s < nsl ? shm[s * 8 + f] : 0.0;
  for (int o = 1; o < nsl; o <<= 1) t = fin_comb(f, t, __shfl_xor_sync(0xffffffffu, t, o));
  if (w1 > w0 && f >= 6) t += fin_tree<NT>(sv, f, s);
  return t;
}

// The step log's record of step s of a sequence of steps that one finalise ends, one CTA a
// cavity, on a stream beside the steps': it waits for step s + 1 (whose launch leaves
// the x walls' Nusselt partials of step s) and runs beside step s + 2, by the finalise's
// sums in the finalise's order.  The finalise writes the last two records.  So every
// record is in host memory two steps later at most; with the finalise's alone they came
// once a sequence, up to 16 steps late, those that a shorter ring has no room for never.
// A logged step takes 1-3% more than an unlogged one (FP64 32^3 11.7 us, 11.4; 64^3 46.4, 44.9;
// 128^3 in 2x2x2 blocks 268, 264; FP32-mixed 256^3 211.1, 210.8): the finalise has to
// wait for the records and is no programmatic dependent of the last step then.
static __global__ void __launch_bounds__(kFinThreads) k_step_record(BcArgs a, int s) {
  constexpr int NT = kFinThreads;
  __shared__ double sv[8 * NT];
  __shared__ double shm[kFinSlices * 8];
  __shared__ double val[8];
  const int cav = blockIdx.x, tid = threadIdx.x, f = tid >> 4;
  const CavConst &C = a.cc[cav];
  for (int g = 0; g < a.nslices; ++g) {
    double acc[8];
    load_slice<NT>(a, a.step_partials, C.slice_q[g], C.slice_q[g + 1], 0, 0, 0, 0, tid, acc);
    const double t = tree_slice<NT>(acc, sv, tid);
    if ((tid & 15) == 0) shm[g * 8 + f] = t;
    __syncthreads();  // (before the next slice, or the wall partials, overwrite sv)
  }
  double t = step_totals<NT>(a.bc_partials, a.wall_ctas ? C.nu_begin : 0, a.wall_ctas ? C.nu_end : 0, a.nslices, shm, sv,
                             tid);
  const bool bad = (tid & 15) == 0 && f < 6 && !isfinite(t);
  if ((tid & 15) == 0) {
    if (f >= 6 && a.mode == 4) t *= C.wscale[f - 6];
    val[f] = f < 5 ? sqrt(t * C.inv_nint) : f == 5 ? C.cfl / t : t * C.inv_nwall;
  }
  const int any = __syncthreads_or(bad);
  if (tid != 0) return;
  CavState &st = a.cs[cav];
  const double tt = s == 0 ? st.t + st.dt0 : st.log_t + st.log_dt;
  const long long step = st.step + s + 1, nonfin = (s == 0 ? 0 : st.log_bad) | (any ? 1 : 0);
  st.log_t = tt;
  st.log_dt = val[5];
  st.log_bad = nonfin;
  StepRecord &o = a.log[((step - 1) % a.log_cap) * a.ncav + cav];
  o.step = step;
  o.t = tt;
  o.dt = val[5];
  for (int q = 0; q < 5; ++q) o.res[q] = val[q];
  o.nu_hot = val[6];
  o.nu_cold = val[7];
  o.flags = *(volatile int *)&st.flags | nonfin;
}

// What a graph's last step leaves beside its sums, in CTAs from `begin` on of the
// same launch: the exchange of the new state's cut faces, then its stored walls.
// (They write ghosts and walls, the finalise reads partials and interior nodes.)
// As a k_between before the finalise they cost every graph 4-6 us more: FP32-mixed
// 128^3 in 2x2x2 blocks, calls of one step, 65 us against 60.6 now.
struct FinTail {
  int begin, ncut;
  ExchArgs x;
  BcArgs walls;
};

template <class S>
__global__ void __launch_bounds__(kFinThreads) k_finalize(BcArgs a, const __grid_constant__ FinTail tail) {
  constexpr int NT = kFinThreads;
  __shared__ double sv[8 * NT];
  __shared__ double shm[kFinSlices * 8];
  __shared__ double shc[8];
  __shared__ double snu[NT / 32];
  __shared__ double st_t[kGraphMax];
  __shared__ double one[8];
  __shared__ bool am_last;
  static_assert(kFinSlices * 8 <= NT && kFinSlices == 16, "one slice total per thread, 16 threads a field");
  static_assert(kBcThreads == NT, "a wall position per thread");
  chain_wait();
  if ((int)blockIdx.x >= tail.begin) {
    const int c = blockIdx.x - tail.begin;
    if (c < tail.ncut) exchange_cta<S, NT>(tail.x, c);
    else bc_cta<S>(tail.walls, c - tail.ncut, false);
    return;
  }
  const int nsl = a.nslices, tid = threadIdx.x, f = tid >> 4, s = tid & 15, M = a.nsteps;
  const int nslice = M * a.ncav * nsl;
  const bool slice = (int)blockIdx.x < nslice;
  int cav, m = M - 1, g = 0;  // cavity, step of the graph, slice
  if (slice) {
    m = blockIdx.x / (a.ncav * nsl);
    const int r = blockIdx.x - m * a.ncav * nsl;
    cav = r / nsl;
    g = r - cav * nsl;
  } else {
    // a wall CTA (FP64, the last step's state): its Nusselt partial (and
    // walls), then it arrives like a slice (thread 0 wrote the partial)
    const int c = blockIdx.x - nslice;
    BcArgs b = a;
    b.bc_partials += m * a.bc_stride;
    cav = a.nu_only ? nu_cta<S>(b, c, snu) : bc_cta<S>(b, c, true);
    if (tid == 0) __threadfence();
  }
  const CavConst &C = a.cc[cav];
  CavState &st = a.cs[cav];
  const bool last_step = m == M - 1;
  double acc[8];
  if (slice) {
    // slice bounds: the step partials' from the host's table; the wall and
    // shell partials' (after a state refresh, the overlapped schedule) in
    // 32-bit arithmetic (counts far below 2^27)
    const unsigned nb = (a.mode == 4 || a.wall_ctas) ? 0u : (unsigned)(C.bc_end - C.bc_begin);
    const unsigned ns = (unsigned)(a.shell_end - a.shell_begin);
    load_slice<NT>(a, a.step_partials + m * a.part_stride, C.slice_q[g], C.slice_q[g + 1], C.bc_begin + nb * g / nsl,
                   C.bc_begin + nb * (g + 1) / nsl, a.shell_begin + ns * g / nsl, a.shell_begin + ns * (g + 1) / nsl,
                   tid, acc);
  }
  // loads for whichever CTA of the step comes last, issued while the partials
  // are in flight: the final state's centre pressure (at most 8 nodes)
  double cp = 0.0;
  if (last_step && a.mode != 1 && tid < C.ncentre) {
    const BlockDev &B = a.blocks[C.centre_blk[tid]];
    cp = load_p<S>((const S *)B.base[a.parity], B.fstride, C.centre_off[tid]);
  }
  // (and, where there is one step alone, the state it advances, which only that CTA writes)
  double t0 = 0.0, dt0 = 0.0, nu_sum0 = 0.0;
  long long step0 = 0;
  int flags0 = 0;
  if (M == 1 && tid == 0) {
    t0 = st.t;
    dt0 = st.dt0;
    nu_sum0 = st.nu_sum;
    step0 = st.step;
    flags0 = st.flags;
  }
  double *mid = a.mid + ((long long)m * a.ncav + cav) * kFinSlices * 8;
  // the step's wall CTAs in this launch
  const int nwall = !a.wall_ctas ? 0 : a.nu_only ? C.nu_end - C.nu_begin : C.bc_end - C.bc_begin;
  const int arrivals = nsl + (last_step ? nwall : 0);
  if (slice) {
    const double tf = tree_slice<NT>(acc, sv, tid);
    if (arrivals == 1) {
      // the only CTA of the step: its totals go straight to the fold
      if (s == 0) shm[f] = tf;
    } else if (s == 0) {
      mid[g * 8 + f] = tf;
      __threadfence();
    }
  }
  if (arrivals > 1) {
    unsigned int *cnt = a.counter + m * a.ncav + cav;
    __syncthreads();
    if (tid == 0) am_last = atomicAdd(cnt, 1u) == (unsigned int)arrivals - 1u;
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    if (tid == 0) *cnt = 0u;
    // the slice totals loaded in parallel
    if (tid < nsl * 8) shm[tid] = mid[tid];
  } else if (nwall) {
    __syncthreads();  // warp 3 is done with rows 6 and 7 of sv (its part of the slice's tree)
  }
  if (tid < 8) shc[tid] = cp;
  // (the graph's earlier steps' wall partials were left by the next step's launch)
  const int w0 = !nwall ? 0 : a.nu_only ? C.nu_begin : C.bc_begin;
  const int w1 = !nwall ? 0 : a.nu_only ? C.nu_end : C.bc_xend;  // (the other walls' are zeros)
  double t = step_totals<NT>(a.bc_partials + m * a.bc_stride, w0, w1, nsl, shm, sv, tid);
  // one thread of each field group finishes its field (the FP64 chains run
  // side by side): residual norms, dt, Nusselt numbers; thread 1 the centre
  StepResult &out = a.rec[(long long)m * a.ncav + cav];
  const bool nonfin = s == 0 && f < 6 && (f == 5 || a.mode != 1) && !isfinite(t);
  if (s == 0) {
    if (f >= 6 && a.mode == 4) t *= C.wscale[f - 6];  // sums of 3 T_w - 4 T_1 + T_2 -> wall fluxes
    const double v = f < 5 ? sqrt(t * C.inv_nint) : f == 5 ? C.cfl / t : t * C.inv_nwall;
    if (M == 1) one[f] = v;
    else if (f < 5) out.res[f] = v;
    else if (f == 5) out.dt = v;
    else out.nu[f - 6] = v;
    if (f == 5 && last_step) {  // the next step starts from this state
      for (int q = 0; q < kStepSlots; ++q) {
        st.smax[q] = 0.0;
        st.sfl[q] = 0u;
        if (cav == 0) a.tile_counter[q] = 0u;
      }
    }
  }
  if (tid == 1 && last_step && a.mode != 1) {  // the pending shift of the final state
    st.c = centre_mean(C.ncentre, shc);
  }
  const int bad = __syncthreads_or(nonfin);
  if (M == 1) {
    // one step: nothing to go through, and no round trips through a.rec.  Calls of one
    // step took 1-2 us more by the way below: FP32-mixed 128^3 65.5 us (63.9 now), in 2x2x2
    // blocks 65.2 (64.0), FP64 275.5 (274.2)
    const bool step = a.mode != 1;  // (mode 1: no step was taken)
    if (tid < 5 && step) st.res[tid] = one[tid];
    if (tid == 5) st.dt = st.dt0 = one[5];
    if (tid == 6) st.nu_hot = one[6];
    if (tid == 7) st.nu_cold = one[7];
    if (tid != 0) return;
    if (bad) atomicOr(&st.flags, 1);
    if (!step) return;
    st.t = t0 + dt0;
    st.step = step0 + 1;
    st.nu_sum = nu_sum0 + one[6];
    if (a.log) {
      StepRecord &o = a.log[(step0 % a.log_cap) * a.ncav + cav];
      o.step = step0 + 1;
      o.t = t0 + dt0;
      o.dt = one[5];
      for (int q = 0; q < 5; ++q) o.res[q] = one[q];
      o.nu_hot = one[6];
      o.nu_cold = one[7];
      o.flags = flags0 | (bad ? 1 : 0);
    }
    return;
  }
  if (tid == 0) out.bad = bad;
  {
    // the cavity's last step to get here goes through all of them
    __threadfence();
    __syncthreads();
    unsigned int *cnt = a.counter + M * a.ncav + cav;
    if (tid == 0) {
      am_last = atomicAdd(cnt, 1u) == (unsigned int)M - 1u;
      if (am_last) *cnt = 0u;
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
  }
  const StepResult *r = a.rec + cav;  // step q at r[q * ncav]
  // the time after each step: the dt of a step is the one before it left
  if (tid < M) sv[tid] = tid == 0 ? st.dt0 : __ldcg(&r[(long long)(tid - 1) * a.ncav].dt);
  const unsigned badm = __ballot_sync(0xffffffffu, tid < M && __ldcg(&r[(long long)tid * a.ncav].bad));
  step0 = st.step;
  flags0 = st.flags;
  __syncthreads();
  if (tid == 0) {
    double tt = st.t;
    for (int q = 0; q < M; ++q) st_t[q] = tt += sv[q];
    st.t = tt;
    st.step = step0 + M;
    double sum = st.nu_sum;
    for (int q = 0; q < M; ++q) sum += __ldcg(&r[(long long)q * a.ncav].nu[0]);
    st.nu_sum = sum;
    if (badm) atomicOr(&st.flags, 1);
  }
  __syncthreads();
  if (tid < M) {
    const StepResult &x = r[(long long)tid * a.ncav];
    double res[5];
    for (int q = 0; q < 5; ++q) res[q] = __ldcg(&x.res[q]);
    const double dt = __ldcg(&x.dt), nh = __ldcg(&x.nu[0]), nc = __ldcg(&x.nu[1]);
    if (tid == M - 1) {
      for (int q = 0; q < 5; ++q) st.res[q] = res[q];
      st.dt = st.dt0 = dt;
      st.nu_hot = nh;
      st.nu_cold = nc;
    }
    if (a.log && M - tid <= min(a.log_cap, 2ll)) {  // the last records, written to host memory (k_step_record's before)
      const long long step = step0 + tid + 1;
      StepRecord &o = a.log[((step - 1) % a.log_cap) * a.ncav + cav];
      o.step = step;
      o.t = st_t[tid];
      o.dt = dt;
      for (int q = 0; q < 5; ++q) o.res[q] = res[q];
      o.nu_hot = nh;
      o.nu_cold = nc;
      o.flags = flags0 | ((badm & (2u << tid) - 1u) ? 1 : 0);
    }
  }
}

// ---------------------------------------------------------------------------
// k_step_f64.  The first a.nnu CTAs take the x walls' Nusselt sums of the state
// the step reads (d), the result of the step before.
//
// Persistent form: as many CTAs as fit on the GPU at once take tiles in
// order from a counter, so the last round is short (one CTA per tile left a
// partial wave of up to a third of the step on 152 SMs); the counter hands
// out every block's coarse tiles before the fine tail tiles, and the next
// tile is fetched while the current one is computed.  Partials stay indexed by
// tile slot: the reductions do not depend on which CTA took a tile.
//
// Three CTAs of 128 an SM (168 registers a thread; the form that reads stored walls
// spills 8 bytes): 256^3 takes 2165 us a step with the 204 registers the compiler
// takes unasked (two CTAs), 1900 with four CTAs (128 registers, spills).
template <int NT, bool FORM>
__global__ void __launch_bounds__(NT, NT == 128 ? 3 : 1) k_step_f64(StepArgs a, const __grid_constant__ BcArgs d) {
  chain_wait();
  if ((int)blockIdx.x < a.nnu) {
    __shared__ double snu[NT / 32];
    nu_cta<double>(d, blockIdx.x, snu);
    return;
  }
  float wfloor = -INFINITY;
  int fcav = -1;
  if (!a.tile_counter) {
    step_tile_f64<NT, FORM>(a, blockIdx.x, nullptr, wfloor, fcav);
    return;
  }
  const double *dc = nullptr;
  if (FORM && a.chained) {
    // what k_between does for the others, in every CTA (one cavity, one block);
    // starting the first tile's loads before it changes nothing (32^3 11.7 us)
    __shared__ double s_dc[2];
    dc = s_dc;
    CavState &st = a.cs[0];
    if (threadIdx.x == 0) {
      const CavConst &C = a.cc[0];
      const double *p = (const double *)a.blocks[0].base[a.parity];
      double c[kMaxCentre];
#pragma unroll
      for (int q = 0; q < kMaxCentre; ++q) c[q] = q < C.ncentre ? __ldcg(p + C.centre_off[q]) : 0.0;
      s_dc[1] = centre_mean(C.ncentre, c);
    } else if (threadIdx.x == 32) {
      const double dt = a.cc[0].cfl / __ldcg(&st.smax[(a.slot + kStepSlots - 1) % kStepSlots]);
      s_dc[0] = dt;
      if ((int)blockIdx.x == a.nnu) {
        const int next = (a.slot + 1) % kStepSlots;
        st.smax[next] = 0.0;
        st.sfl[next] = 0u;
        a.tile_counter[next - a.slot] = 0u;
        if (a.dt_out) *a.dt_out = dt;
      }
    }
    __syncthreads();
  }
  // the first tile of each CTA is its own index; the counter goes on from the grid's size
  __shared__ int s_tile[2];
  int tile = blockIdx.x - a.nnu;
  for (int n = 0; tile < a.ntiles; n ^= 1) {
    if (threadIdx.x == 0) s_tile[n] = (int)(gridDim.x - a.nnu + atomicAdd(a.tile_counter, 1u));
    step_tile_f64<NT, FORM>(a, tile, dc, wfloor, fcav);
    __syncthreads();
    tile = s_tile[n];
  }
  chain_trigger();
}

// k_bc: wall conditions of every wall face node and the Nusselt partials of
// the x walls, one partial pair per CTA (reduced by k_finalize).
// One CTA of the wall conditions: the wall nodes of kBcThreads positions of
// one face (any block size: each thread takes every blockDim.x-th); with
// `reduce`, the CTA's x-wall Nusselt partial (zeros for other faces).  Returns
// the face's cavity.
template <class S>
__device__ __forceinline__ int bc_cta(const BcArgs &a, int cta, bool reduce) {
  __shared__ double sh[kBcThreads / 32];
  const int tid = threadIdx.x, nwarps = blockDim.x / 32;
  int cav = 0;
  double nu_h = 0.0, nu_c = 0.0;
  bool xwall = false, xhigh = false;
  if (a.nfaces > 0) {
    // the face of this CTA: the last one whose first CTA is not after it (a warp-wide search)
    int fi = 0;
    for (int base = 0; base < a.nfaces; base += 32) {
      const int l = base + (tid & 31);
      const unsigned m = __ballot_sync(0xffffffffu, l < a.nfaces && a.faces[l].cta_begin <= cta);
      if (m) fi = base + 31 - __clz(m);
    }
    const WallFace &F = a.faces[fi];
    cav = F.cav;
    xwall = (F.face >> 1) == 0;
    xhigh = F.face & 1;
    for (int sub = tid; sub < kBcThreads; sub += blockDim.x) {
      const int e = (cta - F.cta_begin) * kBcThreads + sub;
      if (e < F.n1 * F.n2) {
        const BlockDev &B = a.blocks[F.block];
        apply_wall<S>(B, a.cc[F.cav], (S *)B.base[a.parity], F.face, e % F.n1 + 1, e / F.n1 + 1, a.t_wall,
                      nu_h, nu_c, a.mode == 1 || a.mode == 5 ? (S *)B.base[a.parity ^ 1] : nullptr);
      }
    }
  }
  if (!reduce) return cav;  // walls only (a stored state's walls made explicit), no reductions
  if (!xwall) {  // only the x walls carry Nusselt sums (a CTA covers one face)
    if (tid == 0) {
      a.bc_partials[2LL * cta] = 0.0;
      a.bc_partials[2LL * cta + 1] = 0.0;
    }
    return cav;
  }
  // a CTA covers one face: the hot (low x) or the cold (high x) sum, the other is zero
  const double v = warp_sum(xhigh ? nu_c : nu_h);
  if ((tid & 31) == 0) sh[tid >> 5] = v;
  __syncthreads();
  if (tid == 0) {
    double t = 0;
    for (int q = 0; q < nwarps; ++q) t += sh[q];
    a.bc_partials[2LL * cta] = xhigh ? 0.0 : t;
    a.bc_partials[2LL * cta + 1] = xhigh ? t : 0.0;
  }
  return cav;
}

template <class S>
__global__ void __launch_bounds__(kBcThreads) k_bc(BcArgs a) {
  bc_cta<S>(a, blockIdx.x, a.mode != 3 && a.mode != 5);
}

// ---------------------------------------------------------------------------
// k_pack / k_unpack (Section 4.5, Listings 1-2, Optimized V3).  One thread per
// (ib, ic) face position; buffer layout p[(ic nb + ib) 2 + d], then
// var[2 nb nc + v nb nc + ic nb + ib].  Depth d counts layers in increasing
// index order.  Pure copies: bit exact.

__device__ __forceinline__ int find_cut(const CutFace *faces, int nfaces, int cta) {
  int lo = 0, hi = nfaces - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (faces[mid].cta_begin <= cta) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <class S>
__device__ __forceinline__ void face_geometry(const BlockDev &B, int face, int ib, int ic, bool ghost,
                                              long long &p_first, long long &v_node, long long &dstep) {
  // face axis a; the face's faster axis (y for x faces, else x) gets ib + 1,
  // the slower one (z, except y for z faces) ic + 1 (selects rather than an
  // indexed array, which would live in local memory)
  const int a = face >> 1, high = face & 1;
  const int na = a == 0 ? B.nx : (a == 1 ? B.ny : B.nz);
  const int b1 = ib + 1, c1 = ic + 1;
  int pl, vl;
  if (!ghost) { pl = high ? na - 1 : 1; vl = high ? na : 1; }
  else { pl = high ? na + 1 : -1; vl = high ? na + 1 : 0; }
  p_first = node_index<S>(B, a == 0 ? pl : b1, a == 0 ? b1 : (a == 1 ? pl : c1), a == 2 ? pl : c1);
  v_node = node_index<S>(B, a == 0 ? vl : b1, a == 0 ? b1 : (a == 1 ? vl : c1), a == 2 ? vl : c1);
  dstep = a == 0 ? 1 : (a == 1 ? (long long)B.pitch : B.plane);
}

template <class S>
__global__ void __launch_bounds__(256) k_pack(ExchArgs a) {
  const int fi = find_cut(a.faces, a.nfaces, blockIdx.x);
  const CutFace &F = a.faces[fi];
  const int e = (blockIdx.x - F.cta_begin) * 256 + threadIdx.x;
  const int plane = F.nb * F.nc;
  if (e >= plane) return;
  const int ib = e % F.nb, ic = e / F.nb;
  const BlockDev &B = a.blocks[F.src];
  const S *q = (const S *)B.base[a.parity];
  long long p_first, v_node, dstep;
  face_geometry<S>(B, F.face, ib, ic, false, p_first, v_node, dstep);
  S *buf = (S *)a.buf + F.buf_off;
  constexpr int NP = Store<S>::NP;  // pressure arrays (FP32-mixed: hi, then lo section)
  for (int pa = 0; pa < NP; ++pa) {
    const S *pq = q + (long long)pa * B.fstride;
    buf[2LL * pa * plane + 2LL * e] = pq[p_first];
    buf[2LL * pa * plane + 2LL * e + 1] = pq[p_first + dstep];
  }
  for (int v = 0; v < Store<S>::NA - NP; ++v)  // u, v, w, T (FP32-mixed: T_hi, T_lo)
    buf[2LL * NP * plane + (long long)v * plane + e] = q[(long long)(NP + v) * B.fstride + v_node];
}

template <class S>
__global__ void __launch_bounds__(256) k_unpack(ExchArgs a) {
  const int fi = find_cut(a.faces, a.nfaces, blockIdx.x);
  const CutFace &F = a.faces[fi];
  const int e = (blockIdx.x - F.cta_begin) * 256 + threadIdx.x;
  const int plane = F.nb * F.nc;
  if (e >= plane) return;
  const int ib = e % F.nb, ic = e / F.nb;
  const BlockDev &B = a.blocks[F.dst];
  S *q = (S *)B.base[a.parity];
  long long p_first, v_node, dstep;
  face_geometry<S>(B, F.face ^ 1, ib, ic, true, p_first, v_node, dstep);
  const S *buf = (const S *)a.buf + F.buf_off;
  constexpr int NP = Store<S>::NP;
  for (int pa = 0; pa < NP; ++pa) {
    S *pq = q + (long long)pa * B.fstride;
    pq[p_first] = buf[2LL * pa * plane + 2LL * e];
    pq[p_first + dstep] = buf[2LL * pa * plane + 2LL * e + 1];
  }
  for (int v = 0; v < Store<S>::NA - NP; ++v)
    q[(long long)(NP + v) * B.fstride + v_node] = buf[2LL * NP * plane + (long long)v * plane + e];
}

// The step's exchange, one CTA of NT threads per 256 face positions
// (CutFace::cta_begin counts such CTAs): the ghost values k_pack followed by
// k_unpack would write, copied straight from the sending block's layers (the
// face buffer is packed only when asked for, by cavity_get_face_buffer).  It
// stands between two steps, so it is written for latency: the face found by a
// warp-wide search, every value of the thread's positions loaded before the
// first store.
template <class S, int NT>
__device__ __forceinline__ void exchange_cta(const ExchArgs &a, int cta) {
  static_assert(256 % NT == 0, "positions per thread");
  constexpr int NPOS = 256 / NT, NP = Store<S>::NP, NA = Store<S>::NA, NV = NP + NA;  // p at depth 2
  // the face of this CTA: the last one whose first CTA is not after it
  int fi = 0;
  for (int base = 0; base < a.nfaces; base += 32) {
    const int l = base + (threadIdx.x & 31);
    const unsigned m = __ballot_sync(0xffffffffu, l < a.nfaces && a.faces[l].cta_begin <= cta);
    if (m) fi = base + 31 - __clz(m);
  }
  const CutFace F = a.faces[fi];
  const BlockDev &B = a.blocks[F.src];
  const BlockDev &D = a.blocks[F.dst];
  const int plane = F.nb * F.nc;
  const S *__restrict__ q = (const S *)B.base[a.parity];
  S *__restrict__ g = (S *)D.base[a.parity];
  const long long fs = B.fstride, fd = D.fstride;
  int e[NPOS];
  long long gp[NPOS], gv[NPOS], gstep = 0;
  S x[NPOS][NV];
#pragma unroll
  for (int r = 0; r < NPOS; ++r) {
    e[r] = (cta - F.cta_begin) * 256 + r * NT + (int)threadIdx.x;
    if (e[r] >= plane) continue;
    const int ib = e[r] % F.nb, ic = e[r] / F.nb;
    long long p_first, v_node, dstep;
    face_geometry<S>(B, F.face, ib, ic, false, p_first, v_node, dstep);
    face_geometry<S>(D, F.face ^ 1, ib, ic, true, gp[r], gv[r], gstep);
#pragma unroll
    for (int pa = 0; pa < NP; ++pa) {
      x[r][2 * pa] = q[pa * fs + p_first];
      x[r][2 * pa + 1] = q[pa * fs + p_first + dstep];
    }
#pragma unroll
    for (int v = 0; v < NA - NP; ++v) x[r][2 * NP + v] = q[(NP + v) * fs + v_node];
  }
#pragma unroll
  for (int r = 0; r < NPOS; ++r) {
    if (e[r] >= plane) continue;
#pragma unroll
    for (int pa = 0; pa < NP; ++pa) {
      g[pa * fd + gp[r]] = x[r][2 * pa];
      g[pa * fd + gp[r] + gstep] = x[r][2 * pa + 1];
    }
#pragma unroll
    for (int v = 0; v < NA - NP; ++v) g[(NP + v) * fd + gv[r]] = x[r][2 * NP + v];
  }
}

// Between two steps of a graph: what the next one waits for.  One CTA per cavity
// takes dt from the maximum and the centre shift from the new state (and clears
// the step's words); a.faces' CTAs exchange the cut faces; the rest (FP64,
// large cavities) store the new state's walls.  2 us for an undivided cavity
// (4-6 with an exchange or walls) where a finalise took 8-19.
//
// The one CTA lets the next step's launch start at once (the step before is
// complete by then: its tile look-ups and first plane loads run beside this),
// the others when they are done: CTAs of a step placed beside the exchange's
// are spread unevenly over the SMs (FP32-mixed 128^3 in 2x2x2 blocks 77 us a
// step, against 64).
constexpr int kBetweenThreads = 128;
template <class S>
__global__ void __launch_bounds__(kBetweenThreads) k_between(ExchArgs a, BcArgs b, int ncut) {
  chain_wait();
  if ((int)blockIdx.x >= b.ncav) {
    const int c = blockIdx.x - b.ncav;
    if (c < ncut) exchange_cta<S, kBetweenThreads>(a, c);
    else bc_cta<S>(b, c - ncut, false);
    return;
  }
  chain_trigger();
  __shared__ double shc[kMaxCentre];
  const CavConst &C = b.cc[blockIdx.x];
  CavState &st = b.cs[blockIdx.x];
  const int tid = threadIdx.x;
  if (tid < kMaxCentre) {
    double v = 0.0;
    if (tid < C.ncentre) {
      const BlockDev &B = a.blocks[C.centre_blk[tid]];
      v = load_p_l2<S>((const S *)B.base[a.parity], B.fstride, C.centre_off[tid]);
    }
    shc[tid] = v;
    __syncwarp(0xffu);
    if (tid == 0) st.c = centre_mean(C.ncentre, shc);
  }
  if (tid == 32) {
    const double t = __ldcg(&st.smax[b.slot]);
    const double dt = C.cfl / t;
    st.dt = dt;
    if (b.dt_out) *b.dt_out = dt;
    for (int q = 0; q < kStepSlots; ++q) {
      st.smax[q] = 0.0;
      st.sfl[q] = 0u;
      if (blockIdx.x == 0) b.tile_counter[q] = 0u;
    }
  }
}

// ---------------------------------------------------------------------------
// initial state, gather / scatter of the interior

// splitmix64 (Steele, Lea & Flood 2014): finaliser of state x + golden gamma
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

struct InitArgs {
  const BlockDev *blocks;
  const CavConst *cc;
  int block;
  int parity;
  unsigned long long seed;
  double noise;
  double t_hot, t_cold;
};

template <class S>
__global__ void k_init(InitArgs a) {
  const BlockDev &B = a.blocks[a.block];
  const long long n = (long long)B.nx * B.ny * B.nz;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int i = (int)(e % B.nx) + 1, j = (int)((e / B.nx) % B.ny) + 1, k = (int)(e / ((long long)B.nx * B.ny)) + 1;
  const CavConst &C = a.cc[B.cav];
  const int I = B.ox + i, J = B.oy + j, K = B.oz + k;
  const uint64_t gidx = (uint64_t)(I - 1) + (uint64_t)C.gn[0] * ((uint64_t)(J - 1) + (uint64_t)C.gn[1] * (uint64_t)(K - 1));
  const double U = (double)(splitmix64(a.seed * (1ULL << 40) + gidx) >> 11) * (1.0 / 9007199254740992.0);
  // explicit round-to-nearest operations (no contraction): the initial state is
  // reproducible bit for bit by any IEEE implementation of the same formula
  const double x = __dmul_rn((double)I, C.h[0]);
  const double lin = __dadd_rn(a.t_hot, __dmul_rn(__dsub_rn(a.t_cold, a.t_hot), x));
  const double pert = __dmul_rn(a.noise, __dsub_rn(__dmul_rn(2.0, U), 1.0));
  store_T<S>((S *)B.base[a.parity], B.fstride, node_index<S>(B, i, j, k), __dadd_rn(lin, pert));
}

// field f (0 = p, 1..4 = u, v, w, T) of node offset o, widened to FP64
template <class S>
__device__ __forceinline__ double get_field(const S *q, long long fs, int f, long long o) {
  if (f == 0) return load_p<S>(q, fs, o);
  if (f == 4) return load_T<S>(q, fs, o);
  return (double)q[(long long)(Store<S>::NP + f - 1) * fs + o];
}
template <class S>
__device__ __forceinline__ void put_field(S *q, long long fs, int f, long long o, double v) {
  if (f == 0) store_p<S>(q, fs, o, v);
  else if (f == 4) store_T<S>(q, fs, o, v);
  else q[(long long)(Store<S>::NP + f - 1) * fs + o] = (S)v;
}

struct MoveArgs {
  const BlockDev *blocks;
  int block;
  int parity;
  int mask;
  int gn[3];
  double *stage;       // [nf][gnz][gny][gnx] FP64, fields of the mask in order
  double pshift;       // subtracted from p on gather
};

template <class S>
__global__ void k_gather(MoveArgs a) {
  const BlockDev &B = a.blocks[a.block];
  const long long n = (long long)B.nx * B.ny * B.nz;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int i = (int)(e % B.nx) + 1, j = (int)((e / B.nx) % B.ny) + 1, k = (int)(e / ((long long)B.nx * B.ny)) + 1;
  const long long g = (long long)(B.ox + i - 1) + (long long)a.gn[0] * ((B.oy + j - 1) + (long long)a.gn[1] * (B.oz + k - 1));
  const long long gN = (long long)a.gn[0] * a.gn[1] * a.gn[2];
  const S *q = (const S *)B.base[a.parity];
  const long long o = node_index<S>(B, i, j, k);
  int slot = 0;
  for (int f = 0; f < kNF; ++f) {
    if (!(a.mask & (1 << f))) continue;
    double v = get_field<S>(q, B.fstride, f, o);
    if (f == 0) v -= a.pshift;
    a.stage[slot * gN + g] = v;
    ++slot;
  }
}

struct BoxArgs {
  const BlockDev *blocks;
  int nblocks;
  int parity;
  int mask;
  int i0, j0, k0, ni, nj, nk;  // global 1-based node box
  double *stage;               // [nf][nk][nj][ni]
  double pshift;
};

template <class S>
__global__ void k_gather_box(BoxArgs a) {
  const long long n = (long long)a.ni * a.nj * a.nk;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int I = a.i0 + (int)(e % a.ni), J = a.j0 + (int)((e / a.ni) % a.nj), K = a.k0 + (int)(e / ((long long)a.ni * a.nj));
  for (int b = 0; b < a.nblocks; ++b) {
    const BlockDev &B = a.blocks[b];
    if (I <= B.ox || I > B.ox + B.nx || J <= B.oy || J > B.oy + B.ny || K <= B.oz || K > B.oz + B.nz) continue;
    const S *q = (const S *)B.base[a.parity];
    const long long o = node_index<S>(B, I - B.ox, J - B.oy, K - B.oz);
    int slot = 0;
    for (int f = 0; f < kNF; ++f) {
      if (!(a.mask & (1 << f))) continue;
      double v = get_field<S>(q, B.fstride, f, o);
      if (f == 0) v -= a.pshift;
      a.stage[slot * n + e] = v;
      ++slot;
    }
    return;
  }
}

template <class S>
__global__ void k_scatter(MoveArgs a) {
  const BlockDev &B = a.blocks[a.block];
  const long long n = (long long)B.nx * B.ny * B.nz;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int i = (int)(e % B.nx) + 1, j = (int)((e / B.nx) % B.ny) + 1, k = (int)(e / ((long long)B.nx * B.ny)) + 1;
  const long long g = (long long)(B.ox + i - 1) + (long long)a.gn[0] * ((B.oy + j - 1) + (long long)a.gn[1] * (B.oz + k - 1));
  const long long gN = (long long)a.gn[0] * a.gn[1] * a.gn[2];
  S *q = (S *)B.base[a.parity];
  const long long o = node_index<S>(B, i, j, k);
  int slot = 0;
  for (int f = 0; f < kNF; ++f) {
    if (!(a.mask & (1 << f))) continue;
    put_field<S>(q, B.fstride, f, o, a.stage[slot * gN + g]);
    ++slot;
  }
}

// p of the stored state is p_true + c: fold a pending shift into the array
// (used before overwriting other fields from the host, so that c can be reset)
template <class S>
__global__ void k_shift_p(const BlockDev *blocks, int block, int parity, double c) {
  const BlockDev &B = blocks[block];
  const long long n = (long long)(B.nx + 4) * (B.ny + 4) * (B.nz + 4);
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int i = (int)(e % (B.nx + 4)) - 1, j = (int)((e / (B.nx + 4)) % (B.ny + 4)) - 1;
  const int k = (int)(e / ((long long)(B.nx + 4) * (B.ny + 4))) - 1;
  S *q = (S *)B.base[parity];
  const long long o = node_index<S>(B, i, j, k);
  store_p<S>(q, B.fstride, o, load_p<S>(q, B.fstride, o) - c);
}

// copy of one stored array of a block (walls and ghosts included) to a dense
// stage; `field` is the array index (FP32-mixed: 0 = p_hi, 1 = p_lo, 2.. = u..T)
template <class S>
__global__ void k_copy_block(const BlockDev *blocks, int block, int parity, int field, double *stage) {
  const BlockDev &B = blocks[block];
  const long long n = (long long)(B.nx + 4) * (B.ny + 4) * (B.nz + 4);
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int i = (int)(e % (B.nx + 4)) - 1, j = (int)((e / (B.nx + 4)) % (B.ny + 4)) - 1;
  const int k = (int)(e / ((long long)(B.nx + 4) * (B.ny + 4))) - 1;
  const S *q = (const S *)B.base[parity];
  stage[e] = (double)q[field * B.fstride + node_index<S>(B, i, j, k)];
}

}  // namespace bdc
