// Discrete adjoint of the explicit step (single-block cavity).
//
// Objective J = (1/N) sum_{n=1..N} Nu_hot(Q^n); controls: the hot-wall
// temperature field theta and Ra.  A step Q^{n+1} = G(Q^n) is: dt = cfl / S,
// S = max over nodes of the spectral bound of Q^n; Q~ = Q^n + dt R(Q^n)
// (Eqs. 1-3); p = p~ - mean of p~ over the centre nodes; walls formed from the
// new interior (Section 2) with the hot-wall temperature theta.  The reverse
// sweep over one step takes Y = dJ/dQ~ on the interior to dJ/dQ~ of the step
// before, in one launch of k_adj_sweep:
//   - at every interior node the reverse of the rates applied to dt Y, gathered:
//     each node sums what its stencil's nodes pass to it (no atomics);
//   - the wall and ghost adjoints moved onto interior nodes 1, 2 through p_w =
//     2 p1 - p2, p_g = 2 p_w - p1, T_w = (4 T1 - T2)/3, and the hot wall's T
//     onto theta, formed in place by the nodes next to a wall;
//   - the objective's terms of the state reversed to (T next to the hot wall);
//   - in the CTA that finishes last: dt's dependence, -cfl dtbar / S^2 times
//     the gradient of the spectral bound at its largest node (dtbar = sum Y R);
//     the Ra adjoint from the buoyancy (g sigma = Ra Pr) and floor (kappa
//     u_ref^2 = kappa Ra Pr) sums; and the centre shift's transpose, the sum
//     of the p adjoint shared over the centre nodes.
// The argmax of the bound depends on the forward state only and is taken for a
// whole recomputed segment in one launch (k_adj_argmax_seg): the FP32 bound
// f32_spectral_exact after an FP32-mixed forward, which sets that forward's dt.
// Subgradients at kinks follow the forward branch (|x| with sign(0) = 0, the
// beta^2 floor, the argmax node).
//
// Precision: the adjoint arrays X, Q hold the reverse sweep's type: FP64 after
// an FP64 forward, FP32 after an FP32-mixed forward, whose trajectory carries
// FP32 precision anyway.  The rates' reverse works on neighbour-minus-centre
// differences; for the FP32-mixed state the p and T differences are formed from
// their hi/lo pairs (as the forward step does), so FP32 arithmetic loses no
// cancellation.  The sums over nodes (dt, g sigma, beta^2 floor, the p adjoint)
// are compensated FP32 sums within a thread (FP64 after an FP64 forward) and
// FP64 from there on; the wall gradient stays FP64.
#pragma once

#include <type_traits>

#include "bdc_device.cuh"
#include "bdc_step_f32.cuh"

namespace bdc {

enum { kScRa = 0, kScCount = 1 };

// The adjoint arrays have the state's layout (node_index, fstride), five
// fields p, u, v, w, T; they are zero off the interior.
struct AdjArgs {
  BlockDev B;             // the state Q^n being reversed to (buffer set base[0], walls stored)
  CavConst C;
  const void *X;          // Y: adjoint of the interior state after the step, centre shift transposed
  void *Q;                // the same of the step before
  double *scal;           // kSc* scalars
  double *thetabar;       // ny*nz, (j-1) + ny (k-1)
  const double *argpart;  // (max, index) pairs of k_adj_argmax_seg for this state
  int nparts;
  double *gpart;          // [CTA][4]: sums of dtbar, g sigma bar, floor bar, p adjoint
  unsigned int *cnt;      // finished CTAs (zero between launches)
  const double *dt;       // dt of this step
  double coef;            // 1 / (N ny nz 2 h_x dT)
  double dfloor;          // d(beta^2 floor)/dRa
  int objective;          // Q^n counts in J
  int kc, tiles_x, tiles_y;
};

// arrays of the stored state: p (pair), u, v, w, T (pair)
template <class R> struct AdjState;
template <> struct AdjState<double> { static constexpr int U = 1, T = 4, PAIR = 0; };
template <> struct AdjState<float> { static constexpr int U = 2, T = 5, PAIR = 1; };

// 1 / sqrt(x) of a positive normal value: FP64 by two Newton steps on the
// reciprocal square root's approximation (rsqrt.approx.ftz.f64, relative error
// below 1e-6: 1.5 e^2 after a step)
__device__ __forceinline__ double rsqrt_r(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double hx = 0.5 * x;
  y = fma(y, fma(-hx * y, y, 0.5), y);
  return fma(y, fma(-hx * y, y, 0.5), y);
}
__device__ __forceinline__ float rsqrt_r(float x) { return vrsqrt(x); }
__device__ __forceinline__ double abs_r(double x) { return fabs(x); }
__device__ __forceinline__ float abs_r(float x) { return fabsf(x); }
// sign with sign(0) = 0
__device__ __forceinline__ double sign_r(double x) { return x == 0.0 ? 0.0 : copysign(1.0, x); }
__device__ __forceinline__ float sign_r(float x) { return x == 0.f ? 0.f : copysignf(1.f, x); }

// a hi/lo pair (FP64: a value), and neighbour minus centre
template <class R> struct Pair { R h, l; };
template <> struct Pair<double> { double h; };
__device__ __forceinline__ float pair_diff(const Pair<float> &a, const Pair<float> &c) { return (a.h - c.h) + (a.l - c.l); }
__device__ __forceinline__ double pair_diff(const Pair<double> &a, const Pair<double> &c) { return a.h - c.h; }
// A value of one plane of an array: a base that is the same for every thread
// (it moves up with the plane) and a thread's 32-bit byte offset inside the
// plane, so that a load needs no address arithmetic of its own.
template <class R>
__device__ __forceinline__ R at(const R *plane, unsigned off) {
  return *reinterpret_cast<const R *>(reinterpret_cast<const char *>(plane) + off);
}
__device__ __forceinline__ Pair<float> pair_at(const float *plane, long long fs, unsigned off) {
  return {at(plane, off), at(plane + fs, off)};
}
__device__ __forceinline__ Pair<double> pair_at(const double *plane, long long, unsigned off) { return {at(plane, off)}; }
__device__ __forceinline__ float pair_less(const Pair<float> &a, float t) { return (a.h - t) + a.l; }
__device__ __forceinline__ double pair_less(const Pair<double> &a, double t) { return a.h - t; }

// a thread's sum over its nodes: compensated in FP32, plain in FP64
template <class R> struct NodeSum;
template <> struct NodeSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ double total() const { return s; }
};
template <> struct NodeSum<float> {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b)));
    s = t;
  }
  __device__ __forceinline__ double total() const { return (double)s + (double)c; }
};

// constants in the sweep's type (FP32: rounded on the host)
template <class R> struct AdjK { R ih2[3], nh[3], ah[3], c4ih[3], b2min, gs, tinf; };
__device__ __forceinline__ AdjK<double> adj_consts(const CavConst &C, double) {
  AdjK<double> k;
  for (int d = 0; d < 3; ++d) {
    k.ih2[d] = C.ih2[d]; k.nh[d] = C.nuhh[d]; k.ah[d] = C.alhh[d]; k.c4ih[d] = C.c4 * C.ih[d];
  }
  k.b2min = C.b2min; k.gs = C.gs; k.tinf = C.t_inf;
  return k;
}
__device__ __forceinline__ AdjK<float> adj_consts(const CavConst &C, float) {
  AdjK<float> k;
  for (int d = 0; d < 3; ++d) {
    k.ih2[d] = C.fh2[d]; k.nh[d] = C.fnh[d]; k.ah[d] = C.fah[d]; k.c4ih[d] = C.fc4 * C.fih[d];
  }
  k.b2min = C.fb2min; k.gs = C.fgs; k.tinf = C.ftinf;
  return k;
}

// What one source node passes to its stencil: r = dt Y (p, u, v, w, T), a_d =
// V_d / (2 h_d), D_d = r_p c4 lambda_d / h_d, b = beta^2 r_p; and for its own
// terms beta^2, lambda_d and 1 / sqrt(V_d^2 + 4 beta^2).
template <class R>
struct AdjCoef {
  R r[5], a[3], D[3], b, b2, lam[3], isq[3];
  bool floored;
};
// lambda_d without 1 / sqrt: the square root is no FP64-pipe operation (sqrt_newton)
__device__ __forceinline__ double lambda_r(double V, double q) { return 0.5 * (fabs(V) + sqrt_newton(q)); }
__device__ __forceinline__ float lambda_r(float V, float q) { return 0.5f * (fabsf(V) + q * rsqrt_r(q)); }
// (D0: the first axis wanted; 2 for a plane that only passes z terms.  OWN: isq
// is wanted)
template <int D0, bool OWN, class R>
__device__ __forceinline__ void adj_coef(const AdjK<R> &K, const R V[3], const R y[5], R dt, AdjCoef<R> &c) {
  R b2 = V[0] * V[0] + V[1] * V[1] + V[2] * V[2];
  c.floored = b2 < K.b2min;
  if (c.floored) b2 = K.b2min;
  c.b2 = b2;
#pragma unroll
  for (int f = 0; f < 5; ++f) c.r[f] = dt * y[f];
  c.b = b2 * c.r[0];
#pragma unroll
  for (int d = D0; d < 3; ++d) {
    const R q = V[d] * V[d] + (R)4 * b2;
    if (OWN) {
      c.isq[d] = rsqrt_r(q);
      c.lam[d] = (R)0.5 * (abs_r(V[d]) + q * c.isq[d]);
    } else {
      c.lam[d] = lambda_r(V[d], q);
    }
    c.a[d] = V[d] * K.ih2[d];
    c.D[d] = c.r[0] * K.c4ih[d] * c.lam[d];
  }
}

// D_z alone: all that the outermost plane at either end of a chunk passes on.  FP64
// only, where its 12 FP64 operations instead of 70 count (32^3 51 -> 46 us a reverse
// step with the halo's square roots, 48^3 131 -> 124); the branch costs the FP32
// sweep its schedule (128^3 110 -> 127).
template <class R>
__device__ __forceinline__ R adj_dz(const AdjK<R> &K, const R V[3], R y0, R dt) {
  R b2 = V[0] * V[0] + V[1] * V[1] + V[2] * V[2];
  if (b2 < K.b2min) b2 = K.b2min;
  return dt * y0 * K.c4ih[2] * lambda_r(V[2], V[2] * V[2] + (R)4 * b2);
}

// ---------------------------------------------------------------------------
// The reverse of one step.  A CTA of 32 x TY columns sweeps a chunk of planes
// upwards.  Each node's outgoing coefficients are formed once per plane: a
// thread adds its own to the accumulators of the planes below and above in its
// column (registers), and passes nine of them to its x and y neighbours through
// shared memory (two buffers, one barrier a plane; the tile's halo nodes are
// formed by the first 4 (32 + TY) threads).  The p accumulators span planes k-2
// .. k+2 of the source plane k, the others k-1 .. k+1; plane k's p is complete
// after plane k+2, so a chunk sweeps two planes more at either end, z terms only.
//
// Why: a gather that recomputed the coefficients of all twelve sources at every
// node (one thread a node, no sweep) was bound by its 1560 instructions a node
// (68% of the issue slots, DRAM at 14%): 131 us at 128^3, with a p-sum kernel
// (12 us), a one-CTA dt kernel (21 us) and a wall fold (5 us) around it.  The
// FP64 form scattered with 41 atomics a node between six small kernels.
constexpr int kAdjTY = 8;
template <class R, int TY>
__host__ __device__ constexpr size_t adj_smem_bytes() { return 2 * 9 * 36 * (TY + 4) * sizeof(R); }

template <class R, int TY>
__global__ void __launch_bounds__(32 * TY, sizeof(R) == 4 ? 2 : 1) k_adj_sweep(const __grid_constant__ AdjArgs a) {
  constexpr int NT = 32 * TY, W = 36, PN = W * (TY + 4);
  constexpr int U = AdjState<R>::U, T0 = AdjState<R>::T;
  enum { R1, R2, R3, R4, AX, AY, DX, DY, BB, NQ };
  extern __shared__ __align__(16) unsigned char adj_smem[];  // [2][NQ][PN]
  static_assert(2 * NQ * PN * sizeof(R) == adj_smem_bytes<R, TY>(), "");
  chain_wait();
  const BlockDev &B = a.B;
  const AdjK<R> K = adj_consts(a.C, R(0));
  const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
  const int tx = blockIdx.x % a.tiles_x, tq = blockIdx.x / a.tiles_x, ty = tq % a.tiles_y, tz = tq / a.tiles_y;
  const int nx = B.nx, ny = B.ny, nz = B.nz;
  const int i0 = tx * 32 + 1, j0 = ty * TY + 1, k0 = tz * a.kc + 1, k1 = min(k0 + a.kc - 1, nz);
  const int i = i0 + lane, j = j0 + wy;
  const bool act = i <= nx && j <= ny;
  const R *q = (const R *)B.base[0];
  const R *Y = (const R *)a.X;
  R *Q = (R *)a.Q;
  const long long fs = B.fstride, pl = B.plane;
  constexpr unsigned E = sizeof(R);
  const unsigned pt = E * B.pitch;  // bytes
  const R dt = (R)*a.dt;
  const R coef = (R)a.coef;
  // the thread's halo node: x halo (4 columns x TY rows), then y halo (4 rows x 32)
  int hpos = -1, hi = 0, hj = 0;
  {
    const int t = threadIdx.x;
    if (t < 4 * TY) {
      const int c = t & 3, r = t >> 2;
      hi = i0 + (c < 2 ? c - 2 : 30 + c);
      hj = j0 + r;
    } else if (t < 4 * TY + 128) {
      const int r = (t - 4 * TY) >> 5;
      hi = i0 + lane;
      hj = j0 + (r < 2 ? r - 2 : TY - 2 + r);
    }
    if (t < 4 * TY + 128) hpos = (hj - j0 + 2) * W + (hi - i0 + 2);
  }
  static_assert(NT >= 4 * TY + 128, "one halo node a thread");
  // (sources on or beyond a wall pass nothing)
  const bool hin = hpos >= 0 && hi >= 1 && hi <= nx && hj >= 1 && hj <= ny;
  const int ic = min(i, nx), jc = min(j, ny);
  // byte offsets inside a plane: the thread's node, its halo node (a plane has under 2^32 bytes)
  const unsigned o = E * (unsigned)(XO<R>::v - 1 + ic + B.pitch * (jc + 1));
  const unsigned ho = hin ? E * (unsigned)(XO<R>::v - 1 + hi + B.pitch * (hj + 1)) : o;
  const R *qk = q + pl * (k0 - 1), *Yk = Y + pl * (k0 - 1);  // plane k - 1 of node index k - 2
  R *Qk = Q + pl * (k0 - 1);
  const int pos = (wy + 2) * W + lane + 2;
  // the column's state: p at planes k-2 .. k+2, u, v, w, T at k-1 .. k+1
  Pair<R> pz[5], tz3[3];
  R vz[3][3];
  pz[2] = pz[3] = pz[4] = Pair<R>{};
  pz[0] = pz[1] = Pair<R>{};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    vz[d][0] = 0;
    vz[d][1] = 0;
    vz[d][2] = at(qk + (U + d) * fs, o);
  }
  tz3[0] = tz3[1] = Pair<R>{};
  tz3[2] = pair_at(qk + T0 * fs, fs, o);
  pz[3] = pair_at(qk, fs, o);
  pz[4] = pair_at(qk + pl, fs, o);
  R P[5] = {0, 0, 0, 0, 0}, F[4][3];
#pragma unroll
  for (int f = 0; f < 4; ++f) F[f][0] = F[f][1] = F[f][2] = 0;
  NodeSum<R> sdt, sgs, sfl, sp;
  const R third = (R)(1.0 / 3.0);
  // the next plane's adjoint and the next plane's halo node, loaded a plane ahead
  R yn[5], hV[3] = {0, 0, 0}, hy[5] = {0, 0, 0, 0, 0};
#pragma unroll
  for (int f = 0; f < 5; ++f) yn[f] = act ? at(Yk + f * fs, o) : (R)0;
  if (hin) {
#pragma unroll
    for (int d = 0; d < 3; ++d) hV[d] = at(qk + 2 * pl + (U + d) * fs, ho);
#pragma unroll
    for (int f = 0; f < 5; ++f) hy[f] = at(Yk + 2 * pl + f * fs, ho);
  }

  for (int k = k0 - 2; k <= k1 + 2; ++k, qk += pl, Yk += pl, Qk += pl) {
    // move the column's queues one plane up
    pz[0] = pz[1]; pz[1] = pz[2]; pz[2] = pz[3]; pz[3] = pz[4];
    tz3[0] = tz3[1]; tz3[1] = tz3[2];
#pragma unroll
    for (int d = 0; d < 3; ++d) { vz[d][0] = vz[d][1]; vz[d][1] = vz[d][2]; }
    if (k <= k1) {
      pz[4] = pair_at(qk + 2 * pl, fs, o);
      tz3[2] = pair_at(qk + pl + T0 * fs, fs, o);
    }
    if (k <= k1 + 1) {
#pragma unroll
      for (int d = 0; d < 3; ++d) vz[d][2] = at(qk + pl + (U + d) * fs, o);
    }
    const bool full = k >= k0 && k <= k1;  // uniform
    const bool outer = sizeof(R) == 8 && (k == k0 - 2 || k == k1 + 2);
    const R V[3] = {vz[0][1], vz[1][1], vz[2][1]};
    R y[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      y[f] = yn[f];
      yn[f] = act && k <= k1 + 1 ? at(Yk + pl + f * fs, o) : (R)0;  // (zero off the interior)
    }
    AdjCoef<R> c;
    if (full) adj_coef<0, true>(K, V, y, dt, c);
    else if (!outer) adj_coef<2, false>(K, V, y, dt, c);
    // z: to the planes below (s = 1) and above (s = -1)
    if (outer) {  // two planes off the chunk: the fourth difference's outer weight alone
      const R D = adj_dz(K, V, y[0], dt);
      if (k < k0) P[4] -= D;
      else P[0] -= D;
    } else {
      const R wm = K.nh[2] + c.a[2], wp = K.nh[2] - c.a[2], tm = K.ah[2] + c.a[2], tp = K.ah[2] - c.a[2];
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        F[f][0] += c.r[1 + f] * wm;
        F[f][2] += c.r[1 + f] * wp;
      }
      const R tlo = c.r[4] * tm, thi = c.r[4] * tp;  // T to planes k-1, k+1
      F[3][0] += tlo;
      F[3][2] += thi;
      F[2][0] += K.ih2[2] * c.b;
      F[2][2] -= K.ih2[2] * c.b;
      const R g = c.r[3] * K.ih2[2], D = c.D[2];
      P[1] += (R)4 * D + g;
      P[3] += (R)4 * D - g;
      P[0] -= D;
      P[4] -= D;
      // what plane 1 passes to the wall and ghost below, and so on, moved onto
      // the two planes they are formed from
      if (k <= 2) {
        if (k == 1) {
          P[2] += (R)2 * g + (R)5 * D;
          P[3] -= g + (R)2 * D;
          F[3][1] += (R)4 * third * tlo;
          F[3][2] -= third * tlo;
        } else if (k == 2) {
          P[1] -= (R)2 * D;
          P[2] += D;
        }
      }
      if (k >= nz - 1) {
        if (k == nz) {
          P[2] += (R)5 * D - (R)2 * g;
          P[1] += g - (R)2 * D;
          F[3][1] += (R)4 * third * thi;
          F[3][0] -= third * thi;
        } else if (k == nz - 1) {
          P[3] -= (R)2 * D;
          P[2] += D;
        }
      }
    }
    if (full) {
      R(*s)[PN] = reinterpret_cast<R(*)[PN]>(adj_smem) + ((k - k0) & 1) * NQ;
      s[R1][pos] = c.r[1]; s[R2][pos] = c.r[2]; s[R3][pos] = c.r[3]; s[R4][pos] = c.r[4];
      s[AX][pos] = c.a[0]; s[AY][pos] = c.a[1]; s[DX][pos] = c.D[0]; s[DY][pos] = c.D[1]; s[BB][pos] = c.b;
      if (hpos >= 0) {
        AdjCoef<R> h;
        adj_coef<0, false>(K, hV, hy, dt, h);
        s[R1][hpos] = h.r[1]; s[R2][hpos] = h.r[2]; s[R3][hpos] = h.r[3]; s[R4][hpos] = h.r[4];
        s[AX][hpos] = h.a[0]; s[AY][hpos] = h.a[1]; s[DX][hpos] = h.D[0]; s[DY][hpos] = h.D[1]; s[BB][hpos] = h.b;
        if (hin && k < k1) {
#pragma unroll
          for (int d = 0; d < 3; ++d) hV[d] = at(qk + pl + (U + d) * fs, ho);
#pragma unroll
          for (int f = 0; f < 5; ++f) hy[f] = at(Yk + pl + f * fs, ho);
        }
      }
      // the node's own terms, before the neighbours' coefficients are needed
      if (act) {
        const Pair<R> p0 = pz[2], t0 = tz3[1];
        R dp[5][3], dm[5][3], d4[3];
        {
          const R px1 = pair_diff(pair_at(qk, fs, o + E), p0), pxm = pair_diff(pair_at(qk, fs, o - E), p0);
          const R py1 = pair_diff(pair_at(qk, fs, o + pt), p0), pym = pair_diff(pair_at(qk, fs, o - pt), p0);
          const R pz1 = pair_diff(pz[3], p0), pzm = pair_diff(pz[1], p0);
          dp[0][0] = px1; dm[0][0] = pxm; dp[0][1] = py1; dm[0][1] = pym; dp[0][2] = pz1; dm[0][2] = pzm;
          d4[0] = (pair_diff(pair_at(qk, fs, o + 2 * E), p0) + pair_diff(pair_at(qk, fs, o - 2 * E), p0)) - (R)4 * (px1 + pxm);
          d4[1] = (pair_diff(pair_at(qk, fs, o + 2 * pt), p0) + pair_diff(pair_at(qk, fs, o - 2 * pt), p0)) - (R)4 * (py1 + pym);
          d4[2] = (pair_diff(pz[4], p0) + pair_diff(pz[0], p0)) - (R)4 * (pz1 + pzm);
        }
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const R *v = qk + (U + f) * fs;
          dp[1 + f][0] = at(v, o + E) - V[f]; dm[1 + f][0] = at(v, o - E) - V[f];
          dp[1 + f][1] = at(v, o + pt) - V[f]; dm[1 + f][1] = at(v, o - pt) - V[f];
          dp[1 + f][2] = vz[f][2] - V[f]; dm[1 + f][2] = vz[f][0] - V[f];
        }
        {
          const R *t = qk + T0 * fs;
          dp[4][0] = pair_diff(pair_at(t, fs, o + E), t0); dm[4][0] = pair_diff(pair_at(t, fs, o - E), t0);
          dp[4][1] = pair_diff(pair_at(t, fs, o + pt), t0); dm[4][1] = pair_diff(pair_at(t, fs, o - pt), t0);
          dp[4][2] = pair_diff(tz3[2], t0); dm[4][2] = pair_diff(tz3[0], t0);
        }
        const R tb = pair_less(t0, K.tinf);
        R divV = 0, diss = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          divV += (dp[1 + d][d] - dm[1 + d][d]) * K.ih2[d];
          diss += K.c4ih[d] * c.lam[d] * d4[d];
        }
        // forward rates (for dt's adjoint: dtbar = sum Y R) and the transported fields' own adjoint
        R dtb = y[0] * (-c.b2 * divV - diss);
        R abar[3] = {0, 0, 0};
        const R nsum = (R)2 * (K.nh[0] + K.nh[1] + K.nh[2]), asum = (R)2 * (K.ah[0] + K.ah[1] + K.ah[2]);
#pragma unroll
        for (int f = 1; f <= 4; ++f) {
          R r = 0;
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const R dh = f == 4 ? K.ah[d] : K.nh[d], df = dp[f][d] - dm[f][d];
            r += dh * (dp[f][d] + dm[f][d]) - c.a[d] * df;
            abar[d] -= c.r[f] * df;
          }
          if (f <= 3) {
            r -= (dp[0][f - 1] - dm[0][f - 1]) * K.ih2[f - 1];
            if (f - 1 == a.C.gaxis) r += K.gs * tb;
          }
          dtb += y[f] * r;
          F[f - 1][1] += y[f] - c.r[f] * (f == 4 ? asum : nsum);
        }
        sdt.add(dtb);
        const R rg = a.C.gaxis == 1 ? c.r[2] : c.r[3];
        F[3][1] += K.gs * rg;
        sgs.add(tb * rg);
        // continuity: R_p = -beta^2 div V - dissipation
        R b2bar = -divV * c.r[0], p6 = 0;
        R vb[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const R lambar = -c.r[0] * K.c4ih[d] * d4[d];
          p6 += c.D[d];
          vb[d] = abar[d] * K.ih2[d] + lambar * (R)0.5 * (sign_r(V[d]) + V[d] * c.isq[d]);
          b2bar += lambar * c.isq[d];
        }
        P[2] += y[0] - (R)6 * p6;
        if (c.floored) sfl.add(b2bar);
#pragma unroll
        for (int d = 0; d < 3; ++d) F[d][1] += c.floored ? vb[d] : vb[d] + (R)2 * V[d] * b2bar;
      }
      __syncthreads();
      if (act) {
#define BDC_ADJ_SIDE(off, sg, A_, D_, d, rg)                                                    \
  {                                                                                            \
    const R ad = (sg) * s[A_][pos + (off)], w = K.nh[d] + ad, wt = K.ah[d] + ad;                \
    F[0][1] += s[R1][pos + (off)] * w;                                                          \
    F[1][1] += s[R2][pos + (off)] * w;                                                          \
    F[2][1] += s[R3][pos + (off)] * w;                                                          \
    F[3][1] += s[R4][pos + (off)] * wt;                                                         \
    F[d][1] += ((sg) * K.ih2[d]) * s[BB][pos + (off)];                                          \
    P[2] += ((sg) * K.ih2[d]) * s[rg][pos + (off)] + (R)4 * s[D_][pos + (off)] - s[D_][pos + 2 * (off)]; \
  }
        BDC_ADJ_SIDE(1, (R)1, AX, DX, 0, R1)
        BDC_ADJ_SIDE(-1, (R)-1, AX, DX, 0, R1)
        BDC_ADJ_SIDE(W, (R)1, AY, DY, 1, R2)
        BDC_ADJ_SIDE(-W, (R)-1, AY, DY, 1, R2)
#undef BDC_ADJ_SIDE
        // the x and y walls' and ghosts' adjoints (as for z above)
        if (i <= 2 || i >= nx - 1) {
          if (i == 1) {
            P[2] += (R)2 * K.ih2[0] * c.r[1] + (R)5 * c.D[0] - (R)2 * s[DX][pos + 1];
            double *th = a.thetabar + (j - 1) + (long long)ny * (k - 1);
            *th += (double)(c.r[4] * (K.ah[0] + c.a[0])) + (a.objective ? 3.0 * a.coef : 0.0);
          }
          if (i == 2) P[2] += c.D[0] - K.ih2[0] * s[R1][pos - 1] - (R)2 * s[DX][pos - 1];
          if (i == nx) P[2] += (R)5 * c.D[0] - (R)2 * K.ih2[0] * c.r[1] - (R)2 * s[DX][pos - 1];
          if (i == nx - 1) P[2] += c.D[0] + K.ih2[0] * s[R1][pos + 1] - (R)2 * s[DX][pos + 1];
          if (a.objective) {  // Nu_hot of the state reversed to
            if (i == 1) F[3][1] -= (R)4 * coef;
            if (i == 2) F[3][1] += coef;
          }
        }
        if (j <= 2 || j >= ny - 1) {
          if (j == 1) {
            P[2] += (R)2 * K.ih2[1] * c.r[2] + (R)5 * c.D[1] - (R)2 * s[DY][pos + W];
            F[3][1] += (R)4 * third * (c.r[4] * (K.ah[1] + c.a[1]));
          }
          if (j == 2) {
            P[2] += c.D[1] - K.ih2[1] * s[R2][pos - W] - (R)2 * s[DY][pos - W];
            F[3][1] -= third * (s[R4][pos - W] * (K.ah[1] + s[AY][pos - W]));
          }
          if (j == ny) {
            P[2] += (R)5 * c.D[1] - (R)2 * K.ih2[1] * c.r[2] - (R)2 * s[DY][pos - W];
            F[3][1] += (R)4 * third * (c.r[4] * (K.ah[1] - c.a[1]));
          }
          if (j == ny - 1) {
            P[2] += c.D[1] + K.ih2[1] * s[R2][pos + W] - (R)2 * s[DY][pos + W];
            F[3][1] -= third * (s[R4][pos + W] * (K.ah[1] - s[AY][pos + W]));
          }
        }
      }
    }
    // planes k - 1 (u, v, w, T) and k - 2 (p) are complete
    if (act && k - 1 >= k0 && k - 1 <= k1) {
#pragma unroll
      for (int f = 0; f < 4; ++f) *reinterpret_cast<R *>(reinterpret_cast<char *>(Qk - pl + (1 + f) * fs) + o) = F[f][0];
    }
    if (act && k - 2 >= k0) {
      *reinterpret_cast<R *>(reinterpret_cast<char *>(Qk - 2 * pl) + o) = P[0];
      sp.add(P[0]);
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) { F[f][0] = F[f][1]; F[f][1] = F[f][2]; F[f][2] = 0; }
    P[0] = P[1]; P[1] = P[2]; P[2] = P[3]; P[3] = P[4]; P[4] = 0;
  }

  // the CTA's node sums, in a fixed order: transposed through shared memory
  // (the sweep's, which is done with), field f summed by the 16 threads 16 f ..
  // 16 f + 15, so that 20 FP64 warp instructions do what a shuffle tree in every
  // warp takes 160 for
  double(*red)[NT] = reinterpret_cast<double(*)[NT]>(adj_smem);
  static_assert(adj_smem_bytes<R, TY>() >= 4 * NT * sizeof(double), "the sums inside the sweep's shared memory");
  const int tid = threadIdx.x, f4 = tid >> 4, l4 = tid & 15;
  __shared__ double sg[4], sb[TY], si[TY];
  __shared__ bool last;
  auto fold4 = [&]() {  // totals of red[0..3][0..NT-1], in threads 16 f .. 16 f + 15 (f < 4)
    double v = 0.0;
    if (f4 < 4) {
      const double *r = &red[f4][l4];
#pragma unroll
      for (int n = 0; n < NT / 16; ++n) v += r[16 * n];
#pragma unroll
      for (int of = 1; of < 16; of <<= 1) v += __shfl_xor_sync(0xffffffffu, v, of);
    }
    return v;
  };
  __syncthreads();
  red[0][tid] = sdt.total(); red[1][tid] = sgs.total(); red[2][tid] = sfl.total(); red[3][tid] = sp.total();
  __syncthreads();
  {
    const double v = fold4();
    if (f4 < 4 && l4 == 0) a.gpart[4 * (long long)blockIdx.x + f4] = v;
  }
  __threadfence();  // (and this CTA's Q, before the last one adds to it)
  __syncthreads();
  if (tid == 0) last = atomicAdd(a.cnt, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  // the last CTA: the sums of all CTAs (thread t takes field t & 3 of CTAs t / 4,
  // t / 4 + NT / 4, ..) and the argmax of the spectral bound (largest value,
  // smallest index among equals), in fixed orders
  {
    double v = 0.0;
    for (int n = tid; n < 4 * (int)gridDim.x; n += NT) v += __ldcg(&a.gpart[n]);
    // (into red as a row per field, the unused places zero)
    for (int e = 0; e < 4; ++e) red[e][tid] = (tid & 3) == e ? v : 0.0;
  }
  double best = -1.0, bidx = 0.0;
  for (int n = tid; n < a.nparts; n += NT) {
    const double v = a.argpart[2 * n], ix = a.argpart[2 * n + 1];
    if (v > best || (v == best && ix < bidx)) { best = v; bidx = ix; }
  }
  for (int of = 16; of > 0; of >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, of), oi = __shfl_xor_sync(0xffffffffu, bidx, of);
    if (ob > best || (ob == best && oi < bidx)) { best = ob; bidx = oi; }
  }
  if (lane == 0) {
    sb[wy] = best;
    si[wy] = bidx;
  }
  __syncthreads();
  const double tot = fold4();
  if (f4 < 4 && l4 == 0) sg[f4] = tot;
  // dt = cfl / S: (-cfl dtbar / S^2) d(bound)/dV at the argmax node, an axis a
  // thread (threads 64, 65, 66); what does not need the sums first
  const int d = tid - 64;
  double gV = 0.0, gb = 0.0, V3[3] = {0.0, 0.0, 0.0};
  bool floored = false;
  long long on = 0;
  if (d >= 0 && d < 3) {
    double S = sb[0], ix = si[0];
    for (int w = 1; w < TY; ++w)
      if (sb[w] > S || (sb[w] == S && si[w] < ix)) { S = sb[w]; ix = si[w]; }
    const long long e = (long long)ix;
    on = node_index<R>(B, (int)(e % nx) + 1, (int)((e / nx) % ny) + 1, (int)(e / ((long long)nx * ny)) + 1);
    for (int x = 0; x < 3; ++x) V3[x] = (double)q[(U + x) * fs + on];
    double b2 = V3[0] * V3[0] + V3[1] * V3[1] + V3[2] * V3[2];
    floored = b2 < a.C.b2min;
    if (floored) b2 = a.C.b2min;
    const double V = d == 0 ? V3[0] : d == 1 ? V3[1] : V3[2], ih = d == 0 ? a.C.ih[0] : d == 1 ? a.C.ih[1] : a.C.ih[2];
    const double isq = rsqrt_r(V * V + 4.0 * b2), k = -a.C.cfl * ih / (S * S);  // per dtbar
    gV = 0.5 * k * (sign_r(V) + V * isq);
    gb = k * isq;
  }
  __syncthreads();
  if (tid < a.C.ncentre) {
    // the centre shift's transpose (at most 8 nodes)
    R *e = Q + a.C.centre_off[tid];
    *e = (R)((double)__ldcg(e) - sg[3] / (double)a.C.ncentre);
  }
  if (d >= 0 && d < 3) {
    const double dtbar = sg[0];
    const double b2bar = dtbar * (__shfl_sync(7u, gb, 0) + __shfl_sync(7u, gb, 1) + __shfl_sync(7u, gb, 2));
    const double V = d == 0 ? V3[0] : d == 1 ? V3[1] : V3[2];
    R *x = Q + (1 + d) * fs + on;
    *x = (R)(__ldcg(x) + (R)(dtbar * gV + (floored ? 0.0 : 2.0 * V * b2bar)));
    if (d == 0) {
      // the step's Ra adjoint from the buoyancy (g sigma = Ra Pr) and floor
      // (kappa u_ref^2 = kappa Ra Pr) sums
      a.scal[kScRa] += a.C.nu * sg[1] + a.dfloor * (sg[2] + (floored ? b2bar : 0.0));
      *a.cnt = 0u;
    }
  }
}

// Before the first reverse step: the objective's terms of the final state (the
// p adjoint is zero: nothing for the centre shift).
template <class R>
__global__ void k_adj_start(AdjArgs a) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x, ny = a.B.ny;
  if (e >= ny * a.B.nz) return;
  R *x = (R *)a.Q + 4 * a.B.fstride + node_index<R>(a.B, 1, e % ny + 1, e / ny + 1);
  x[0] = (R)(-4.0 * a.coef);
  x[1] = (R)a.coef;
  a.thetabar[e] = 3.0 * a.coef;
}

// Largest spectral bound of the state in buffer set 0 of block B and its
// node (smallest linear index among equal values: each thread visits its
// nodes in increasing index), over the rows of CTA `cta` of `ncta`; thread 0
// writes (max, index) to out2.  Every thread of the CTA calls it.
template <class S>
__device__ __forceinline__ void adj_argmax_part(const BlockDev &B, const CavConst &C, const int n[3], int cta, int ncta,
                                                double *out2) {
  // a warp per interior row (j, k), strided over the grid's warps (no index
  // division); a thread visits its nodes in increasing linear interior index
  // e = (i - 1) + nx ((j - 1) + ny (k - 1)), so it keeps the first of equal values
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5, nwq = blockDim.x >> 5;
  const int nx = n[0], ny = n[1], rows = ny * n[2];
  const S *q = (const S *)B.base[0];
  const long long fs = B.fstride;
  constexpr int NP = Store<S>::NP;  // u, v, w follow the p array(s)
  double best = -1.0, bidx = 0.0;
  float bestf = -1.f;               // FP32 path: the running maximum in FP32
  long long bidxl = 0;
  float wfloor = 0.f;  // FP64 path: at or below an exact bound a lane of this warp reached
  const F32K<float> K32 = f32_spectral_consts(C);
  for (int r = cta * nwq + wq; r < rows; r += ncta * nwq) {
    const long long o0 = node_index<S>(B, 0, r % ny + 1, r / ny + 1), e0 = (long long)nx * r - 1;
    for (int i = 1 + lane; i <= nx; i += 32) {
      const long long o = o0 + i;
      const S u = q[NP * fs + o], v = q[(NP + 1) * fs + o], w = q[(NP + 2) * fs + o];
      if constexpr (std::is_same<S, float>::value) {
        // the FP32-mixed step sets dt from the FP32 bound f32_spectral_exact
        // (also its initial dt): the argmax of that same value, at every node
        const float sv = f32_spectral_exact(K32, u, v, w);
        if (sv > bestf) {
          bestf = sv;
          bidxl = e0 + i;
        }
      } else {
        if (__fmul_rn(spectral_est_f32(C, u, v, w), 1.00001f) >= wfloor) {
          // exact FP64 bound only where an FP32 estimate (relative error < 1e-6)
          // raised by 1e-5 could reach the running maximum: the argmax is unchanged
          const double sv = spectral_f64(C, u, v, w);
          if (sv > best) {
            best = sv;
            bidx = (double)(e0 + i);
          }
        }
        // a warp-shared floor (a value some lane's node attained exactly), so that
        // the FP64 path runs only when a node of the warp could reach it:
        // non-negative floats order like their bit patterns
        const float bf = best > 0.0 ? __double2float_rd(best) : 0.f;
        wfloor = fmaxf(wfloor, __uint_as_float(__reduce_max_sync(__activemask(), __float_as_uint(bf))));
      }
    }
  }
  if constexpr (std::is_same<S, float>::value) {
    if (bestf >= 0.f) {
      best = (double)bestf;
      bidx = (double)bidxl;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o), oi = __shfl_xor_sync(0xffffffffu, bidx, o);
    if (ob > best || (ob == best && oi < bidx)) { best = ob; bidx = oi; }
  }
  __shared__ double sb[8], si[8];
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) { sb[w] = best; si[w] = bidx; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < (int)(blockDim.x >> 5); ++q)
      if (sb[q] > best || (sb[q] == best && si[q] < bidx)) { best = sb[q]; bidx = si[q]; }
    out2[0] = best;
    out2[1] = bidx;
  }
}

// The argmax of every state of a recomputed segment (it depends on the
// forward state only): grid (parts, slots), slot s's state in buffer set 0 of
// blocks[s]; (max, index) pairs at argpart[2 (s parts + part)].
template <class S>
__global__ void __launch_bounds__(256) k_adj_argmax_seg(const BlockDev *blocks, CavConst C,
                                                         double *argpart) {
  adj_argmax_part<S>(blocks[blockIdx.y], C, C.gn, blockIdx.x, gridDim.x,
                     argpart + 2 * ((long long)blockIdx.y * gridDim.x + blockIdx.x));
}

}  // namespace bdc
