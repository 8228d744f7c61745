// Element-tile DD sweep (Algorithm 1) with the wave state in registers: a
// thread owns one element column and H elements above each other (P columns
// by H*P rows of nodes), so the position of every node inside its element,
// and with it every stiffness coefficient, is known at compile time.
//
// Layout.  Thread (bx, by) of the subdomain's grid of LX x NB tiles owns the
// nodes of columns P bx .. P bx + P - 1 and rows H P by .. H P (by + 1) - 1.
// With H = 2 (FP32) the rows r and r + P of the two elements share their
// coefficients and sit in one float2, so every update is one packed two-lane
// FMA (__ffma2_rn).  The subdomain's last column (chain A, sye elements and
// the corner) and last row (chain B, sxe elements) are 1D chains: lane e of a
// chain owns the P nodes of its element.
//
// Stiffness apply, (A p) / (Wx Wy) = (Kx p) / Wx + (Ky p) / Wy:
//   inside a tile from registers, P + 1 taps per node; a node shared by two
//   elements (a = 0) takes from the element before it one partial sum
//     T = sum_{b < P} Kref[P][b] p_b / (2 w_0),
//   formed by that element's owner from its own nodes alone (the b = P term
//   stays with the node), and the owner needs one value, the p of the next
//   element's first node.  So neighbours exchange two numbers per row (x) or
//   column (y) of a tile and time step, both known as soon as p is updated:
//   one exchange and one barrier per step.  x neighbours are lanes of one
//   warp (shuffles); y neighbours and the chains exchange through shared
//   memory, double-buffered by step parity.  At the subdomain's ends the
//   partial sum is the node's own (the one-element row is twice the
//   two-element one, diagonal apart).
//
// FUSE: the whole subdomain is one warp (or part of one: small subdomains
// share a warp), which also runs the chains; the barrier is __syncwarp.
// Otherwise the chains have warps of their own, and subdomains whose state
// exceeds one SM's registers take a thread-block cluster, each CTA a slab of
// bands, whose end warps exchange with the neighbouring slabs' through
// distributed shared memory (st.async with mbarriers).
//
// Bound: the FMA pipe at 19 FMAs per node and step (P = 3); what keeps it from
// there is the chains (a sixth of a fused warp's instructions, on half of its
// lanes) and the few warps that the registers leave room for (1.7 per
// scheduler at 1024 one-warp subdomains).  Measured, 20 WaveHoltz iterations:
// 1024 subdomains of 25 x 25 nodes, P = 3, N_t = 55: 1073 us with the one-warp
// column kernel (hz_sweep_warp.cuh: 4 shuffles and 30 instructions per node row
// and step), 570 us here; 16 of 17 x 17, P = 2, N_t = 79: 610, 157 us; 1024 of
// 129 x 129, P = 4, N_t = 48: 59.8 ms with the cluster of warp bands, 108.6 ms
// with the cluster kernel, 20.7 ms here.  A launch with clusters is a separate
// instantiation: its few branches per step alone cost the others 20 to 40%.
//
// Taken by size (tile_shape, tile_default in hz_sweep_tile_dispatch.cu):
// sxe <= 32 and sye <= 32 elements, fixed WaveHoltz count or per-subdomain
// tolerance, zero interface boundary mass (eta = 0), cold start.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "hz_complex_io.cuh"
#include "hz_gll_const.h"
#include "hz_internal.h"
#include "hz_norm_acc.cuh"

namespace hz {
namespace tile_sweep {

namespace cg = cooperative_groups;

// ---- reference rows: c[0][b], b = 1..P: Kref[0][b] / (2 w_0) (shared node,
// own element; by symmetry also T's coefficients, c[0][P - b] for node b);
// c[0][0]: Kref[0][0] / w_0; c[a][b], 0 < a < P: Kref[a][b] / w_a.
//
// Rounding them to FP32 one by one leaves a row sum of about one unit in the
// last place of the diagonal, which every time step applies to a smooth p with
// the same sign: on the 1024^2 workload's 129 x 129-node subdomains (P = 4)
// the sweep's error was 6.4e-6, with the rows below it is 8e-7.  The off-diagonal entries are therefore
// rounded to one of their three to nine nearest values so that the diagonal, minus
// their sum, is representable (the row annihilates constants), and among
// those choices so that the second moments, weighted over the element's rows,
// cancel (that is the relative error of the wave number, equal at every node)
// with the first moments small.
// FP64 rows are rounded one by one: against long double, 10 WaveHoltz iterations
// on 25 x 25 nodes (P = 3, N_t = 55) are off by 1.7e-15 to 2e-15, by 4.3e-15 to
// 5.6e-15 when Kref and the weights are applied one after the other, and by 3e-15
// to 4e-15 with the diagonal as minus the sum.
template <typename Real>
struct TileRows {
  Real c[kMaxP][kMaxP + 1][kMaxP + 1] = {};
};
HZ_HD constexpr double ulp32(double v) {
  v = gllc::cabs(v);
  double u = 1.0;
  while (u > v) u *= 0.5;
  while (2.0 * u <= v) u *= 2.0;
  return u / 8388608.0;  // 2^-23
}
template <typename Real>
HZ_HD constexpr TileRows<Real> make_tile_rows() {
  TileRows<Real> r{};
  for (int P = 1; P <= 5; ++P) {
    const gllc::Gll g = gllc::make_gll(P);
    double total = 0.0;  // second moments of the rows so far
    for (int a = 0; a < P; ++a) {
      if (sizeof(Real) == 4 && 2 * a > P) break;  // the mirrored rows follow below
      double v[kMaxP + 1] = {};
      for (int b = 0; b <= P; ++b) v[b] = g.K[a * (P + 1) + b] / g.w[a] * (a == 0 && b > 0 ? 0.5 : 1.0);
      if (sizeof(Real) == 8) {
        for (int b = 0; b <= P; ++b) r.c[P - 1][a][b] = (Real)v[b];
        continue;
      }
      const double copies = a == 0 ? 2.0 : 1.0;  // a shared node has its row's off-diagonals on both sides
      const double weight = (a == 0 || 2 * a < P ? 2.0 : 1.0) * g.w[a];  // of the row and its mirror image
      double best = -1.0, moment = 0.0;
      const int tries = P == 5 ? 3 : P == 4 && a == 0 ? 9 : 5;
      int combos = 1;
      for (int b = 0; b < P; ++b) combos *= tries;
      for (int m = 0; m < combos; ++m) {
        double c[kMaxP + 1] = {};
        double sum = 0.0, m1 = 0.0, m2 = 0.0;
        int k = m;
        for (int b = 0; b <= P; ++b) {
          if (b == a) continue;
          c[b] = (double)(float)v[b] + (k % tries - tries / 2) * ulp32(v[b]);
          k /= tries;
          const double d = g.x[b] - g.x[a];
          sum += copies * c[b];
          m1 += (a == 0 ? 0.0 : (c[b] - v[b]) * d);
          m2 += copies * (c[b] - v[b]) * d * d;
        }
        c[a] = (double)(float)(-sum);
        const double cost = 1e6 * gllc::cabs(c[a] + sum) + 0.1 * gllc::cabs(m1) + gllc::cabs(total + weight * m2);
        if (best < 0.0 || cost < best) {
          best = cost;
          moment = weight * m2;
          for (int b = 0; b <= P; ++b) r.c[P - 1][a][b] = (Real)c[b];
        }
      }
      total += moment;
    }
    // the mirrored rows with the same values
    if (sizeof(Real) == 4)
      for (int a = P / 2 + 1; a < P; ++a)
        for (int b = 0; b <= P; ++b) r.c[P - 1][a][b] = r.c[P - 1][P - a][P - b];
  }
  return r;
}
static __constant__ TileRows<float> kTileRowsF = make_tile_rows<float>();
static __constant__ TileRows<double> kTileRowsD = make_tile_rows<double>();

// ---- the register type: Real, or float2 holding a row of each of two elements
template <typename Real, int H>
struct VecT;
template <>
struct VecT<float, 1> {
  using V = float;
  using Tab = float4;
};
template <>
struct VecT<float, 2> {
  using V = float2;
  using Tab = float4;
};
struct alignas(32) Quad64 {
  double x, y, z, w;
};
template <>
struct VecT<double, 1> {
  using V = double;
  using Tab = Quad64;
};
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
template <typename V, typename Real>
__device__ __forceinline__ V bc(Real x) {
  if constexpr (sizeof(V) == sizeof(Real)) return x;
  else return make_float2(x, x);
}
__device__ __forceinline__ float lo(float v) { return v; }
__device__ __forceinline__ float hi(float v) { return v; }
__device__ __forceinline__ double lo(double v) { return v; }
__device__ __forceinline__ double hi(double v) { return v; }
__device__ __forceinline__ float lo(float2 v) { return v.x; }
__device__ __forceinline__ float hi(float2 v) { return v.y; }
template <int H, typename V, typename Real>
__device__ __forceinline__ V half_of(Real l, Real h) {  // H = 2: (l, h)
  if constexpr (H == 2) return make_float2(l, h);
  else return l;
}
template <int H, typename V>
__device__ __forceinline__ auto get(V v, int h) {
  if constexpr (H == 2) return h ? v.y : v.x;
  else return v;
}
template <int H, typename V, typename Real>
__device__ __forceinline__ void put_half(V& v, int h, Real x) {
  if constexpr (H == 2) {
    if (h) v.y = x;
    else v.x = x;
  } else {
    v = x;
  }
}
__device__ __forceinline__ float shfl_down1(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double shfl_down1(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float2 shfl_down1(float2 v) {
  return make_float2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ float shfl_up1(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double shfl_up1(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float2 shfl_up1(float2 v) {
  return make_float2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}

// Coefficient (a, b) of an element's row: a constant-bank operand for scalar
// types; packed ones sit in registers, mirrored (c[a][b] = c[P-a][P-b]) so
// that only the first half of the rows is kept.
template <typename V, typename Real, int P>
struct Coef {
  static constexpr bool kPacked = sizeof(V) != sizeof(Real);
  V k[kPacked ? P / 2 + 1 : 1][kPacked ? P + 1 : 1];
  static __device__ __forceinline__ Real c(int a, int b) {
    if constexpr (sizeof(Real) == 8) return kTileRowsD.c[P - 1][a][b];
    else return kTileRowsF.c[P - 1][a][b];
  }
  __device__ __forceinline__ void init() {
    if constexpr (kPacked) {
#pragma unroll
      for (int a = 0; a <= P / 2; ++a)
#pragma unroll
        for (int b = 0; b <= P; ++b) k[a][b] = bc<V>(c(a < P ? a : 0, b));
    }
  }
  __device__ __forceinline__ V at(int a, int b) const {  // 0 < a < P
    if constexpr (kPacked) {
      return 2 * a > P ? k[P - a][P - b] : k[a][b];
    } else {
      return c(a, b);
    }
  }
  __device__ __forceinline__ V k0(int b) const {
    if constexpr (kPacked) return k[0][b];
    else return c(0, b);
  }
  __device__ __forceinline__ V diag() const { return k0(0); }            // shared node, both elements
  __device__ __forceinline__ V own(int b) const { return k0(b); }       // b = 1..P
  __device__ __forceinline__ V hand(int b) const { return k0(P - b); }  // T, b = 0..P-1
};

// A buffer of n elements' P values each, as planes of vector accesses (quads,
// then a pair, then a single; P = 3 floats: a padded quad), so that an
// element's nodes move in one or two shared-memory instructions.
template <int P, typename Real>
struct RowBuf;
// Shared-memory stores under a condition that never become branches: kernels of
// several warps (the compiler's own choice costs 64 subdomains of 97 x 97 nodes,
// P = 3, 218 us against 202; one-warp kernels schedule better with it).
__device__ __forceinline__ unsigned smem_addr(const void* q) { return (unsigned)__cvta_generic_to_shared(q); }
__device__ __forceinline__ void st_if(bool on, unsigned addr, float a) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.shared.f32 [%1], %2; }" ::"r"((unsigned)on), "r"(addr), "f"(a)
               : "memory");
}
__device__ __forceinline__ void st_if(bool on, unsigned addr, float a, float b) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.shared.v2.f32 [%1], {%2, %3}; }" ::"r"((unsigned)on),
               "r"(addr), "f"(a), "f"(b)
               : "memory");
}
__device__ __forceinline__ void st_if(bool on, unsigned addr, float a, float b, float c, float d) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.shared.v4.f32 [%1], {%2, %3, %4, %5}; }" ::"r"((unsigned)on),
               "r"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}
__device__ __forceinline__ void st_if(bool on, unsigned addr, double a) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.shared.f64 [%1], %2; }" ::"r"((unsigned)on), "r"(addr), "d"(a)
               : "memory");
}
__device__ __forceinline__ void st_if(bool on, unsigned addr, double a, double b) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.shared.v2.f64 [%1], {%2, %3}; }" ::"r"((unsigned)on),
               "r"(addr), "d"(a), "d"(b)
               : "memory");
}
template <int P>
struct RowBuf<P, float> {
  static constexpr int kQ = P / 4 + (P % 4 == 3 ? 1 : 0);  // quads
  static constexpr bool kP2 = P % 4 == 2, kP1 = P % 4 == 1;
  __host__ __device__ static constexpr int size(int n) { return 4 * kQ * n + ((kP2 ? 2 : kP1 ? 1 : 0) * n + 3) / 4 * 4; }
  static __device__ __forceinline__ float at(const float (&v)[P], int k) { return k < P ? v[k < P ? k : 0] : 0.f; }
  static __device__ __forceinline__ void st(float* buf, int n, int idx, const float (&v)[P]) {
#pragma unroll
    for (int f = 0; f < kQ; ++f)
      reinterpret_cast<float4*>(buf)[f * n + idx] =
          make_float4(at(v, 4 * f), at(v, 4 * f + 1), at(v, 4 * f + 2), at(v, 4 * f + 3));
    if (kP2) reinterpret_cast<float2*>(buf + 4 * kQ * n)[idx] = make_float2(at(v, 4 * kQ), at(v, 4 * kQ + 1));
    if (kP1) buf[4 * kQ * n + idx] = at(v, 4 * kQ);
  }
  template <bool PRED>
  static __device__ __forceinline__ void st(bool on, float* buf, int n, int idx, const float (&v)[P]) {
    if constexpr (!PRED) {
      if (on) st(buf, n, idx, v);
      return;
    }
    const unsigned b = smem_addr(buf);
#pragma unroll
    for (int f = 0; f < kQ; ++f)
      st_if(on, b + 16 * (f * n + idx), at(v, 4 * f), at(v, 4 * f + 1), at(v, 4 * f + 2), at(v, 4 * f + 3));
    if (kP2) st_if(on, b + 16 * kQ * n + 8 * idx, at(v, 4 * kQ), at(v, 4 * kQ + 1));
    if (kP1) st_if(on, b + 16 * kQ * n + 4 * idx, at(v, 4 * kQ));
  }
  static __device__ __forceinline__ void ld(const float* buf, int n, int idx, float (&v)[P]) {
#pragma unroll
    for (int f = 0; f < kQ; ++f) {
      const float4 t = reinterpret_cast<const float4*>(buf)[f * n + idx];
      const float u[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * f + k < P) v[4 * f + k < P ? 4 * f + k : 0] = u[k];
    }
    if (kP2) {
      const float2 t = reinterpret_cast<const float2*>(buf + 4 * kQ * n)[idx];
      v[4 * kQ < P ? 4 * kQ : 0] = t.x;
      v[4 * kQ + 1 < P ? 4 * kQ + 1 : 0] = t.y;
    }
    if (kP1) v[4 * kQ < P ? 4 * kQ : 0] = buf[4 * kQ * n + idx];
  }
  static __device__ __forceinline__ float* first(float* buf, int idx) { return buf + (kQ ? 4 : kP2 ? 2 : 1) * idx; }
  // the same store into another CTA's buffer, signalled to its mbarrier
  static constexpr int kBytes = 16 * kQ + (kP2 ? 8 : kP1 ? 4 : 0);
  static __device__ __forceinline__ void st_async(unsigned buf, int n, int idx, const float (&v)[P], unsigned mb) {
#pragma unroll
    for (int f = 0; f < kQ; ++f)
      asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                       buf + 16 * (f * n + idx)),
                   "f"(at(v, 4 * f)), "f"(at(v, 4 * f + 1)), "f"(at(v, 4 * f + 2)), "f"(at(v, 4 * f + 3)), "r"(mb)
                   : "memory");
    if (kP2)
      asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(
                       buf + 16 * kQ * n + 8 * idx),
                   "f"(at(v, 4 * kQ)), "f"(at(v, 4 * kQ + 1)), "r"(mb)
                   : "memory");
    if (kP1) st_async1(buf + 16 * kQ * n + 4 * idx, at(v, 4 * kQ), mb);
  }
  static __device__ __forceinline__ void st_async1(unsigned addr, float v, unsigned mb) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(addr), "f"(v), "r"(mb)
                 : "memory");
  }
};
template <int P>
struct RowBuf<P, double> {
  static constexpr int kD = P / 2;  // pairs
  __host__ __device__ static constexpr int size(int n) { return (2 * kD * n + (P % 2) * n + 3) / 4 * 4; }
  static __device__ __forceinline__ void st(double* buf, int n, int idx, const double (&v)[P]) {
#pragma unroll
    for (int f = 0; f < kD; ++f) reinterpret_cast<double2*>(buf)[f * n + idx] = make_double2(v[2 * f], v[2 * f + 1]);
    if (P % 2) buf[2 * kD * n + idx] = v[P - 1];
  }
  template <bool PRED>
  static __device__ __forceinline__ void st(bool on, double* buf, int n, int idx, const double (&v)[P]) {
    if constexpr (!PRED) {
      if (on) st(buf, n, idx, v);
      return;
    }
    const unsigned b = smem_addr(buf);
#pragma unroll
    for (int f = 0; f < kD; ++f) st_if(on, b + 16 * (f * n + idx), v[2 * f], v[2 * f + 1]);
    if (P % 2) st_if(on, b + 16 * kD * n + 8 * idx, v[P - 1]);
  }
  static __device__ __forceinline__ void ld(const double* buf, int n, int idx, double (&v)[P]) {
#pragma unroll
    for (int f = 0; f < kD; ++f) {
      const double2 t = reinterpret_cast<const double2*>(buf)[f * n + idx];
      v[2 * f] = t.x;
      v[2 * f + 1] = t.y;
    }
    if (P % 2) v[P - 1] = buf[2 * kD * n + idx];
  }
  static __device__ __forceinline__ double* first(double* buf, int idx) { return buf + (kD ? 2 : 1) * idx; }
  static constexpr int kBytes = 8 * P;
  static __device__ __forceinline__ void st_async(unsigned buf, int n, int idx, const double (&v)[P], unsigned mb) {
#pragma unroll
    for (int f = 0; f < kD; ++f)
      asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(
                       buf + 16 * (f * n + idx)),
                   "d"(v[2 * f]), "d"(v[2 * f + 1]), "r"(mb)
                   : "memory");
    if (P % 2) st_async1(buf + 16 * kD * n + 8 * idx, v[P - 1], mb);
  }
  static __device__ __forceinline__ void st_async1(unsigned addr, double v, unsigned mb) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(addr), "d"(v), "r"(mb)
                 : "memory");
  }
};

// p and p-dot of a node, and its two filter sums: for FP32 scalars each pair
// sits in one 64-bit register pair, so that both sums take one packed FMA.
template <typename V>
struct Pair {
  V a, b;
};
template <>
struct alignas(8) Pair<float> {
  float a, b;
};
__device__ __forceinline__ void accumulate(Pair<float>& v, float ka, float kb, const Pair<float>& s) {
  const float2 r = __ffma2_rn(make_float2(ka, kb), make_float2(s.a, s.b), make_float2(v.a, v.b));
  v.a = r.x;
  v.b = r.y;
}
template <typename V>
__device__ __forceinline__ void accumulate(Pair<V>& v, V ka, V kb, const Pair<V>& s) {
  v.a = vfma(ka, s.a, v.a);
  v.b = vfma(kb, s.b, v.b);
}

// beta f of a tile's node (real and imaginary part), one vector access.
template <typename V>
struct alignas(2 * sizeof(V)) SrcPair {
  V re, im;
};

// Shared memory of one subdomain slab (a CTA, or a lane group of a fused
// warp), in units of Real from a 16-byte aligned base.
struct Lay {
  int row;          // length of a row buffer over the LX tiles
  int col;          // length of a column buffer over the slab's elements and the node after them
  int py, ty;       // [2][nb + 1][row]: p of each band's first row; T handed into it
  int cp, ta;       // [2][col]: p of chain A; T of the last tiles
  int tax;          // [2]: T handed into the slab's first chain A node
  int tw, ts;       // edge tables: west column [rows][4], south row [cols][4]: alpha - 1, beta b (re, im)
  int src;          // source: [P P][threads] SrcPair
  int stash;        // previous iterate (tolerance mode)
  int total;
};
template <int P, typename Real>
__host__ __device__ inline Lay make_lay(int H, int LX, int nb, int threads, bool src, bool tol) {
  Lay y;
  y.row = RowBuf<P, Real>::size(LX);
  y.col = RowBuf<P, Real>::size(nb * H + 1);
  int o = 0;
  y.py = o; o += 2 * (nb + 1) * y.row;
  y.ty = o; o += 2 * (nb + 1) * y.row;
  y.cp = o; o += 2 * y.col;
  y.ta = o; o += 2 * y.col;
  y.tax = o; o += 4;
  y.tw = o; o += 4 * (nb * H * P + 1);
  y.ts = o; o += 4 * (LX * P + 1);
  o = (o + 3) / 4 * 4;
  y.src = o;
  if (src) o += threads * 2 * P * P * H;
  y.stash = o;
  if (tol) o += threads * 2 * (P * P * H + P + 1);
  y.total = (o + 3) / 4 * 4;
  return y;
}

struct TileArgs {
  SweepArgs base;
  int count;      // subdomains of the launch
  int LX, lxs;    // tiles in x (a power of two), its log2
  int nb, nbt;    // bands per CTA (slab), bands of the subdomain
  int spw, gs;    // FUSE: subdomains per warp, lanes per subdomain
  int wm;         // main warps (not FUSE)
  int offB;       // first edge lane of chain B
  int mute;       // clusters (tests): 1: the second slab's first row goes nowhere
  double wx[kMaxP], wy[kMaxP];  // lumped weight of node a (a = 0: shared by two elements)
};

// What a warp runs: the tiles, the chains, or both (one-warp subdomains).
// The roles are separate instantiations, so that neither carries the other's
// registers; they meet at the same barriers.
enum Role { kBoth = 0, kTiles = 1, kChains = 2 };

struct TolShared {
  unsigned long long mbar[2][2][4];  // clusters: arrivals by step parity; the same, seen by nobody
  // tolerance mode: per-warp and per-CTA partial norms, the decision
  double red[32][2];
  double part[2];
  int stop;
  int gave_up;  // clusters: a wait for a neighbouring slab's data ran out
};

// ---- exchange between the slabs of a cluster.  A cluster barrier per step
// costs every warp a release fence and the wait for the slowest CTA; here only
// the warps at a slab's ends wait, for the bytes that the neighbouring slab
// stores straight into their buffers (st.async counts them on an mbarrier,
// where the sender has announced them):
// 144 subdomains of 129 x 129 nodes, P = 4: 754 us with a cluster barrier per
// step (arrival and wait apart), 652 us; 9 of 97 x 97, P = 3: 140, 103 us.
// Barriers by step parity and by what arrives: a row of T (from the slab
// before), a row of p (from the one after), chain A's T and p.
enum { kTilePrev = 0, kTileNext = 1, kChainPrev = 2, kChainNext = 3 };
__device__ __forceinline__ unsigned peer_addr(unsigned addr, int rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_init(unsigned mb) { asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory"); }
// The sender announces its bytes on the neighbour's barrier, which is the
// barrier's one arrival of the step.  (The receiver may not: once it stops
// waiting it would arrive on a barrier whose phase has not ended.)  Relaxed:
// the bytes order themselves, a release here costs 60%.
__device__ __forceinline__ void mbar_expect(bool on, unsigned mb, unsigned bytes) {
  asm volatile(
      "{ .reg .pred q; setp.ne.u32 q, %0, 0; @q mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%1], %2; }" ::"r"(
          (unsigned)on),
      "r"(mb), "r"(bytes)
      : "memory");
}
// Waits for the phase; false after about a second and kLateLooks more looks
// (the clock also runs while the slabs are not scheduled).  The caller then
// stops waiting and the sweep's results are void: a slab that never answers
// must not hang the device.
constexpr int kLateLooks = 64;
__device__ __forceinline__ bool mbar_wait(unsigned mb, unsigned phase) {
  const long long t0 = clock64();
  int late = 0;
  do {
    unsigned ok;
    asm volatile(
        "{ .reg .pred q; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 q, [%1], %2; selp.u32 %0, 1, 0, q; }"
        : "=r"(ok)
        : "r"(mb), "r"(phase)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > 2000000000LL) ++late;
  } while (late < kLateLooks);
  return false;
}

// Block barrier met by warps at different places of the program (the roles).
__device__ __forceinline__ void block_bar() { asm volatile("bar.sync 0;" ::: "memory"); }

template <typename Real, int P, int H, int ROLE, bool SHARED, bool SRC, bool ISO, bool CLUS, bool TOL>
__device__ __forceinline__ void tile_body(const TileArgs& x, unsigned char* smem_raw, TolShared* ts) {
  constexpr bool FUSE = ROLE == kBoth, MAIN = ROLE != kChains, CHAIN = ROLE != kTiles;
  using V = typename VecT<Real, H>::V;
  using Tab = typename VecT<Real, H>::Tab;
  constexpr int RH = H * P;  // node rows of a tile
  const SweepArgs& a = x.base;
  cg::cluster_group cluster = cg::this_cluster();
  const int CL = CLUS ? (int)cluster.num_blocks() : 1;
  const int rk = CLUS ? (int)cluster.block_rank() : 0;
  const bool firstC = !CLUS || rk == 0, lastC = !CLUS || rk == CL - 1;
  const int LX = x.LX;
  const int lane = threadIdx.x & 31;
  const int grp = FUSE ? lane / x.gs : 0;
  const int k0 = FUSE ? blockIdx.x * x.spw + grp : blockIdx.x / CL;
  const bool have = grp < (FUSE ? x.spw : 1) && k0 < x.count;
  const int l = sweep_subdomain(a, have ? k0 : 0);
  const int sxi = l % a.Sx, syi = l / a.Sx;
  const int nlx = a.nlx, nly = a.nly, sxe = a.sxe;
  const int band0 = rk * x.nb;                                   // first band of the slab
  const int nb = (x.nbt - band0 < x.nb) ? x.nbt - band0 : x.nb;  // its bands
  const int row0 = band0 * RH;                                   // its first node row
  const int nA = nb * H;                                         // its chain A elements
  const int t = FUSE ? lane - grp * x.gs : (int)threadIdx.x;     // lane of the subdomain's tile grid
  const int nthr = FUSE ? x.gs : (int)blockDim.x;                // threads of this subdomain (slab)
  const int bx = t & (LX - 1), by = t >> x.lxs;
  const bool live = MAIN && have && bx < sxe && by < nb;
  const int byc = live ? by : 0;
  const int e = FUSE ? t : (int)threadIdx.x - 32 * x.wm;  // edge lane
  const bool inA = CHAIN && have && e < nA;
  const bool inB = CHAIN && have && lastC && e >= x.offB && e < x.offB + sxe;
  const bool inE = inA || inB;
  const int eB = inB ? e - x.offB : 0, eA = inA ? e : 0;
  const bool corner = inA && lastC && e == nA - 1;

  using RB = RowBuf<P, Real>;
  const bool tol = TOL && a.wh_tol > 0.0;
  const Lay y = make_lay<P, Real>(H, LX, x.nb, nthr, SRC, tol);
  const int ncol = x.nb * H + 1;  // elements of a column buffer
  Real* sm = reinterpret_cast<Real*>(smem_raw) + (FUSE ? grp * y.total : 0);
  const int64_t nn = (int64_t)nlx * nly;
  const Real* betaG = static_cast<const Real*>(a.beta) + (int64_t)l * nn;
  const Real* alphaG = static_cast<const Real*>(a.alpha) + (int64_t)l * nn;
  const double* lamL = a.lam_in + (int64_t)l * 4 * a.NE * 2;
  const double* kedgeL = a.kedge + (int64_t)l * 4 * a.NE;
  const bool ifW = sxi > 0, ifE = sxi < a.Sx - 1, ifS = syi > 0, ifN = syi < a.Sy - 1;
  const double sxs = 4.0 * (1.0 / ((2.0 * a.hx2) * (2.0 * a.hx2)));  // 4 / hx^2

  // right-hand side of node (i, j): split source and incoming lambda
  auto node_b = [&](int i, int j, double& br, double& bi) {
    br = bi = 0.0;
    if (SRC) {
      const double shx = ((i == 0 && ifW) || (i == nlx - 1 && ifE)) ? 0.5 : 1.0;
      const double shy = ((j == 0 && ifS) || (j == nly - 1 && ifN)) ? 0.5 : 1.0;
      const int64_t I = (int64_t)sxi * a.snxP + i, J = (int64_t)syi * a.snyP + j;
      const double2 s = load_complex(a.rhs, J * a.NXg + I);
      br = shx * shy * s.x;
      bi = shx * shy * s.y;
    }
    auto add = [&](double w, int ed, int q) {
      br += w * lamL[2 * (ed * a.NE + q)];
      bi += w * lamL[2 * (ed * a.NE + q) + 1];
    };
    if (i == 0 && ifW) add(a.wys[j], 0, j);
    if (i == nlx - 1 && ifE) add(a.wys[j], 1, j);
    if (j == 0 && ifS) add(a.wxs[i], 2, i);
    if (j == nly - 1 && ifN) add(a.wxs[i], 3, i);
  };

  // the exchange buffers start at zero: entries that nobody writes (before the
  // first band, of tiles past the subdomain) are read and multiplied by zero
  for (int q = t; q < y.tw; q += nthr) sm[q] = Real(0);

  // ---- edge tables: the west column's rows and the south row's columns,
  // one node per thread (alpha - 1 and beta b: a source enters there too)
  if (have) {
    for (int q = t; q < nb * RH + (firstC ? sxe * P : 0); q += nthr) {
      const bool west = q < nb * RH;
      const int i = west ? 0 : q - nb * RH, j = west ? row0 + q : 0;
      const int64_t n = (int64_t)j * nlx + i;
      const double be = (double)betaG[n];
      double br, bi;
      node_b(i, j, br, bi);
      Real* dst = sm + (west ? y.tw + 4 * q : y.ts + 4 * i);
      dst[0] = (Real)((double)alphaG[n] - 1.0);
      dst[1] = (Real)(be * br);
      dst[2] = (Real)(be * bi);
    }
  }

  // ---- tile coefficients: -beta' = -beta Wx Wy (4 / hx^2)
  // and with a source beta f of every node, which the time loop reads from
  // shared memory: in registers the paired tiles spilled (25 x 25 nodes, P = 3,
  // 1024 subdomains, 5 WaveHoltz iterations: 163 us, 134 us from shared memory)
  V nbet[P][P];
  SrcPair<V>* srcT = reinterpret_cast<SrcPair<V>*>(sm + y.src) + t;  // [P P][threads]
#pragma unroll
  for (int r = 0; r < P; ++r)
#pragma unroll
    for (int c = 0; c < P; ++c) {
      nbet[r][c] = bc<V>(Real(0));
      SrcPair<V> f{bc<V>(Real(0)), bc<V>(Real(0))};
#pragma unroll
      for (int h = 0; h < H; ++h) {
        if (live) {
          const int i = bx * P + c, j = row0 + by * RH + h * P + r;
          // the subdomain's first column and row have half the shared weight
          const double wx = (c == 0 && bx == 0) ? 0.5 * x.wx[0] : x.wx[c];
          const double wy = (r == 0 && j == 0) ? 0.5 * x.wy[0] : x.wy[r];
          const double be = (double)betaG[(int64_t)j * nlx + i];
          put_half<H>(nbet[r][c], h, (Real)(-be * wx * wy * sxs));
          if (SRC && i > 0 && j > 0) {  // first column and row: in the tables
            const int64_t I = (int64_t)sxi * a.snxP + i, J = (int64_t)syi * a.snyP + j;
            const double2 s = load_complex(a.rhs, J * a.NXg + I);
            put_half<H>(f.re, h, (Real)(be * s.x));
            put_half<H>(f.im, h, (Real)(be * s.y));
          }
        }
      }
      if (SRC && MAIN) srcT[(r * P + c) * nthr] = f;
    }

  // ---- chain nodes (index P: the corner, on chain A's last lane)
  Real ebet[P + 1], eal[P + 1], ebr[P + 1], ebi[P + 1];
#pragma unroll
  for (int q = 0; q <= P; ++q) {
    ebet[q] = eal[q] = ebr[q] = ebi[q] = Real(0);
    if (q < P ? inE : corner) {
      const int i = inA ? nlx - 1 : eB * P + q, j = inA ? row0 + e * P + q : nly - 1;
      const int ci = inA ? 0 : q, cj = inA ? q % P : 0;
      const double wx = (inA || i == 0) ? 0.5 * x.wx[0] : x.wx[ci];
      const double wy = (inB || j == 0 || q == P) ? 0.5 * x.wy[0] : x.wy[cj];
      const int64_t n = (int64_t)j * nlx + i;
      const double be = (double)betaG[n];
      double br, bi;
      node_b(i, j, br, bi);
      ebet[q] = (Real)(-be * wx * wy * sxs);
      eal[q] = alphaG[n];
      ebr[q] = (Real)(be * br);
      ebi[q] = (Real)(be * bi);
    }
  }
  unsigned mb0 = 0, mbP = 0, mbN = 0, smP = 0, smN = 0;  // this slab's barriers; the neighbours' barriers and buffers
  if constexpr (CLUS) {
    mb0 = smem_addr(ts->mbar);
    if (threadIdx.x == 0) {
      ts->gave_up = 0;
      for (int k = 0; k < 16; ++k) mbar_init(mb0 + 8 * k);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (!firstC) {
      mbP = peer_addr(mb0, rk - 1);
      smP = peer_addr(smem_addr(sm), rk - 1);
      if (MAIN && x.mute && rk == 1) {  // tests: the second slab's first row goes nowhere
        mbP = mb0 + 64;
        smP = smem_addr(sm);
      }
    }
    if (!lastC) {
      mbN = peer_addr(mb0, rk + 1);
      smN = peer_addr(smem_addr(sm), rk + 1);
    }
  }
  if (CLUS) cluster.sync();  // every CTA's buffers and barriers are ready before a neighbour uses them
  else if (FUSE) __syncwarp();
  else block_bar();

  Coef<V, Real, P> K;
  K.init();
  Coef<Real, Real, P> Ke;
  const Tab* tab = static_cast<const Tab*>(a.tab);
  const Real sigma = Real(a.sigma), omega = Real(a.omega);
  const Real cpi = Real(a.cpi), spi = Real(a.spi), scale = Real(a.two_over_nt);
  const V vsig = bc<V>(sigma);
  const double rys = (a.hx2 / a.hy2) * (a.hx2 / a.hy2);  // (4 / hy^2) / (4 / hx^2)
  // FP32: rys in two terms, in every y term of a row, or its rounding is left
  // over where the row should annihilate constants, at every time step with
  // the same sign (P = 4, N_t = 464, rys 0.99 half units off: error 1.9e-6
  // with one term in the partial sum T, 5.6e-7 with two everywhere)
  constexpr bool kLow = sizeof(Real) == 4;
  const V ry = bc<V>((Real)rys), ryl = bc<V>((Real)(rys - (double)(Real)rys));
  const Real rye = lo(ry), ryle = lo(ryl);
  auto scale_y = [&](V v) { return kLow ? vfma(ry, v, vmul(ryl, v)) : vmul(ry, v); };
  auto scale_ye = [&](Real v) { return kLow ? rye * v + ryle * v : rye * v; };
  const bool firstx = bx == 0, lastx = live && bx == sxe - 1;
  const bool firsty = by == 0 && firstC;
  // slabs of a cluster: the slab before takes this one's first row, the next
  // one the T of its last band; the warps that hold these bands wait for the
  // neighbours' in turn, the thread of a band's first tile announces its bytes
  const bool sendPrev = live && by == 0 && !firstC, sendNext = live && by == nb - 1 && !lastC;
  const int w0 = (int)(threadIdx.x & ~31u);  // the warp's first thread: its bands are w0 / LX .. (w0 + 31) / LX
  const bool waitPrev = MAIN && CLUS && !firstC && w0 == 0;
  const bool waitNext = MAIN && CLUS && !lastC && w0 <= nb * LX - 1 && nb * LX - 1 <= w0 + 31;
  const bool chainPrev = CHAIN && CLUS && !firstC && (int)(threadIdx.x >> 5) == x.wm;
  const bool chainNext = CHAIN && CLUS && !lastC && (int)(threadIdx.x >> 5) == x.wm;
  bool answered = true;
  unsigned phase = 0;  // of the barriers of the current parity
  // the tile's nodes on the west column and the south row: alpha - 1 and
  // beta b in registers (zero on the other tiles: no branch in the time loop)
  V wal[P], wbr[P], wbi[P];
  Real sal[P], sbr[P], sbi[P];  // south row, columns 1 .. P-1
#pragma unroll
  for (int r = 0; r < P; ++r) {
    wal[r] = wbr[r] = wbi[r] = bc<V>(Real(0));
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const bool south = r == 0 && h == 0 && firsty && !firstx;
      if (live && (firstx || south)) {
        const Real* w = sm + (south ? y.ts + 4 * (bx * P) : y.tw + 4 * (by * RH + h * P + r));
        put_half<H>(wal[r], h, w[0]);
        put_half<H>(wbr[r], h, w[1]);
        put_half<H>(wbi[r], h, w[2]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < P; ++c) {
    sal[c] = sbr[c] = sbi[c] = Real(0);
    if (c > 0 && live && firsty) {
      const Real* w = sm + y.ts + 4 * (bx * P + c);
      sal[c] = w[0];
      sbr[c] = w[1];
      sbi[c] = w[2];
    }
  }
  const int pr_ = (x.nb + 1) * y.row;  // one parity of a row buffer
  const bool lastE = (inA && e == nA - 1) || (inB && eB == sxe - 1);
  const bool firstE = inA ? (e == 0 && firstC) : eB == 0;
  const int en = inB ? LX : ncol, ei = inB ? eB : eA;  // chain lane: its buffer's length, its element
  // the subdomain's first column and row: twice the own part, nothing received
  const Real mx = firstx ? Real(2) : Real(1), rx = firstx ? Real(0) : Real(1);
  const V my = half_of<H, V>(firsty ? Real(2) : Real(1), Real(1));
  const V rry = half_of<H, V>(firsty ? Real(0) : rye, rye), rryl = half_of<H, V>(firsty ? Real(0) : ryle, ryle);

  Pair<V> s[P][P], v[P][P];         // p, p-dot; the filter sums
  Pair<Real> es[P + 1], ev[P + 1];  // the chain's
#pragma unroll
  for (int r = 0; r < P; ++r)
#pragma unroll
    for (int c = 0; c < P; ++c) v[r][c].a = v[r][c].b = bc<V>(Real(0));
#pragma unroll
  for (int q = 0; q <= P; ++q) ev[q].a = ev[q].b = Real(0);

  // Several steps per turn of a one-warp kernel's time loop, an even number, so
  // that each parity's buffers are fixed offsets.  1024 subdomains of 25 x 25
  // nodes, P = 3, by 1 / 2 / 4 / 6 / 8 steps: 650 / 635 / 588 / 573 / 695 us; with
  // a source by 1 / 2 / 4 / 6: 736 / 743 / 705 / 745; twice as many, not square, by
  // 1 / 2 / 4 / 6: 452 / 413 / 382 / 461; the tolerance mode has its best at 2.
  // P = 4 and 5 spill (96 to 256 bytes at P = 5).
  constexpr bool kPairs = P == 3 && H == 2;
  constexpr int kTurn = !FUSE || P > 3 ? 1 : !kPairs ? (SRC ? 1 : 2) : TOL ? 2 : ISO && !SRC ? 6 : 4;
  constexpr bool kTwo = kTurn > 1;  // parity known at compile time
  int cur = 0, m_done = 0;
  bool done = false;  // tolerance met (FUSE: this lane group; else the whole subdomain)
  for (int m = 0; m < a.m_wh; ++m) {
    if (tol) {  // previous iterate
      Real* st = sm + y.stash;
      int k = 0;
#pragma unroll
      for (int r = 0; r < P; ++r)
#pragma unroll
        for (int c = 0; c < P; ++c)
#pragma unroll
          for (int h = 0; h < H; ++h, ++k) {
            st[(2 * k) * nthr + t] = get<H>(v[r][c].a, h);
            st[(2 * k + 1) * nthr + t] = get<H>(v[r][c].b, h);
          }
#pragma unroll
      for (int q = 0; q <= P; ++q, ++k) {
        st[(2 * k) * nthr + t] = ev[q].a;
        st[(2 * k + 1) * nthr + t] = ev[q].b;
      }
    }
    {
      const Tab t0 = tab[0];
#pragma unroll
      for (int r = 0; r < P; ++r)
#pragma unroll
        for (int c = 0; c < P; ++c) {
          s[r][c].a = v[r][c].a;
          // Re{-i w u e^{-i pi/N_t}}
          s[r][c].b = vmul(bc<V>(omega), vfma(v[r][c].b, bc<V>(cpi), vmul(v[r][c].a, bc<V>(-spi))));
          v[r][c].a = vmul(bc<V>((Real)t0.z), s[r][c].a);
          v[r][c].b = vmul(bc<V>((Real)t0.w), s[r][c].b);
        }
#pragma unroll
      for (int q = 0; q <= P; ++q) {
        es[q].a = ev[q].a;
        es[q].b = omega * (ev[q].b * cpi - ev[q].a * spi);
        ev[q].a = t0.z * es[q].a;
        ev[q].b = t0.w * es[q].b;
      }
    }
    Tab tb = tab[1];
    if (kTwo) __syncwarp();  // the first step may write the buffers that the last iteration's last step read
#pragma unroll kTurn
    for (int nu = 1; nu < a.Nt; ++nu) {
      if (kTwo) cur = nu & 1;
      const Tab tn = tab[nu + 1];  // prefetch (the table has N_t + 1 entries)
      Real* PY = sm + y.py + cur * pr_;
      Real* TY = sm + y.ty + cur * pr_;
      Real* CP = sm + y.cp + cur * y.col;
      Real* TA = sm + y.ta + cur * y.col;
      V Ty[P], xe[P], xt[P], A[P][P];
      Real eext = Real(0), erec = Real(0), eT = Real(0);
      // ---- p, the partial sums for the neighbours, and the exchange
      if constexpr (MAIN) {
#pragma unroll
        for (int r = 0; r < P; ++r)
#pragma unroll
          for (int c = 0; c < P; ++c) s[r][c].a = vfma(vsig, s[r][c].b, s[r][c].a);
        Real p0[P], th[P];
#pragma unroll
        for (int c = 0; c < P; ++c) Ty[c] = vmul(K.hand(0), s[0][c].a);
#pragma unroll
        for (int b = 1; b < P; ++b)
#pragma unroll
          for (int c = 0; c < P; ++c) Ty[c] = vfma(K.hand(b), s[b][c].a, Ty[c]);
#pragma unroll
        for (int c = 0; c < P; ++c) {
          p0[c] = lo(s[0][c].a);
          th[c] = hi(Ty[c]);
        }
        RB::template st<!FUSE>(live, PY + byc * y.row, LX, bx, p0);
        RB::template st<!FUSE>(live, TY + (byc + 1) * y.row, LX, bx, th);
        if constexpr (CLUS) {
          const unsigned z = sizeof(Real);
          if (sendPrev) RB::st_async(smP + z * (y.py + cur * pr_ + x.nb * y.row), LX, bx, p0, mbP + 8 * (4 * cur + kTileNext));
          if (sendNext) RB::st_async(smN + z * (y.ty + cur * pr_), LX, bx, th, mbN + 8 * (4 * cur + kTilePrev));
        }
        V Tx[P];
#pragma unroll
        for (int r = 0; r < P; ++r) Tx[r] = vmul(K.hand(0), s[r][0].a);
#pragma unroll
        for (int b = 1; b < P; ++b)
#pragma unroll
          for (int r = 0; r < P; ++r) Tx[r] = vfma(K.hand(b), s[r][b].a, Tx[r]);
#pragma unroll
        for (int r = 0; r < P; ++r) {
          xe[r] = shfl_down1(s[r][0].a);
          xt[r] = shfl_up1(Tx[r]);
          // The first column multiplies what it gets by zero; in a warp of
          // several subdomains that may be another one's infinity or NaN.
          if (SHARED && firstx) xt[r] = bc<V>(Real(0));
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {
          Real tv[P];
#pragma unroll
          for (int r = 0; r < P; ++r) tv[r] = get<H>(Tx[r], h);
          RB::template st<!FUSE>(lastx, TA, ncol, byc * H + h, tv);
        }
      }
      if constexpr (CHAIN) {
#pragma unroll
        for (int q = 0; q <= P; ++q) es[q].a += sigma * es[q].b;
        eT = Ke.hand(0) * es[0].a;
#pragma unroll
        for (int b = 1; b < P; ++b) eT += Ke.hand(b) * es[b].a;
        eext = shfl_down1(es[0].a);
        erec = shfl_up1(eT);
        Real tv[P];
#pragma unroll
        for (int q = 0; q < P; ++q) tv[q] = es[q].a;
        RB::template st<!FUSE>(inE, inB ? PY + nb * y.row : CP, en, ei, tv);
        if constexpr (FUSE) {
          if (corner) *RB::first(CP, nA) = es[P].a;
          if (inB && lastE) *RB::first(TA, nA) = eT;
        } else {
          st_if(corner, smem_addr(RB::first(CP, nA)), es[P].a);
          st_if(inB && lastE, smem_addr(RB::first(TA, nA)), eT);
        }
        if constexpr (CLUS) {
          const unsigned z = sizeof(Real);
          const int cpo = (int)(RB::first(sm + y.cp + cur * y.col, ncol - 1) - sm);
          if (inA && e == 0 && !firstC) RB::st_async1(smP + z * cpo, es[0].a, mbP + 8 * (4 * cur + kChainNext));
          if (inA && lastE && !lastC) RB::st_async1(smN + z * (y.tax + cur), eT, mbN + 8 * (4 * cur + kChainPrev));
        }
      }
      if constexpr (CLUS) {  // what this slab stores in this step (predicated: no divergence here)
        const unsigned bytes = MAIN ? sxe * RB::kBytes : sizeof(Real);
        mbar_expect(MAIN ? sendPrev && bx == 0 : inA && e == 0 && !firstC,
                    mbP + 8 * (4 * cur + (MAIN ? kTileNext : kChainNext)), bytes);
        mbar_expect(MAIN ? sendNext && bx == 0 : inA && lastE && !lastC,
                    mbN + 8 * (4 * cur + (MAIN ? kTilePrev : kChainPrev)), bytes);
      }
      const V ct = bc<V>((Real)tb.x), st = bc<V>((Real)tb.y), kz = bc<V>((Real)tb.z), kw = bc<V>((Real)tb.w);
      // ---- the part of the stiffness that the tile's own nodes give:
      // A = X + (hx/hy)^2 Y (ISO: square elements), row by row with the row's
      // columns side by side: independent FMA chains
      if constexpr (MAIN) {
#pragma unroll
        for (int r = 0; r < P; ++r) {
          // x sums beside the y sums (one addition more, shorter chains) or going
          // on from them: 765 / 757 us for P = 4, 32 x 32 elements at 144
          // subdomains, but 666 / 743 for P = 5, 8 x 8 at 1024
          constexpr bool kBeside = H == 1 && P <= 4;
          V X[P], Y[P];
          X[0] = bc<V>(Real(0));  // the first column's own x taps
#pragma unroll
          for (int b = 0; b < P; ++b) {
#pragma unroll
            for (int c = 0; c < P; ++c) {
              if (c > 0 && kBeside) X[c] = b == 0 ? vmul(K.at(c, 0), s[r][0].a) : vfma(K.at(c, b), s[r][b].a, X[c]);
              else if (c == 0 && b > 0) X[0] = b == 1 ? vmul(K.own(1), s[r][1 % P].a) : vfma(K.own(b), s[r][b].a, X[0]);
              if (r > 0) Y[c] = b == 0 ? vmul(K.at(r, 0), s[0][c].a) : vfma(K.at(r, b), s[b][c].a, Y[c]);
              else if (b > 0) Y[c] = b == 1 ? vmul(K.own(1), s[1 % P][c].a) : vfma(K.own(b), s[b][c].a, Y[c]);
            }
          }
          // a shared node: its diagonal, and twice the own part at the subdomain's end
          if (r == 0) {
#pragma unroll
            for (int c = 0; c < P; ++c) {
              const V dy = vmul(K.diag(), s[0][c].a);
              Y[c] = P > 1 ? vfma(my, Y[c], dy) : dy;
            }
          }
          if (!ISO) {  // (hx/hy)^2, its FP32 rounding made up by a second term
#pragma unroll
            for (int c = 0; c < P; ++c) Y[c] = scale_y(Y[c]);
          }
          A[r][0] = vfma(K.diag(), s[r][0].a, Y[0]);
          if (P > 1) A[r][0] = vfma(bc<V>(mx), X[0], A[r][0]);
#pragma unroll
          for (int b = 0; b < P; ++b)
#pragma unroll
            for (int c = 1; c < P; ++c)
              if (!kBeside) A[r][c] = vfma(K.at(c, b), s[r][b].a, b == 0 ? Y[c] : A[r][c]);
#pragma unroll
          for (int c = 1; c < P; ++c)
            if (kBeside) A[r][c] = vadd(X[c], Y[c]);
        }
        // edge columns and rows: (alpha - 1) p-dot + beta b
#pragma unroll
        for (int r = 0; r < P; ++r)
          s[r][0].b = vfma(wal[r], s[r][0].b, vfma(wbr[r], ct, vfma(wbi[r], st, s[r][0].b)));
#pragma unroll
        for (int c = 1; c < P; ++c) {
          const Real f = lo(s[0][c].b);
          put_half<H>(s[0][c].b, 0, vfma(sal[c], f, vfma(sbr[c], (Real)tb.x, vfma(sbi[c], (Real)tb.y, f))));
        }
        if (SRC) {
#pragma unroll
          for (int r = 0; r < P; ++r)
#pragma unroll
            for (int c = 0; c < P; ++c) {
              const SrcPair<V> f = srcT[(r * P + c) * nthr];
              s[r][c].b = vfma(f.re, ct, vfma(f.im, st, s[r][c].b));
            }
        }
      }
      if (FUSE || CLUS) __syncwarp();  // (clusters: 2% faster with the warps reconverged before the barrier, blocks slower)
      if (!FUSE) block_bar();
      if constexpr (CLUS) {
        const unsigned mb = mb0 + 32 * cur;
        if (answered && (MAIN ? waitPrev : chainPrev)) answered = mbar_wait(mb + 8 * (MAIN ? kTilePrev : kChainPrev), phase);
        if (answered && (MAIN ? waitNext : chainNext)) answered = mbar_wait(mb + 8 * (MAIN ? kTileNext : kChainNext), phase);
        __syncwarp();
      }
      // ---- what the neighbours sent, and the update
      auto update_tiles = [&]() {
        Real ey[P], ty[P];
        RB::ld(PY + (byc + 1) * y.row, LX, bx, ey);
        RB::ld(TY + byc * y.row, LX, bx, ty);
#pragma unroll
        for (int h = 0; h < H; ++h) {
          Real tv[P];
          RB::ld(CP, ncol, byc * H + h, tv);
#pragma unroll
          for (int r = 0; r < P; ++r)
            if (lastx) put_half<H>(xe[r], h, tv[r]);
        }
        V ye[P];
#pragma unroll
        for (int c = 0; c < P; ++c) {
          ye[c] = half_of<H, V>(H == 2 ? hi(s[0][c].a) : ey[c], ey[c]);
          if (!ISO) ye[c] = scale_y(ye[c]);
          const V T = half_of<H, V>(ty[c], lo(Ty[c]));
          if (!ISO && kLow) A[0][c] = vfma(rryl, T, A[0][c]);
          A[0][c] = vfma(rry, T, A[0][c]);
        }
        const V mkP = vmul(bc<V>(mx), K.own(P)), myP = vmul(my, K.own(P));
#pragma unroll
        for (int r = 0; r < P; ++r) {
#pragma unroll
          for (int c = 0; c < P; ++c) A[r][c] = vfma(c == 0 ? mkP : K.at(c, P), xe[r], A[r][c]);
          A[r][0] = vfma(bc<V>(rx), xt[r], A[r][0]);
#pragma unroll
          for (int c = 0; c < P; ++c) A[r][c] = vfma(r == 0 ? myP : K.at(r, P), ye[c], A[r][c]);
#pragma unroll
          for (int c = 0; c < P; ++c) s[r][c].b = vfma(nbet[r][c], A[r][c], s[r][c].b);
#pragma unroll
          for (int c = 0; c < P; ++c) accumulate(v[r][c], kz, kw, s[r][c]);
        }
      };
      // ---- the chains
      auto update_chains = [&]() {
        Real cr[P];
        RB::ld(inB ? TY + nb * y.row : TA, en, ei, cr);
        const Real cpn = *RB::first(CP, nA), ca = *RB::first(TA, nA);
        if (lastE) eext = cpn;
        if (CLUS && inA && e == 0) erec = sm[y.tax + cur];
        const Real ec = (Real)tb.x, esn = (Real)tb.y;
#pragma unroll
        for (int q = 0; q < P; ++q) {
          Real S;  // along the chain
          if (q == 0) {
            Real o = Ke.own(P) * eext;
#pragma unroll
            for (int b = 1; b < P; ++b) o += Ke.own(b) * es[b].a;
            S = (o + Ke.diag() * es[0].a) + (firstE ? o : erec);
          } else {
            S = Ke.at(q, P) * eext;
#pragma unroll
            for (int b = 0; b < P; ++b) S += Ke.at(q, b) * es[b].a;
          }
          const Real C = Ke.diag() * es[q].a + Real(2) * cr[q];
          // the y sum is the chain's own on chain A, the one across it on chain B
          const Real Ac = ISO ? S + C : inA ? C + scale_ye(S) : S + scale_ye(C);
          es[q].b = eal[q] * es[q].b + ebet[q] * Ac + ebr[q] * ec + ebi[q] * esn;
          accumulate(ev[q], (Real)tb.z, (Real)tb.w, es[q]);
        }
        // the corner (zero coefficients elsewhere)
        const Real d = Ke.diag() * es[P].a;
        const Real Y = d + Real(2) * eT;
        const Real Ac = (d + Real(2) * ca) + (ISO ? Y : scale_ye(Y));
        es[P].b = eal[P] * es[P].b + ebet[P] * Ac + ebr[P] * ec + ebi[P] * esn;
        accumulate(ev[P], (Real)tb.z, (Real)tb.w, es[P]);
      };
      // (paired one-warp kernels: the chains before the tiles, 585 / 573 us)
      if constexpr (CHAIN && kPairs && FUSE) update_chains();
      if constexpr (MAIN) update_tiles();
      if constexpr (CHAIN && !(kPairs && FUSE)) update_chains();
      tb = tn;
      if (CLUS) phase ^= cur;  // the barriers' phase turns when parity 1 has been used
      if (!kTwo) cur ^= 1;
    }
    // u^{(m+1)} = (2/N_t) v
#pragma unroll
    for (int r = 0; r < P; ++r)
#pragma unroll
      for (int c = 0; c < P; ++c) {
        v[r][c].a = vmul(bc<V>(scale), v[r][c].a);
        v[r][c].b = vmul(bc<V>(scale), v[r][c].b);
      }
#pragma unroll
    for (int q = 0; q <= P; ++q) {
      ev[q].a *= scale;
      ev[q].b *= scale;
    }
    if (!done) m_done = m + 1;
    if (tol) {
      // per-subdomain stop: ||u^{m+1} - u^m|| <= wh_tol ||u^{m+1}||.  A lane
      // group of a shared warp that has stopped keeps its iterate.
      const Real* st = sm + y.stash;
      double dn = 0.0, un = 0.0;
      NormAcc acc;
      if constexpr (sizeof(Real) == 4) {
        float big = 0.f;
        auto largest = [&](float nr, float ni, int k) {
          big = fmaxf(fmaxf(big, fmaxf(fabsf(nr), fabsf(ni))),
                      fmaxf(fabsf(st[(2 * k) * nthr + t]), fabsf(st[(2 * k + 1) * nthr + t])));
        };
        int k = 0;
#pragma unroll
        for (int r = 0; r < P; ++r)
#pragma unroll
          for (int c = 0; c < P; ++c)
#pragma unroll
            for (int h = 0; h < H; ++h, ++k)
              if (live) largest(get<H>(v[r][c].a, h), get<H>(v[r][c].b, h), k);
#pragma unroll
        for (int q = 0; q <= P; ++q, ++k)
          if (q < P ? inE : corner) largest(ev[q].a, ev[q].b, k);
        acc.start(big);
      }
      int k = 0;
      auto count = [&](Real nr, Real ni, Real orr, Real oi) {
        if constexpr (sizeof(Real) == 4) {
          acc.add(make_float2(nr, ni), make_float2(orr, oi));
        } else {
          const double dr = nr - orr, di = ni - oi;
          dn += dr * dr + di * di;
          un += nr * nr + ni * ni;
        }
      };
#pragma unroll
      for (int r = 0; r < P; ++r)
#pragma unroll
        for (int c = 0; c < P; ++c)
#pragma unroll
          for (int h = 0; h < H; ++h, ++k) {
            const Real orr = st[(2 * k) * nthr + t], oi = st[(2 * k + 1) * nthr + t];
            if (live) count(get<H>(v[r][c].a, h), get<H>(v[r][c].b, h), orr, oi);
            if (done) {
              put_half<H>(v[r][c].a, h, orr);
              put_half<H>(v[r][c].b, h, oi);
            }
          }
#pragma unroll
      for (int q = 0; q <= P; ++q, ++k) {
        const Real orr = st[(2 * k) * nthr + t], oi = st[(2 * k + 1) * nthr + t];
        if (q < P ? inE : corner) count(ev[q].a, ev[q].b, orr, oi);
        if (done) {
          ev[q].a = orr;
          ev[q].b = oi;
        }
      }
      if constexpr (sizeof(Real) == 4) acc.finish(dn, un);
      if (FUSE) {
        for (int o = x.gs >> 1; o > 0; o >>= 1) {
          dn += __shfl_xor_sync(0xffffffffu, dn, o);
          un += __shfl_xor_sync(0xffffffffu, un, o);
        }
        if (dn <= a.wh_tol * a.wh_tol * un) done = true;
        if (__all_sync(0xffffffffu, done || !have)) break;
      } else {
        // per-warp sums, then one thread per CTA, then every CTA adds the
        // cluster's in the same order, so all take the same decision
        double(*red)[2] = ts->red;
        double* part = ts->part;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          dn += __shfl_xor_sync(0xffffffffu, dn, o);
          un += __shfl_xor_sync(0xffffffffu, un, o);
        }
        if (lane == 0) {
          red[threadIdx.x >> 5][0] = dn;
          red[threadIdx.x >> 5][1] = un;
        }
        block_bar();
        if (threadIdx.x == 0) {
          double D = 0.0, U = 0.0;
          for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            D += red[w][0];
            U += red[w][1];
          }
          part[0] = D;
          part[1] = U;
        }
        if (CLUS) cluster.sync();
        if (threadIdx.x == 0) {
          double D = 0.0, U = 0.0;
          for (int r = 0; r < CL; ++r) {
            const double* pr = CLUS ? cluster.map_shared_rank(part, r) : part;
            D += pr[0];
            U += pr[1];
          }
          ts->stop = (D <= a.wh_tol * a.wh_tol * U) ? 1 : 0;
        }
        if (CLUS) cluster.sync();  // remote reads of part done, stop visible to the CTA
        else block_bar();
        if (ts->stop) break;
      }
    }
  }

  if constexpr (CLUS) {
    if (!answered)
      for (int k = 0; k < CL; ++k) *cluster.map_shared_rank(&ts->gave_up, k) = 1;
    cluster.sync();  // the neighbours' last pushes have landed, and word of waits that ran out
    if (ts->gave_up) {
      // No result rather than a wrong one: NaN in the subdomain's solution
      // and in what it sends.  A push that nobody waited for may still be
      // under way: a microsecond's work, given a hundred before this CTA ends.
      const Real nan = Real(__int_as_float(0x7fffffff));
#pragma unroll
      for (int r = 0; r < P; ++r)
#pragma unroll
        for (int c = 0; c < P; ++c) v[r][c].a = v[r][c].b = bc<V>(nan);
#pragma unroll
      for (int q = 0; q <= P; ++q) ev[q].a = ev[q].b = nan;
      for (const long long t0 = clock64(); clock64() - t0 < 200000;) {
      }
      if (threadIdx.x == 0) atomicOr(a.flags, 2);
    }
  }
  // ---- outputs
  bool bad = false;
  auto out = [&](int i, int j, Real re, Real im) {
    if (!isfinite(re) || !isfinite(im)) bad = true;
    if (a.u_sub) store_complex(a.u_sub, (int64_t)l * nn + (int64_t)j * nlx + i, make_double2(re, im));
  };
  if (live) {
#pragma unroll
    for (int r = 0; r < P; ++r)
#pragma unroll
      for (int h = 0; h < H; ++h)
#pragma unroll
        for (int c = 0; c < P; ++c)
          out(bx * P + c, row0 + by * RH + h * P + r, get<H>(v[r][c].a, h), get<H>(v[r][c].b, h));
  }
#pragma unroll
  for (int q = 0; q <= P; ++q)
    if (q < P ? inE : corner)
      out(inA ? nlx - 1 : eB * P + q, inA ? row0 + e * P + q : nly - 1, ev[q].a, ev[q].b);
  if (bad) atomicOr(a.flags, 1);
  if (t == 0 && have && firstC && a.wh_iter_max) {
    atomicMax(a.wh_iter_max, m_done);
    atomicAdd(a.wh_iter_sum, (unsigned long long)m_done);
  }
  // the four edges' solutions staged in shared memory (the exchange buffers:
  // their last reads lie behind the barrier below), so that every thread
  // takes entries of the transmission update.  W, E: local rows; S, N: columns
  if (FUSE) __syncwarp();
  else if (!CLUS) block_bar();  // (clusters: the barrier above)
  const int rowsC = nb * RH + (lastC ? 1 : 0);  // node rows of this slab
  const int nrow = nb * RH + 1;
  Real* uW = sm + y.tw;       // [rows][2]
  Real* uE = uW + 2 * nrow;   // [rows][2]
  Real* uS = sm + y.ts;       // [cols][2]
  Real* uN = uS + 2 * nlx;    // [cols][2]
  auto stage = [&](Real* dst, int q, Real re, Real im) {
    dst[2 * q] = re;
    dst[2 * q + 1] = im;
  };
  if (live && firstx) {
#pragma unroll
    for (int r = 0; r < P; ++r)
#pragma unroll
      for (int h = 0; h < H; ++h) stage(uW, by * RH + h * P + r, get<H>(v[r][0].a, h), get<H>(v[r][0].b, h));
  }
  if (live && firsty) {
#pragma unroll
    for (int c = 0; c < P; ++c) stage(uS, bx * P + c, lo(v[0][c].a), lo(v[0][c].b));
  }
#pragma unroll
  for (int q = 0; q <= P; ++q) {
    if (q < P ? inA : corner) {
      stage(uE, e * P + q, ev[q].a, ev[q].b);
      if (e == 0 && q == 0 && firstC) stage(uS, nlx - 1, ev[q].a, ev[q].b);
      if (q == P) stage(uN, nlx - 1, ev[q].a, ev[q].b);
    }
    if (q < P && inB) {
      stage(uN, eB * P + q, ev[q].a, ev[q].b);
      if (eB == 0 && q == 0) stage(uW, nb * RH, ev[q].a, ev[q].b);
    }
  }
  if (FUSE) __syncwarp();
  else block_bar();
  if (have) {
    const int NE = a.NE;
    for (int k = t; k < 4 * NE; k += nthr) {
      const int ed = k / NE, q = k - ed * NE;
      const int len = ed < 2 ? nly : nlx;
      // the slab writes its own rows of W and E, the first CTA S, the last one
      // N and every slot's padding (q >= len)
      int loc = q;
      if (q >= len) {
        if (!lastC) continue;
      } else if (ed < 2) {
        loc = q - row0;
        if (loc < 0 || loc >= rowsC) continue;
      } else if (ed == 2 ? !firstC : !lastC) {
        continue;
      }
      const bool iface = ed == 0 ? ifW : ed == 1 ? ifE : ed == 2 ? ifS : ifN;
      double2 v = make_double2(0.0, 0.0);
      int64_t dst = ((int64_t)l * 4 + ed) * NE + q;
      if (iface) {
        const int rn = ed == 0 ? l - 1 : ed == 1 ? l + 1 : ed == 2 ? l - a.Sx : l + a.Sx;
        dst = ((int64_t)rn * 4 + (ed ^ 1)) * NE + q;
        if (q < len) {
          const Real* us = (ed == 0 ? uW : ed == 1 ? uE : ed == 2 ? uS : uN) + 2 * loc;
          const double ur = (double)us[0], ui = (double)us[1];
          const double kk = kedgeL[ed * NE + q];
          const double2 lr = load_complex(lamL, ed * NE + q);
          // -lambda + 2 k (eta - i zeta) u, eta = 0
          v.x = -lr.x + 2.0 * kk * (a.eta * ur + a.zeta * ui);
          v.y = -lr.y + 2.0 * kk * (a.eta * ui - a.zeta * ur);
        }
      }
      store_complex(a.lam_out, dst, v);
    }
  }
}

// LANES: lanes of a one-warp subdomain are 1 the whole warp, 2 a part of it;
// 0: more than one warp.  (1 and 2 apart: selecting zeros costs the benchmark's
// one-warp subdomains 2.7%, those that share a warp 0.5%.)
// TOL: the tolerance mode too.  FP32 sweeps of a fixed count have instantiations
// without it, which have a register or two more and time loops of their own:
// 1024 subdomains of 129 x 129 nodes, P = 4: 22.7 -> 20.7 ms; 48 of 37 x 31, P = 3:
// 198 -> 187 us; 128 x 128, P = 5, 4 x 4 elements each: 1051 -> 1015 us.
// One block per SM as the launch bound: without it some of them are compiled
// for 64 or 74 registers (16 subdomains of 17 x 17, P = 2: 357 us against 166).
template <typename Real, int P, int H, int LANES, bool SRC, bool ISO, bool CLUS, bool TOL, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) sweep_tile_kernel(const __grid_constant__ TileArgs x) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if constexpr (LANES > 0) {
    tile_body<Real, P, H, kBoth, LANES == 2, SRC, ISO, CLUS, TOL>(x, smem_raw, nullptr);
  } else {
    __shared__ TolShared ts;
    if ((int)(threadIdx.x >> 5) < x.wm) tile_body<Real, P, H, kTiles, false, SRC, ISO, CLUS, TOL>(x, smem_raw, &ts);
    else tile_body<Real, P, H, kChains, false, SRC, ISO, CLUS, TOL>(x, smem_raw, &ts);
  }
}

}  // namespace tile_sweep
}  // namespace hz
