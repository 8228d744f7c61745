// FP64 kernels around the sweep: leapfrog coefficients, right-hand side,
// global operator residual, assembly of subdomain copies, and the vector
// operations of the outer Krylov iteration.  All stream their data once with
// coalesced x-fastest access.  The right-hand side and the assembly are
// HBM-bound; the residual and the Krylov vector kernels do enough FP64
// arithmetic per byte that this part's FP64 pipe bounds them, so they are
// written with the fewest FP64 operations (FMA chains).  Reductions are
// two-pass with a fixed summation order (deterministic results).
#include <cuda_runtime.h>

#include <atomic>

#include <cmath>

#include "hz_complex_io.cuh"
#include "hz_internal.h"

namespace hz {
namespace {

constexpr int kRedThreads = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block sum of NV values per thread into out[0..NV-1] (thread 0 holds result).
template <int NV>
__device__ void block_sum(double (&v)[NV], double* out) {
  __shared__ double sh[NV][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    double x = warp_sum(v[k]);
    if (lane == 0) sh[k][warp] = x;
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double x = (lane < nw) ? sh[k][lane] : 0.0;
      x = warp_sum(x);
      if (lane == 0) out[k] = x;
    }
  }
}

// ---- leapfrog coefficients (Sec. 5): per subdomain node
//   M = W / c^2 (W = Wx_i Wy_j, or the mapped mesh's lumped weight),
//   H = (edge weights over all four subdomain edges) / c
//   alpha = (M - theta H)/(M + theta H), beta = sigma/(M + theta H)
__global__ void prepare_kernel(const __grid_constant__ PrepArgs a) {
  const int l = blockIdx.y;
  const int nn = a.nlx * a.nly;
  const int sxi = l % a.Sx, syi = l / a.Sx;
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < nn; n += gridDim.x * blockDim.x) {
    const int i = n % a.nlx, j = n / a.nlx;
    const int64_t I = (int64_t)sxi * a.snxP + i, J = (int64_t)syi * a.snyP + j;
    const double c = a.c[J * a.NXg + I];
    // lumped weight and edge weights: products of the 1D tables on a Cartesian
    // mesh, the map's per-node values on a mapped one
    const double* E = a.Esub ? a.Esub + (int64_t)l * 4 * a.NE : nullptr;
    const double W = a.Wsub ? a.Wsub[(int64_t)l * nn + n] : a.wxs[i] * a.wys[j];
    const double eS = E ? E[2 * a.NE + i] : a.wxs[i], eN = E ? E[3 * a.NE + i] : a.wxs[i];
    const double eW = E ? E[0 * a.NE + j] : a.wys[j], eE = E ? E[1 * a.NE + j] : a.wys[j];
    const double M = W / (c * c);
    // impedance damping on every subdomain edge: weight 1 on the outer
    // boundary, zeta on interfaces (the interface condition's d_t part)
    const double fS = syi > 0 ? a.zeta : 1.0, fN = syi < a.Sy - 1 ? a.zeta : 1.0;
    const double fW = sxi > 0 ? a.zeta : 1.0, fE = sxi < a.Sx - 1 ? a.zeta : 1.0;
    const double Hw = (j == 0 ? fS * eS : 0.0) + (j == a.nly - 1 ? fN * eN : 0.0) + (i == 0 ? fW * eW : 0.0) +
                      (i == a.nlx - 1 ? fE * eE : 0.0);
    const double H = Hw / c;
    const double den = M + a.theta * H;
    const double be = a.sigma / den;
    const double al = (M - a.theta * H) / den;
    const int64_t k = (int64_t)l * nn + n;
    a.beta64[k] = be;
    a.alpha64[k] = al;
    a.beta32[k] = (float)be;
    a.alpha32[k] = (float)al;
  }
  if (blockIdx.x == 0) {
    for (int k = threadIdx.x; k < 4 * a.NE; k += blockDim.x) {
      const int e = k / a.NE, t = k % a.NE;
      const int len = (e < 2) ? a.nly : a.nlx;
      double val = 0.0;
      if (t < len) {
        const int i = (e == 0) ? 0 : (e == 1) ? a.nlx - 1 : t;
        const int j = (e == 2) ? 0 : (e == 3) ? a.nly - 1 : t;
        const int64_t I = (int64_t)sxi * a.snxP + i, J = (int64_t)syi * a.snyP + j;
        val = a.omega / a.c[J * a.NXg + I];
      }
      a.kedge[(int64_t)l * 4 * a.NE + k] = val;
    }
  }
}

// ---- b = (f, phi) + <g, phi>, lumped GLL quadrature (Sec. 4)
__global__ void rhs_kernel(const __grid_constant__ GlobalArgs a, const double* __restrict__ f,
                           const double* __restrict__ gb, double* __restrict__ b) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = blockIdx.y;
  if (I >= a.NXg) return;
  const int64_t n = (int64_t)J * a.NXg + I;
  const double wx = a.Wxg[I], wy = a.Wyg[J];
  double br = wx * wy * f[2 * n], bi = wx * wy * f[2 * n + 1];
  const int64_t oS = 0, oE = a.NXg, oN = a.NXg + a.NYg, oW = 2 * a.NXg + a.NYg;
  if (J == 0) { br += wx * gb[2 * (oS + I)]; bi += wx * gb[2 * (oS + I) + 1]; }
  if (J == a.NYg - 1) { br += wx * gb[2 * (oN + I)]; bi += wx * gb[2 * (oN + I) + 1]; }
  if (I == 0) { br += wy * gb[2 * (oW + J)]; bi += wy * gb[2 * (oW + J) + 1]; }
  if (I == a.NXg - 1) { br += wy * gb[2 * (oE + J)]; bi += wy * gb[2 * (oE + J) + 1]; }
  b[2 * n] = br;
  b[2 * n + 1] = bi;
}

// 1 / x for finite x > 0 by Newton's iteration y <- y (2 - x y) from an FP32
// reciprocal: each step squares the relative error (2^-22, 2^-44, below one
// unit in the last place), four FP64 FMAs instead of a division's dozen.  The
// FP32 values are cut out of and put back into the FP64 words by shifts (the
// conversion instructions run at the FP64 rate).  Outside FP32's range the
// division itself.
__device__ __forceinline__ double recip(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  if (hi - (937u << 20) >= (172u << 20)) return 1.0 / x;  // outside 2^-86 .. 2^86
  const float f = __uint_as_float(((hi - (896u << 20)) << 3) | (lo >> 29));  // x cut to 23 bits
  const unsigned q = __float_as_uint(__frcp_rn(f));
  double y = __hiloint2double((int)((q >> 3) + (896u << 20)), (int)(q << 29));
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}

// ---- r = b - (A - i w H - w^2 M) u on the global grid (Sec. 4), FP64.
//   A u = Wx Wy [(Kx u) / Wx + (Ky u) / Wy], the assembled 1D rows divided by
// their lumped weights (host tables a.Kx, a.Ky by node class), so that
//   r = b - Wx Wy [(Kx u) / Wx + (Ky u) / Wy - (w/c)^2 u] + i (w/c) Hw u,
// the last term on the outer boundary only; both centre taps and -(w/c)^2 make
// one coefficient of the node's own value (a.Kd by the two classes).
// The FP64 pipe bounds it (about 1.7 FMA per clock and SM).  A thread per node
// ran the 2P + 1 taps of the widest row class on every lane and two divisions:
// 106 us on 769 x 769 nodes, P = 3, with the sums' second launch; 51 us now (41 us
// is 33 FP64 instructions per node at the pipe's measured rate).  Here a thread owns the P nodes of one
// element in one node row: the x class of a node is known at compile time, the
// y class is uniform in the warp, so a node runs only its own taps (5 instead
// of 7 on average at P = 3), and one reciprocal serves both divisions.  The
// mesh's last node column has blocks of its own, a thread per node (as a
// 33rd lane's work it cost a whole warp per row).  Blocks of four rows: more
// of them than eight rows give, for an even load of the SMs.
constexpr int kResRows = 4;
struct ResNode {  // what a node adds to the two sums
  double rr = 0.0, bb = 0.0;
};
// S: the node's taps including its own value's
template <bool PAIR>
__device__ __forceinline__ void residual_node(int64_t n, double W, double h, double2 u, double2 S,
                                              const double* __restrict__ b, double* __restrict__ r, ResNode& sum) {
  double2 bn = make_double2(0.0, 0.0);
  if (b) bn = load_complex<PAIR>(b, n);
  double rr = fma(-W, S.x, bn.x);
  double ri = fma(-W, S.y, bn.y);
  if (h != 0.0) {
    rr = fma(-h, u.y, rr);
    ri = fma(h, u.x, ri);
  }
  store_complex<PAIR>(r, n, make_double2(rr, ri));
  sum.rr = fma(rr, rr, fma(ri, ri, sum.rr));
  if (b) sum.bb = fma(bn.x, bn.x, fma(bn.y, bn.y, sum.bb));
}

template <int P, bool PAIR>
__global__ void __launch_bounds__(32 * kResRows)
    residual_kernel(const __grid_constant__ GlobalArgs a, int nbx, int nmain, const double* __restrict__ b,
                    const double* __restrict__ u, double* __restrict__ r, double* __restrict__ part,
                    unsigned* __restrict__ ticket, double* __restrict__ norms2) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ResNode sum;
  if ((int)blockIdx.x < nmain) {
    const int ex = (int)(blockIdx.x % nbx) * 32 + lane;
    const int J = (int)(blockIdx.x / nbx) * kResRows + warp;
    if (ex < a.nx && J < a.NYg) {
      const int64_t n0 = (int64_t)J * a.NXg + (int64_t)ex * P;
      double2 v[P + 1], S[P];
#pragma unroll
      for (int k = 0; k <= P; ++k) v[k] = load_complex_ro<PAIR>(u, n0 + k);
      // y: the element row's own nodes, and on a shared row the element below
      const int ay = J % P;
      const int cy = J == 0 ? P : J == a.NYg - 1 ? P + 1 : ay;
      double t[P];
#pragma unroll
      for (int k = 0; k < P; ++k) {
        t[k] = a.omega * recip(a.c[n0 + k]);
        const double d = fma(-t[k], t[k], k == 0 && ex == 0 ? a.Kd[P][cy] : a.Kd[k][cy]);
        S[k] = make_double2(d * v[k].x, d * v[k].y);
      }
      auto yrow = [&](int off) {  // row J + off, 0 < |off| <= P
        const double cf = a.Ky[cy][P + off];
        const int64_t row = n0 + (int64_t)off * a.NXg;
#pragma unroll
        for (int k = 0; k < P; ++k) {
          const double2 w = load_complex_ro<PAIR>(u, row + k);
          S[k].x = fma(cf, w.x, S[k].x);
          S[k].y = fma(cf, w.y, S[k].y);
        }
      };
      if (J < a.NYg - 1) {
#pragma unroll
        for (int t = 0; t <= P; ++t)
          if (t != ay) yrow(t - ay);
      }
      if (ay == 0 && J > 0) {
#pragma unroll
        for (int t = 1; t <= P; ++t) yrow(-t);
      }
      // x: the element's own nodes; node 0 also the element to the left
#pragma unroll
      for (int k = 1; k <= P; ++k) {
        const double cf = ex > 0 ? a.Kx[0][P + k] : a.Kx[P][P + k];
        S[0].x = fma(cf, v[k].x, S[0].x);
        S[0].y = fma(cf, v[k].y, S[0].y);
      }
      if (ex > 0) {
#pragma unroll
        for (int k = 1; k <= P; ++k) {
          const double2 w = load_complex_ro<PAIR>(u, n0 - k);
          S[0].x = fma(a.Kx[0][P - k], w.x, S[0].x);
          S[0].y = fma(a.Kx[0][P - k], w.y, S[0].y);
        }
      }
#pragma unroll
      for (int q = 1; q < P; ++q)
#pragma unroll
        for (int k = 0; k <= P; ++k) {
          if (k == q) continue;
          S[q].x = fma(a.Kx[q][P + k - q], v[k].x, S[q].x);
          S[q].y = fma(a.Kx[q][P + k - q], v[k].y, S[q].y);
        }
      const double Wy = a.Wyg[J];
      const bool yb = J == 0 || J == a.NYg - 1;
#pragma unroll
      for (int q = 0; q < P; ++q) {
        const double Wx = a.Wxg[ex * P + q];
        double h = 0.0;
        if (yb || (q == 0 && ex == 0)) h = t[q] * ((yb ? Wx : 0.0) + (q == 0 && ex == 0 ? Wy : 0.0));
        residual_node<PAIR>(n0 + q, Wx * Wy, h, v[q], S[q], b, r, sum);
      }
    }
  } else {
    const int J = ((int)blockIdx.x - nmain) * 32 * kResRows + (int)threadIdx.x;
    if (J < a.NYg) {
      const int I = a.NXg - 1;
      const int64_t n = (int64_t)J * a.NXg + I;
      const int cy = J == 0 ? P : J == a.NYg - 1 ? P + 1 : J % P;
      const double t = a.omega * recip(a.c[n]), d = fma(-t, t, a.Kd[P + 1][cy]);
      const double2 un = load_complex_ro<PAIR>(u, n);
      double2 S = make_double2(d * un.x, d * un.y);
      for (int k = -P; k <= P; ++k) {
        if (k == 0) continue;
        if (J + k >= 0 && J + k < a.NYg) {  // taps outside the row's class have coefficient 0
          const double2 w = load_complex_ro<PAIR>(u, n + (int64_t)k * a.NXg);
          S.x = fma(a.Ky[cy][P + k], w.x, S.x);
          S.y = fma(a.Ky[cy][P + k], w.y, S.y);
        }
        if (k < 0) {
          const double2 w = load_complex_ro<PAIR>(u, n + k);
          S.x = fma(a.Kx[P + 1][P + k], w.x, S.x);
          S.y = fma(a.Kx[P + 1][P + k], w.y, S.y);
        }
      }
      const double Wx = a.Wxg[I], Wy = a.Wyg[J];
      residual_node<PAIR>(n, Wx * Wy, t * (Wy + (J == 0 || J == a.NYg - 1 ? Wx : 0.0)), un, S, b, r, sum);
    }
  }
  if (!norms2) return;
  // the block's sums in a fixed order, one warp per sum (a warp reduction in
  // every warp is as many FP64 instructions as the taps of half a node)
  constexpr int kT = 32 * kResRows;
  __shared__ double sh[2][kT];
  __shared__ bool last;
  sh[0][threadIdx.x] = sum.rr;
  sh[1][threadIdx.x] = sum.bb;
  __syncthreads();
  if (warp < 2) {
    double x = 0.0;
    if (warp == 0 || b) {
#pragma unroll
      for (int k = 0; k < kResRows; ++k) x += sh[warp][32 * k + lane];
      x = warp_sum(x);
    }
    if (lane == 0) {
      part[2 * (int64_t)blockIdx.x + warp] = x;
      __threadfence();
    }
  }
  // the last block to finish adds the blocks' sums, in block order (the ticket
  // wraps to zero for the next call)
  __syncthreads();
  if (threadIdx.x == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  double x0 = 0.0, x1 = 0.0;
  for (int k = threadIdx.x; k < (int)gridDim.x; k += kT) {
    const double2 p = __ldcg(reinterpret_cast<const double2*>(part) + k);
    x0 += p.x;
    x1 += p.y;
  }
  sh[0][threadIdx.x] = x0;
  sh[1][threadIdx.x] = x1;
  __syncthreads();
  if (warp < 2) {
    double x = 0.0;
#pragma unroll
    for (int k = 0; k < kResRows; ++k) x += sh[warp][32 * k + lane];
    x = warp_sum(x);
    if (lane == 0) norms2[warp] = x;
  }
}

// out[k] = sum_blk part[blk * width + k], fixed order; one block per k.
__global__ void reduce_partials_kernel(const double* __restrict__ part, int nblocks, int width,
                                       double* __restrict__ out) {
  const int k = blockIdx.x;
  double v[1] = {0.0};
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) v[0] += part[(int64_t)b * width + k];
  __shared__ double res[1];
  block_sum<1>(v, res);
  if (threadIdx.x == 0) out[k] = res[0];
}

// u += average of the subdomain copies at every global node, weighted by the
// lumped-mass share of each copy (1/count on a uniform mesh: 1, 1/2 on
// interfaces, 1/4 at cross points; a.share on a mapped mesh).
__global__ void assemble_add_kernel(const __grid_constant__ AssembleArgs a, const double* __restrict__ u_sub,
                                    double* __restrict__ u) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = blockIdx.y;
  if (I >= a.NXg) return;
  int sx1 = I / a.snxP, sx0 = sx1;
  if (sx1 >= a.Sx) { sx1 = a.Sx - 1; sx0 = sx1; }
  else if (I % a.snxP == 0 && I > 0) sx0 = sx1 - 1;
  int sy1 = J / a.snyP, sy0 = sy1;
  if (sy1 >= a.Sy) { sy1 = a.Sy - 1; sy0 = sy1; }
  else if (J % a.snyP == 0 && J > 0) sy0 = sy1 - 1;
  const double uniform = 1.0 / (double)((sx1 - sx0 + 1) * (sy1 - sy0 + 1));
  const int64_t nn = (int64_t)a.nlx * a.nly;
  double sr = 0.0, si = 0.0;
  for (int sy = sy0; sy <= sy1; ++sy)
    for (int sx = sx0; sx <= sx1; ++sx) {
      const int l = sy * a.Sx + sx;
      const int i = I - sx * a.snxP, j = J - sy * a.snyP;
      const int64_t k = (int64_t)l * nn + (int64_t)j * a.nlx + i;
      const double sh = a.share ? a.share[k] : 1.0;
      sr += sh * u_sub[2 * k];
      si += sh * u_sub[2 * k + 1];
    }
  const double scale = a.share ? 1.0 : uniform;
  const int64_t n = (int64_t)J * a.NXg + I;
  u[2 * n] += scale * sr;
  u[2 * n + 1] += scale * si;
}

// ---- Krylov vector kernels (vectors of n2 doubles = n2/2 complex values)
// On this part FP64 arithmetic, not memory, bounds these kernels (the FP64
// pipe retires about 1/65 of the FP32 rate), so they are written for the
// fewest FP64 instructions: every complex multiply-accumulate is four fma()
// (no separate multiply and add), the real variants skip the imaginary half,
// and the difference w = v - S v and the final norm ride along with the dot
// and update passes instead of running as passes of their own.
//
// multi_dot: one block per contiguous chunk of the vectors: the chunk of w is
// staged in shared memory once, then the block's warps take the basis vectors
// in turn (coalesced reads of each V_k chunk, two accumulator pairs per lane,
// one warp reduction per vector), so every element of V and w is read from
// memory once per call.  part[(blk * nv + k) * 2 + {0, 1}].
constexpr int kDotWarps = 8;
template <bool REAL, bool DIFF>
__global__ void __launch_bounds__(kDotWarps * 32)
    multi_dot_kernel(const double* __restrict__ V, int64_t ld, int nv, const double* __restrict__ w,
                     const double* __restrict__ w_sub, double* __restrict__ w_out, int64_t nc, int chunk,
                     double* __restrict__ part) {
  extern __shared__ double2 ws[];
  const int64_t r0 = (int64_t)blockIdx.x * chunk;
  const int rows = (int)((nc - r0) < chunk ? (nc - r0) : chunk);
  for (int q = threadIdx.x; q < rows; q += blockDim.x) {
    double2 x = reinterpret_cast<const double2*>(w)[r0 + q];
    if (DIFF) {
      const double2 y = reinterpret_cast<const double2*>(w_sub)[r0 + q];
      x.x -= y.x;
      x.y -= y.y;
      reinterpret_cast<double2*>(w_out)[r0 + q] = x;
    }
    ws[q] = x;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int k = warp; k < nv; k += kDotWarps) {
    const double2* vk = reinterpret_cast<const double2*>(V + (int64_t)k * ld) + r0;
    // conj(a) b = (a.x b.x + a.y b.y) + i (a.x b.y - a.y b.x)
    double sr0 = 0.0, si0 = 0.0, sr1 = 0.0, si1 = 0.0;
    int q = lane;
#pragma unroll 2
    for (; q + 32 < rows; q += 64) {
      const double2 a = vk[q], b = ws[q], c = vk[q + 32], d = ws[q + 32];
      sr0 = fma(a.x, b.x, sr0);
      sr0 = fma(a.y, b.y, sr0);
      sr1 = fma(c.x, d.x, sr1);
      sr1 = fma(c.y, d.y, sr1);
      if (!REAL) {
        si0 = fma(a.x, b.y, si0);
        si0 = fma(-a.y, b.x, si0);
        si1 = fma(c.x, d.y, si1);
        si1 = fma(-c.y, d.x, si1);
      }
    }
    if (q < rows) {
      const double2 a = vk[q], b = ws[q];
      sr0 = fma(a.x, b.x, sr0);
      sr0 = fma(a.y, b.y, sr0);
      if (!REAL) {
        si0 = fma(a.x, b.y, si0);
        si0 = fma(-a.y, b.x, si0);
      }
    }
    const double sr = warp_sum(sr0 + sr1);
    const double si = REAL ? 0.0 : warp_sum(si0 + si1);
    if (lane == 0) {
      double* p = part + ((int64_t)blockIdx.x * nv + k) * 2;
      p[0] = sr;
      p[1] = si;
    }
  }
}

// w -= sum_k h_k V_k, one complex entry per thread and iteration, basis
// vectors taken two at a time into separate accumulators; NORM: the block's
// partial ||w_new||^2 into norm_part[2 blk] (0 into norm_part[2 blk + 1]).
template <bool REAL, bool NORM>
__global__ void multi_axpy_kernel(const double* __restrict__ V, int64_t ld, int nv, const double* __restrict__ h,
                                  double* __restrict__ w, int64_t nc, double* __restrict__ norm_part) {
  extern __shared__ double hs[];
  for (int k = threadIdx.x; k < 2 * nv; k += blockDim.x) hs[k] = h[k];
  __syncthreads();
  double2* w2 = reinterpret_cast<double2*>(w);
  double nrm[1] = {0.0};
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nc; q += (int64_t)gridDim.x * blockDim.x) {
    // (hr + i hi)(v.x + i v.y) = (hr v.x - hi v.y) + i (hr v.y + hi v.x)
    double2 acc = w2[q], acc1 = make_double2(0.0, 0.0);
    int k = 0;
#pragma unroll 2
    for (; k + 1 < nv; k += 2) {
      const double2 v = reinterpret_cast<const double2*>(V + (int64_t)k * ld)[q];
      const double2 u = reinterpret_cast<const double2*>(V + (int64_t)(k + 1) * ld)[q];
      const double hr = hs[2 * k], hr1 = hs[2 * k + 2];
      acc.x = fma(-hr, v.x, acc.x);
      acc.y = fma(-hr, v.y, acc.y);
      acc1.x = fma(-hr1, u.x, acc1.x);
      acc1.y = fma(-hr1, u.y, acc1.y);
      if (!REAL) {
        const double hi = hs[2 * k + 1], hi1 = hs[2 * k + 3];
        acc.x = fma(hi, v.y, acc.x);
        acc.y = fma(-hi, v.x, acc.y);
        acc1.x = fma(hi1, u.y, acc1.x);
        acc1.y = fma(-hi1, u.x, acc1.y);
      }
    }
    if (k < nv) {
      const double2 v = reinterpret_cast<const double2*>(V + (int64_t)k * ld)[q];
      const double hr = hs[2 * k];
      acc.x = fma(-hr, v.x, acc.x);
      acc.y = fma(-hr, v.y, acc.y);
      if (!REAL) {
        const double hi = hs[2 * k + 1];
        acc.x = fma(hi, v.y, acc.x);
        acc.y = fma(-hi, v.x, acc.y);
      }
    }
    acc.x += acc1.x;
    acc.y += acc1.y;
    w2[q] = acc;
    if (NORM) nrm[0] = fma(acc.x, acc.x, fma(acc.y, acc.y, nrm[0]));
  }
  if (NORM) {
    __shared__ double res[1];
    block_sum<1>(nrm, res);
    if (threadIdx.x == 0) {
      norm_part[2 * blockIdx.x] = res[0];
      norm_part[2 * blockIdx.x + 1] = 0.0;
    }
  }
}

__global__ void axpby_kernel(double a, const double* __restrict__ x, double b, double* __restrict__ y, int64_t n2) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n2; q += (int64_t)gridDim.x * blockDim.x)
    y[q] = a * x[q] + b * y[q];
}

// y = x / sqrt(n2[0]) (0 if the norm is 0): normalises the next Krylov vector
// on the device, without a round trip to the host (y may be x).  With flags_src
// the solve's 4 status words are staged beside the Hessenberg column, so one
// device-to-host copy carries both.
__global__ void scale_inv_norm_kernel(const double* x, const double* __restrict__ n2, double* y, int64_t n,
                                      const int* __restrict__ flags_src, int* __restrict__ flags_dst) {
  if (flags_src && blockIdx.x == 0 && threadIdx.x < 4) flags_dst[threadIdx.x] = flags_src[threadIdx.x];
  const double v = n2[0];
  const double s = v > 0.0 ? 1.0 / sqrt(v) : 0.0;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    y[q] = s * x[q];
}

int grid_for(int64_t n, int threads) {
  int64_t g = (n + threads - 1) / threads;
  const int64_t cap = (int64_t)sm_count() * 8;  // 8 resident blocks of 256 threads per SM
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

// Blocks of the residual kernel: element columns x node rows, then the last node column.
int residual_main_blocks(const GlobalArgs& a) { return (a.nx + 31) / 32 * ((a.NYg + kResRows - 1) / kResRows); }

template <int P>
hz_status launch_residual_P(const GlobalArgs& a, const double* b, const double* u, double* r, double* part,
                            unsigned* ticket, double* norms2, cudaStream_t st) {
  // a caller's array off the 16-byte grid: entries as two doubles each
  const bool pair = is_pair_aligned(b) && is_pair_aligned(u) && is_pair_aligned(r);
  auto kern = pair ? residual_kernel<P, true> : residual_kernel<P, false>;
  kern<<<residual_blocks(a), 32 * kResRows, 0, st>>>(a, (a.nx + 31) / 32, residual_main_blocks(a), b, u, r, part, ticket,
                                                     norms2);
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

}  // namespace

hz_status launch_prepare(const PrepArgs& a, int L, cudaStream_t st) {
  const int nn = a.nlx * a.nly;
  dim3 grd((nn + 255) / 256, L);
  prepare_kernel<<<grd, 256, 0, st>>>(a);
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_rhs(const GlobalArgs& a, const double* f, const double* gb, double* b, cudaStream_t st) {
  dim3 grd((a.NXg + 127) / 128, a.NYg);
  rhs_kernel<<<grd, 128, 0, st>>>(a, f, gb, b);
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

int residual_blocks(const GlobalArgs& a) {
  return residual_main_blocks(a) + (a.NYg + 32 * kResRows - 1) / (32 * kResRows);
}

hz_status launch_residual(const GlobalArgs& a, const double* b, const double* u, double* r, double* part,
                          unsigned* ticket, double* norms2, cudaStream_t st) {
  switch (a.P) {
    case 1: return launch_residual_P<1>(a, b, u, r, part, ticket, norms2, st);
    case 2: return launch_residual_P<2>(a, b, u, r, part, ticket, norms2, st);
    case 3: return launch_residual_P<3>(a, b, u, r, part, ticket, norms2, st);
    case 4: return launch_residual_P<4>(a, b, u, r, part, ticket, norms2, st);
    case 5: return launch_residual_P<5>(a, b, u, r, part, ticket, norms2, st);
    case 6: return launch_residual_P<6>(a, b, u, r, part, ticket, norms2, st);
    case 7: return launch_residual_P<7>(a, b, u, r, part, ticket, norms2, st);
    default: return fail(HZ_ERR_UNSUPPORTED, "degree outside 1..7");
  }
}

hz_status launch_reduce_partials(const double* part, int nblocks, int width, double* out, cudaStream_t st) {
  reduce_partials_kernel<<<width, kRedThreads, 0, st>>>(part, nblocks, width, out);
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_assemble_add(const AssembleArgs& a, const double* u_sub, double* u, cudaStream_t st) {
  dim3 grd((a.NXg + 127) / 128, a.NYg);
  assemble_add_kernel<<<grd, 128, 0, st>>>(a, u_sub, u);
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

int sm_count() {
  constexpr int kMaxDev = 64;
  static std::atomic<int> cache[kMaxDev];  // 0 = not looked up yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
    (void)cudaGetLastError();
    return 1;  // grid-stride kernels stay correct with any grid
  }
  int v = cache[dev].load(std::memory_order_relaxed);
  if (v > 0) return v;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) {
    (void)cudaGetLastError();
    v = 1;
  }
  cache[dev].store(v, std::memory_order_relaxed);
  return v;
}

// blocks for multi_dot: 2 per SM, chunks of at most 4096 complex entries (64 KB of shared memory)
int vec_blocks(int64_t n2) {
  const int64_t nc = n2 / 2;
  int64_t nb = 2 * (int64_t)sm_count();
  if ((nc + nb - 1) / nb > 4096) nb = (nc + 4095) / 4096;
  if (nb > nc) nb = nc > 0 ? nc : 1;
  return (int)nb;
}

template <bool REAL, bool DIFF>
hz_status launch_multi_dot_T(const double* V, int64_t ld, int nv, const double* w, const double* w_sub, double* w_out,
                             int64_t nc, int chunk, size_t smem, double* part, int nblocks, cudaStream_t st) {
  if (smem > 48 * 1024)
    HZ_CUDA(cudaFuncSetAttribute(multi_dot_kernel<REAL, DIFF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  multi_dot_kernel<REAL, DIFF><<<nblocks, kDotWarps * 32, smem, st>>>(V, ld, nv, w, w_sub, w_out, nc, chunk, part);
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_multi_dot(const double* V, int64_t ld, int nv, const double* w, const double* w_sub, double* w_out,
                           int64_t n2, bool real_dot, double* part, int nblocks, cudaStream_t st) {
  if ((w_sub == nullptr) != (w_out == nullptr)) return fail(HZ_ERR_INVALID_ARG, "multi_dot: w_sub and w_out go together");
  const int64_t nc = n2 / 2;
  const int chunk = (int)((nc + nblocks - 1) / nblocks);
  const size_t smem = (size_t)chunk * sizeof(double2);
  if (real_dot)
    return w_sub ? launch_multi_dot_T<true, true>(V, ld, nv, w, w_sub, w_out, nc, chunk, smem, part, nblocks, st)
                 : launch_multi_dot_T<true, false>(V, ld, nv, w, w_sub, w_out, nc, chunk, smem, part, nblocks, st);
  return w_sub ? launch_multi_dot_T<false, true>(V, ld, nv, w, w_sub, w_out, nc, chunk, smem, part, nblocks, st)
               : launch_multi_dot_T<false, false>(V, ld, nv, w, w_sub, w_out, nc, chunk, smem, part, nblocks, st);
}

int axpy_blocks(int64_t n2) { return grid_for(n2 / 2, 256); }

hz_status launch_multi_axpy(const double* V, int64_t ld, int nv, const double* h, double* w, int64_t n2,
                            bool real_coef, cudaStream_t st, double* norm_part) {
  const int64_t nc = n2 / 2;
  const int g = axpy_blocks(n2);
  const size_t smem = (size_t)2 * nv * sizeof(double);
  if (smem > 48 * 1024) {
    // nv above 3072 basis vectors: not reachable with the restart bound, refuse rather than launch
    return fail(HZ_ERR_UNSUPPORTED, "multi_axpy: too many basis vectors");
  }
  if (real_coef) {
    if (norm_part) multi_axpy_kernel<true, true><<<g, 256, smem, st>>>(V, ld, nv, h, w, nc, norm_part);
    else multi_axpy_kernel<true, false><<<g, 256, smem, st>>>(V, ld, nv, h, w, nc, nullptr);
  } else {
    if (norm_part) multi_axpy_kernel<false, true><<<g, 256, smem, st>>>(V, ld, nv, h, w, nc, norm_part);
    else multi_axpy_kernel<false, false><<<g, 256, smem, st>>>(V, ld, nv, h, w, nc, nullptr);
  }
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_scale_inv_norm(const double* x, const double* norm2, double* y, int64_t n2, cudaStream_t st,
                                const int* flags_src, int* flags_dst) {
  scale_inv_norm_kernel<<<grid_for(n2, 256), 256, 0, st>>>(x, norm2, y, n2, flags_src, flags_dst);
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

// One thread per complex entry of the listed slots; slot k occupies entries
// [k NE, (k+1) NE) of the packed buffer.  A slot (l, e) outside the lambda
// vector (l not in 0..L-1 or e not in 0..3) is skipped: gather writes zeros
// for it, scatter writes nothing.
template <bool PAIR>
__global__ void lambda_slots_kernel(const int32_t* __restrict__ slots, int count, int NE, int L, const double* src,
                                    double* dst, int gather) {
  const int64_t total = (int64_t)count * NE;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
    const int k = (int)(q / NE), t = (int)(q % NE);
    const int l = slots[2 * k], e = slots[2 * k + 1];
    const bool ok = l >= 0 && l < L && e >= 0 && e < 4;
    const int64_t slot = ((int64_t)l * 4 + e) * NE + t;
    if (gather) store_complex<PAIR>(dst, q, ok ? load_complex<PAIR>(src, slot) : make_double2(0.0, 0.0));
    else if (ok) store_complex<PAIR>(dst, slot, load_complex<PAIR>(src, q));
  }
}

hz_status launch_lambda_slots(const int32_t* slots, int count, int NE, int L, const double* src, double* dst,
                              bool gather, cudaStream_t st) {
  const int64_t total = (int64_t)count * NE;
  auto kern = is_pair_aligned(src) && is_pair_aligned(dst) ? lambda_slots_kernel<true> : lambda_slots_kernel<false>;
  kern<<<grid_for(total, 256), 256, 0, st>>>(slots, count, NE, L, src, dst, gather ? 1 : 0);
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_axpby(double a, const double* x, double b, double* y, int64_t n2, cudaStream_t st) {
  axpby_kernel<<<grid_for(n2, 256), 256, 0, st>>>(a, x, b, y, n2);
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

}  // namespace hz
