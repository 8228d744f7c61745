// Element-form DD sweep on curved quadrilaterals (FP32, P <= 4), one element
// per thread: the thread keeps the (P+1)^2 nodes of its element, their metric
// and their wave state in registers for the whole WaveHoltz loop, so that the
// gradient, the fluxes and the contraction D^T F (Sec. 4, Sec. 6.1) are FMAs
// on registers with constant-bank coefficients.
//
// A node shared by several elements is kept by each of them.  Per time step
// the elements exchange their contributions to A p along their edges, first
// with the x neighbours (lanes of the same warp: shuffles), then the row sums
// with the y neighbours (shared memory, one barrier per step, double-buffered
// by step parity).  Every copy of a node adds the same two pairs of numbers,
// (a + b) + (c + d) up to the order inside a sum, so the copies agree bitwise
// and only the contributions travel, never p.
//
// Bound: the FMA pipe (41 FMAs per node and step at P = 3, counting the copies
// of shared nodes).  The one-thread-per-node kernel (hz_sweep_mapped.cuh)
// moves every operand of the two contractions through shared memory, with two
// or three barriers per step: 1024 subdomains of 25 x 25 nodes, P = 3, N_t = 74,
// 10 WaveHoltz iterations: 4353 us there, 1127 us here (43% of the FP32 rate).
#pragma once

#include <cuda_runtime.h>

#include "hz_complex_io.cuh"
#include "hz_internal.h"
#include "hz_norm_acc.cuh"

namespace hz {
namespace mapped_tile {

struct Args {
  MappedSweepArgs m;
  float D[(kMaxP + 1) * (kMaxP + 1)];
  int count;
  int LX, lxs;   // element columns of the lane grid (a power of two), its log2
  int spw, gs;   // one-warp subdomains: subdomains per warp, lanes per subdomain
};

// Shared memory of one subdomain, in floats (4-float aligned parts).
struct Lay {
  int ex;       // [2][sny][2][M][LX]: row sums of each element's first and last node row
  int tw, te;   // edge tables, west and east column by row: alpha - 1, beta b (re, im), gamma
  int ts, tn;   // south and north row by column (zero at the corners: in tw, te)
  int src;      // [nl][2]: beta x source (with a source only)
  int stash;    // previous iterate (tolerance mode)
  int total;
};
__host__ __device__ inline Lay make_lay(int P, int LX, int nlx, int nly, int sny, int threads, bool src, bool tol) {
  const int M = P + 1;
  Lay y;
  int o = 0;
  y.ex = o; o += 2 * sny * 2 * M * LX;
  y.tw = o; o += 4 * nly;
  y.te = o; o += 4 * nly;
  y.ts = o; o += 4 * nlx;
  y.tn = o; o += 4 * nlx;
  y.src = o; if (src) o += 2 * nlx * nly;
  y.stash = o; if (tol) o += 2 * M * M * threads;
  y.total = (o + 3) / 4 * 4;
  return y;
}

template <int P, bool ONE, bool SRC>
__global__ void __launch_bounds__(ONE ? 32 : 256) sweep_mapped_tile_kernel(const __grid_constant__ Args x) {
  constexpr int M = P + 1, N2 = M * M;
  const SweepArgs& a = x.m.base;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[8][2];
  __shared__ int stop;
  const int lane = threadIdx.x & 31;
  const int grp = ONE ? lane / x.gs : 0;
  const int k0 = ONE ? blockIdx.x * x.spw + grp : blockIdx.x;
  const bool have = k0 < x.count;
  const int l = sweep_subdomain(a, have ? k0 : 0);
  const int sxi = l % a.Sx, syi = l / a.Sx;
  const int nlx = a.nlx, nly = a.nly, snx = x.m.snx, sny = x.m.sny;
  const int t = ONE ? lane - grp * x.gs : (int)threadIdx.x;
  const int nthr = ONE ? x.gs : (int)blockDim.x;
  const int ex = t & (x.LX - 1), ey = t >> x.lxs;
  const bool live = have && ex < snx && ey < sny;
  const int exc = live ? ex : 0, eyc = live ? ey : 0;
  const bool tol = a.wh_tol > 0.0;
  const Lay y = make_lay(P, x.LX, nlx, nly, sny, nthr, SRC, tol);
  float* sm = reinterpret_cast<float*>(smem_raw) + (ONE ? grp * y.total : 0);

  const int64_t nn = (int64_t)nlx * nly;
  const float* betaG = static_cast<const float*>(a.beta) + (int64_t)l * nn;
  const float* alphaG = static_cast<const float*>(a.alpha) + (int64_t)l * nn;
  const double* lamL = a.lam_in + (int64_t)l * 4 * a.NE * 2;
  const double* kedgeL = a.kedge + (int64_t)l * 4 * a.NE;
  const double* wE = x.m.wedge + (int64_t)l * 4 * a.NE;
  const bool ifW = sxi > 0, ifE = sxi < a.Sx - 1, ifS = syi > 0, ifN = syi < a.Sy - 1;

  for (int q = t; q < y.tw; q += nthr) sm[q] = 0.f;
  // ---- edge tables, one edge node per thread
  for (int q = t; q < 2 * (nlx + nly); q += nthr) {
    int i, j;
    float* dst;
    bool own = true;  // a corner belongs to its column
    if (q < nly) { i = 0; j = q; dst = sm + y.tw + 4 * j; }
    else if (q < 2 * nly) { i = nlx - 1; j = q - nly; dst = sm + y.te + 4 * j; }
    else {
      i = (q - 2 * nly) % nlx;
      j = q - 2 * nly < nlx ? 0 : nly - 1;
      dst = sm + (j == 0 ? y.ts : y.tn) + 4 * i;
      own = i > 0 && i < nlx - 1;
    }
    const int64_t n = (int64_t)j * nlx + i;
    const double be = (double)betaG[n];
    double br = 0.0, bi = 0.0, hm = 0.0;
    auto edge = [&](int e, int k) {
      const double w = wE[e * a.NE + k];
      br += w * lamL[2 * (e * a.NE + k)];
      bi += w * lamL[2 * (e * a.NE + k) + 1];
      hm += w * kedgeL[e * a.NE + k];
    };
    if (i == 0 && ifW) edge(0, j);
    if (i == nlx - 1 && ifE) edge(1, j);
    if (j == 0 && ifS) edge(2, i);
    if (j == nly - 1 && ifN) edge(3, i);
    dst[0] = own ? (float)((double)alphaG[n] - 1.0) : 0.f;
    dst[1] = own ? (float)(be * br) : 0.f;
    dst[2] = own ? (float)(be * bi) : 0.f;
    dst[3] = own ? (float)(-be * a.eta * hm) : 0.f;  // interface boundary mass
  }
  if (SRC) {
    for (int q = t; q < (int)nn; q += nthr) {
      const int i = q % nlx, j = q / nlx;
      const int64_t I = (int64_t)sxi * a.snxP + i, J = (int64_t)syi * a.snyP + j;
      const double sh = x.m.share[(int64_t)l * nn + q] * (double)betaG[q];
      sm[y.src + 2 * q] = (float)(sh * a.rhs[2 * (J * a.NXg + I)]);
      sm[y.src + 2 * q + 1] = (float)(sh * a.rhs[2 * (J * a.NXg + I) + 1]);
    }
  }

  // ---- the element's metric and coefficients
  float g0[M][M], g1[M][M], g2[M][M], nbet[M][M];
#pragma unroll
  for (int b = 0; b < M; ++b)
#pragma unroll
    for (int c = 0; c < M; ++c) {
      g0[b][c] = g1[b][c] = g2[b][c] = nbet[b][c] = 0.f;
      if (live) {
        const float* g = static_cast<const float*>(x.m.geo) + (((int64_t)l * sny + ey) * snx + ex) * N2 * 3 + 3 * (b * M + c);
        g0[b][c] = g[0];
        g1[b][c] = g[1];
        g2[b][c] = g[2];
        nbet[b][c] = -betaG[(int64_t)(ey * P + b) * nlx + ex * P + c];
      }
    }
  const bool firstx = live && ex == 0, lastx = live && ex == snx - 1;
  const bool firsty = live && ey == 0, lasty = live && ey == sny - 1;
  const float ml = live && ex > 0 ? 1.f : 0.f, mr = live && ex < snx - 1 ? 1.f : 0.f;
  const float mb = live && ey > 0 ? 1.f : 0.f, mt = live && ey < sny - 1 ? 1.f : 0.f;
  const int eb = live && ey > 0 ? ey - 1 : eyc, et = live && ey < sny - 1 ? ey + 1 : eyc;

  const float4* tab = static_cast<const float4*>(a.tab);
  const float sigma = (float)a.sigma, omega = (float)a.omega;
  const float cpi = (float)a.cpi, spi = (float)a.spi, scale = (float)a.two_over_nt;
  float2 s[M][M], v[M][M];  // p, p-dot; the filter sums
#pragma unroll
  for (int b = 0; b < M; ++b)
#pragma unroll
    for (int c = 0; c < M; ++c) {
      v[b][c] = make_float2(0.f, 0.f);
      if (a.u0 && live) {  // warm start
        const int64_t n = (int64_t)l * nn + (int64_t)(ey * P + b) * nlx + ex * P + c;
        v[b][c] = make_float2((float)a.u0[2 * n], (float)a.u0[2 * n + 1]);
      }
    }
  if (ONE) __syncwarp();
  else __syncthreads();

  // row buffers: [parity][element row][first / last node row][node][element column]
  const int rstr = x.LX * M, par = sny * 2 * rstr;
  auto st_row = [&](float* buf, const float (&r)[M]) {
    if constexpr (M == 4) reinterpret_cast<float4*>(buf)[exc] = make_float4(r[0], r[1], r[2], r[3]);
    else if constexpr (M == 2) reinterpret_cast<float2*>(buf)[exc] = make_float2(r[0], r[1]);
    else
#pragma unroll
      for (int c = 0; c < M; ++c) buf[c * x.LX + exc] = r[c];
  };
  auto ld_row = [&](const float* buf, float (&r)[M]) {
    if constexpr (M == 4) {
      const float4 q = reinterpret_cast<const float4*>(buf)[exc];
      r[0] = q.x; r[1] = q.y; r[2] = q.z; r[3] = q.w;
    } else if constexpr (M == 2) {
      const float2 q = reinterpret_cast<const float2*>(buf)[exc];
      r[0] = q.x; r[1] = q.y;
    } else {
#pragma unroll
      for (int c = 0; c < M; ++c) r[c] = buf[c * x.LX + exc];
    }
  };

  int cur = 0, m_done = 0;
  bool done = false;
  for (int m = 0; m < a.m_wh; ++m) {
    if (tol) {
      float* st = sm + y.stash;
#pragma unroll
      for (int k = 0; k < N2; ++k) {
        st[(2 * k) * nthr + t] = v[k / M][k % M].x;
        st[(2 * k + 1) * nthr + t] = v[k / M][k % M].y;
      }
    }
    {
      const float4 t0 = tab[0];
#pragma unroll
      for (int b = 0; b < M; ++b)
#pragma unroll
        for (int c = 0; c < M; ++c) {
          s[b][c].x = v[b][c].x;
          s[b][c].y = omega * (v[b][c].y * cpi - v[b][c].x * spi);  // Re{-i w u e^{-i pi/N_t}}
          v[b][c].x = t0.z * s[b][c].x;
          v[b][c].y = t0.w * s[b][c].y;
        }
    }
    float4 tb = tab[1];
    for (int nu = 1; nu < a.Nt; ++nu) {
      const float4 tn = tab[nu + 1];  // prefetch (the table has N_t + 1 entries)
#pragma unroll
      for (int b = 0; b < M; ++b)
#pragma unroll
        for (int c = 0; c < M; ++c) s[b][c].x = fmaf(sigma, s[b][c].y, s[b][c].x);
      // element contributions A_e p, one node row of fluxes at a time
      float A[M][M];
#pragma unroll
      for (int q = 0; q < M; ++q) {
        float f1[M], f2[M], ux[M], ue[M];
#pragma unroll
        for (int k = 0; k < M; ++k)
#pragma unroll
          for (int c = 0; c < M; ++c) {
            ux[c] = k == 0 ? x.D[c * M] * s[q][0].x : fmaf(x.D[c * M + k], s[q][k].x, ux[c]);
            ue[c] = k == 0 ? x.D[q * M] * s[0][c].x : fmaf(x.D[q * M + k], s[k][c].x, ue[c]);
          }
#pragma unroll
        for (int c = 0; c < M; ++c) {
          f1[c] = fmaf(g1[q][c], ue[c], g0[q][c] * ux[c]);
          f2[c] = fmaf(g2[q][c], ue[c], g1[q][c] * ux[c]);
        }
#pragma unroll
        for (int b = 0; b < M; ++b)
#pragma unroll
          for (int c = 0; c < M; ++c) A[b][c] = q == 0 ? x.D[b] * f2[c] : fmaf(x.D[q * M + b], f2[c], A[b][c]);
        // x part of row q: may come after the first y terms of it only for q > 0
#pragma unroll
        for (int k = 0; k < M; ++k)
#pragma unroll
          for (int c = 0; c < M; ++c) A[q][c] = fmaf(x.D[k * M + c], f1[k], A[q][c]);
      }
      // x neighbours (by rows of elements: the ends multiply what they get by
      // zero, which may not be another subdomain's infinity or NaN), then the
      // row sums to the y neighbours
      const int width = ONE ? x.LX : 32;
#pragma unroll
      for (int b = 0; b < M; ++b) {
        const float fr = __shfl_down_sync(0xffffffffu, A[b][0], 1, width);
        const float fl = __shfl_up_sync(0xffffffffu, A[b][P], 1, width);
        A[b][0] = fmaf(ml, fl, A[b][0]);
        A[b][P] = fmaf(mr, fr, A[b][P]);
      }
      float* X = sm + y.ex + cur * par;
      if (live) {
        st_row(X + (2 * ey) * rstr, A[0]);
        st_row(X + (2 * ey + 1) * rstr, A[P]);
      }
      if (ONE) __syncwarp();
      else __syncthreads();
      float rb[M], rt[M];
      ld_row(X + (2 * eb + 1) * rstr, rb);
      ld_row(X + (2 * et) * rstr, rt);
#pragma unroll
      for (int c = 0; c < M; ++c) {
        A[0][c] = fmaf(mb, rb[c], A[0][c]);
        A[P][c] = fmaf(mt, rt[c], A[P][c]);
      }
      // subdomain edges: (alpha - 1) p-dot + beta b + gamma p
      auto fix = [&](float2& q, const float* w) {
        const float4 e = *reinterpret_cast<const float4*>(w);
        q.y = fmaf(e.x, q.y, fmaf(e.y, tb.x, fmaf(e.z, tb.y, fmaf(e.w, q.x, q.y))));
      };
      if (firstx) {
#pragma unroll
        for (int b = 0; b < M; ++b) fix(s[b][0], sm + y.tw + 4 * (ey * P + b));
      }
      if (lastx) {
#pragma unroll
        for (int b = 0; b < M; ++b) fix(s[b][P], sm + y.te + 4 * (ey * P + b));
      }
      if (firsty) {
#pragma unroll
        for (int c = 0; c < M; ++c) fix(s[0][c], sm + y.ts + 4 * (ex * P + c));
      }
      if (lasty) {
#pragma unroll
        for (int c = 0; c < M; ++c) fix(s[P][c], sm + y.tn + 4 * (ex * P + c));
      }
#pragma unroll
      for (int b = 0; b < M; ++b)
#pragma unroll
        for (int c = 0; c < M; ++c) {
          if (SRC) {
            const float2 f = *reinterpret_cast<const float2*>(sm + y.src + 2 * ((eyc * P + b) * nlx + exc * P + c));
            s[b][c].y = fmaf(f.x, tb.x, fmaf(f.y, tb.y, s[b][c].y));
          }
          s[b][c].y = fmaf(nbet[b][c], A[b][c], s[b][c].y);
          v[b][c] = __ffma2_rn(make_float2(tb.z, tb.w), s[b][c], v[b][c]);
        }
      tb = tn;
      cur ^= 1;
    }
#pragma unroll
    for (int b = 0; b < M; ++b)
#pragma unroll
      for (int c = 0; c < M; ++c) {
        v[b][c].x *= scale;  // u^{(m+1)} = (2/N_t) v
        v[b][c].y *= scale;
      }
    if (!done) m_done = m + 1;
    if (tol) {
      // per-subdomain stop; a shared node counts once, for the element it starts
      const float* st = sm + y.stash;
      double dn = 0.0, un = 0.0;
      NormAcc acc;
      float big = 0.f;
#pragma unroll
      for (int k = 0; k < N2; ++k)
        big = fmaxf(fmaxf(big, fmaxf(fabsf(v[k / M][k % M].x), fabsf(v[k / M][k % M].y))),
                    fmaxf(fabsf(st[(2 * k) * nthr + t]), fabsf(st[(2 * k + 1) * nthr + t])));
      acc.start(big);
#pragma unroll
      for (int b = 0; b < M; ++b)
#pragma unroll
        for (int c = 0; c < M; ++c) {
          const int k = b * M + c;
          const float orr = st[(2 * k) * nthr + t], oi = st[(2 * k + 1) * nthr + t];
          if (live && (c < P || lastx) && (b < P || lasty)) {
            acc.add(v[b][c], make_float2(orr, oi));
          }
          if (done) v[b][c] = make_float2(orr, oi);
        }
      acc.finish(dn, un);
      if (ONE) {
        for (int o = x.gs >> 1; o > 0; o >>= 1) {
          dn += __shfl_xor_sync(0xffffffffu, dn, o);
          un += __shfl_xor_sync(0xffffffffu, un, o);
        }
        if (dn <= a.wh_tol * a.wh_tol * un) done = true;
        if (__all_sync(0xffffffffu, done || !have)) break;
      } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          dn += __shfl_xor_sync(0xffffffffu, dn, o);
          un += __shfl_xor_sync(0xffffffffu, un, o);
        }
        if (lane == 0) {
          red[threadIdx.x >> 5][0] = dn;
          red[threadIdx.x >> 5][1] = un;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
          double D = 0.0, U = 0.0;
          for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            D += red[w][0];
            U += red[w][1];
          }
          stop = (D <= a.wh_tol * a.wh_tol * U) ? 1 : 0;
        }
        __syncthreads();
        if (stop) break;
      }
    }
  }

  // ---- outputs: a shared node is written by the element it starts
  bool bad = false;
  if (live) {
#pragma unroll
    for (int b = 0; b < M; ++b)
#pragma unroll
      for (int c = 0; c < M; ++c) {
        if (!isfinite(v[b][c].x) || !isfinite(v[b][c].y)) bad = true;
        if (a.u_sub && (c < P || lastx) && (b < P || lasty))
          store_complex(a.u_sub, (int64_t)l * nn + (int64_t)(ey * P + b) * nlx + ex * P + c,
                        make_double2(v[b][c].x, v[b][c].y));
      }
  }
  if (bad) atomicOr(a.flags, 1);
  if (t == 0 && have && a.wh_iter_max) {
    atomicMax(a.wh_iter_max, m_done);
    atomicAdd(a.wh_iter_sum, (unsigned long long)m_done);
  }
  // the edges' solutions in the edge tables' place (last read before the barrier)
  if (ONE) __syncwarp();
  else __syncthreads();
  auto stage = [&](int tabo, int q, float2 w) { *reinterpret_cast<float2*>(sm + tabo + 4 * q) = w; };
#pragma unroll
  for (int k = 0; k < M; ++k) {
    if (firstx) stage(y.tw, ey * P + k, v[k][0]);
    if (lastx) stage(y.te, ey * P + k, v[k][P]);
    if (firsty) stage(y.ts, ex * P + k, v[0][k]);
    if (lasty) stage(y.tn, ex * P + k, v[P][k]);
  }
  if (ONE) __syncwarp();
  else __syncthreads();
  if (have) {
    const int NE = a.NE;
    for (int k = t; k < 4 * NE; k += nthr) {
      const int ed = k / NE, q = k - ed * NE;
      const int len = ed < 2 ? nly : nlx;
      const bool iface = ed == 0 ? ifW : ed == 1 ? ifE : ed == 2 ? ifS : ifN;
      double2 w = make_double2(0.0, 0.0);
      int64_t dst = ((int64_t)l * 4 + ed) * NE + q;
      if (iface) {
        const int rn = ed == 0 ? l - 1 : ed == 1 ? l + 1 : ed == 2 ? l - a.Sx : l + a.Sx;
        dst = ((int64_t)rn * 4 + (ed ^ 1)) * NE + q;
        if (q < len) {
          const float* us = sm + (ed == 0 ? y.tw : ed == 1 ? y.te : ed == 2 ? y.ts : y.tn) + 4 * q;
          const double ur = (double)us[0], ui = (double)us[1];
          const double kk = kedgeL[ed * NE + q];
          const double2 lr = load_complex(lamL, ed * NE + q);
          // -lambda + 2 k (eta - i zeta) u
          w.x = -lr.x + 2.0 * kk * (a.eta * ur + a.zeta * ui);
          w.y = -lr.y + 2.0 * kk * (a.eta * ui - a.zeta * ur);
        }
      }
      store_complex(a.lam_out, dst, w);
    }
  }
}

template <int P, bool SRC>
hz_status launch_src(const MappedSweepArgs& m, int count, cudaStream_t st) {
  Args x{};
  x.m = m;
  for (int k = 0; k < (P + 1) * (P + 1); ++k) x.D[k] = (float)m.D[k];
  x.count = count;
  x.LX = tile_pow2(m.snx);
  while ((1 << x.lxs) < x.LX) ++x.lxs;
  const int lanes = x.LX * m.sny;
  const bool tol = m.base.wh_tol > 0.0;
  if (m.snx > 32 || lanes > 256) return HZ_ERR_UNSUPPORTED;
  const bool one = lanes <= 32;
  const int threads = one ? tile_pow2(lanes) : (lanes + 31) / 32 * 32;
  const Lay y = make_lay(P, x.LX, m.base.nlx, m.base.nly, m.sny, threads, SRC, tol);
  x.gs = threads;
  x.spw = one ? 32 / threads : 1;
  const size_t smem = (size_t)x.spw * y.total * sizeof(float);
  // the kernel's limit is this constant and not the launch's own size: another
  // thread's smaller launch would lower it between the two calls
  constexpr int kMaxSmem = 200 * 1024;
  if (smem > kMaxSmem) return HZ_ERR_UNSUPPORTED;
  auto kern = one ? sweep_mapped_tile_kernel<P, true, SRC> : sweep_mapped_tile_kernel<P, false, SRC>;
  if (smem > 48 * 1024) HZ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  kern<<<(count + x.spw - 1) / x.spw, one ? 32 : threads, smem, st>>>(x);
  note_launch();
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

template <int P>
hz_status launch(const MappedSweepArgs& m, int count, cudaStream_t st) {
  return m.base.rhs ? launch_src<P, true>(m, count, st) : launch_src<P, false>(m, count, st);
}

}  // namespace mapped_tile
}  // namespace hz
