// Column-strip solve: a persistent launch over (instance, column group) tasks.
//
// The columns of a block of random vectors are independent recursions
// (Eq. (rn) acts on each |r> separately), and one column of a small or
// mid-size lattice fits the shared memory of one SM.  A task is a few columns
// of one instance; a cluster of C CTAs (FP32: C = 1) takes tasks from a device
// queue and runs all products of its columns without touching global memory:
// v_n in one of two shared-memory buffers (read by neighbours, v_{n+1} goes to
// the other one), v_{n-1} and the thread's own v_n in registers.
//
// Layout.  The lattice is a stack of rows along its last dimension, each row a
// plane of U sites (2D: one lattice line, 3D: one xy-plane).  CTA q of the
// cluster owns a band of rows, cut into strips; a thread owns one plane
// position of one strip and keeps that column of up to H sites in registers.
// Neighbours along the last dimension are its own registers (the strip's two
// end neighbours are read once per product, through distributed shared memory
// where another CTA owns them); in-plane neighbours are conflict-free shared
// loads at offsets that are constant along the strip.  That leaves 2 (2D) or 4
// (3D) loads and one store of shared memory per site and product, and the
// loads of four sites are issued together.
//
// Arithmetic.  Each site's FMAs are in the order of the fused step, so v_{n+1}
// is bit for bit the fused step's.  The first product, (1/2) (2 H~) v_0, runs
// with halved coefficients (exact).
//
// Dots.  FP64: every thread adds its strip's terms as it computes them, and
// the threads' sums go through the lanes (xor 16 first: half a warp goes on
// with <v_n|v_n>, the other half with <v_{n+1}|v_n>), the warps and the CTAs.
// FP32: a compensated (Kahan) sum of FP32-rounded products depends on its
// order in its last digits (of order 1e-9 of a moment on the lattices that fit
// here), so the dots are taken in a second sweep over v_n and v_{n+1} in
// shared memory whose chains, lane trees and warp order are those of the
// global-memory batch form in its default configuration (clusters of four,
// chunks of four passes): the moments are that form's bit for bit.  The sweep
// runs in the phase of the next product (three buffers), so that one barrier
// serves both, and packs the two dots of a site into one f32x2 chain.
//
// The sum order depends on the layout and C alone, which depend on the
// instance alone: a column's moments do not depend on the other tasks.
//
// Measured (FP32, 256 uneven 2D instances of 16..128 sites a side, 16 vectors):
// 26.1 ms per batch against 38.7 for the global-memory form, whose products are
// chains of L2 round trips; 2.6 us per product and column of 96 x 96 sites, of
// which 1.1 the recursion, 0.8 the dot chains and 0.7 their reduction (timed with
// each left out in turn).  Bound by the latency of the chains at 16 warps per SM:
// issue 47 % active; of 6.8 warps' cycles per issue 2.2 wait on fixed latencies, 2.2
// at the barrier and 1.2 for shared memory.  A batch takes the form where it is
// estimated faster (cols_faster in kpm_batch_api.cu).
#pragma once

#include "kpm_cols.h"
#include "kpm_fixed.cuh"
#include "kpm_rng.cuh"
#include "kpm_step.cuh"

namespace kpm {
namespace cols {

constexpr int BT = COLS_THREADS;
constexpr int NW = BT / 32;

__device__ __forceinline__ float ldc(uint32_t a, float) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ double ldc(uint32_t a, double) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ long long ldc(uint32_t a, long long) {
  long long v;
  asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t map_addr(const void* p, uint32_t rank) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  uint32_t d;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(rank));
  return d;
}
__device__ __forceinline__ void arrive() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void wait() {
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// The two dots of a site, (<v_n|v_n>, <v_{n+1}|v_n>), as compensated pairs
// (value s - c).
struct Pair2 {
  float2 s, c;
};
__device__ __forceinline__ void dot1(Pair2& a, float x, float y) {
  kahan2(a.s, a.c, make_float2(__fmul_rn(x, x), __fmul_rn(y, x)));
}

// First row of CTA r's band when `rows` rows are split among C CTAs.
__device__ __forceinline__ int band0(int rows, int C, int r) {
  return (int)(((int64_t)rows * r) / C);
}

// ------------------------------------------------------------------ FP64
// All products of one task on this CTA (rank q of C), strips of at most H
// rows; strips are at least H - G rows high, so only the last G rows of a
// thread need a bounds test (H and G are even; sites go in groups of up to 4).
template <int DIMS, bool DS, int H, int G>
__device__ __noinline__ void run_rows(const ColsTask& k, int q, int C, unsigned char* smem) {
  using T = double;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int L = k.geom.L[DIMS - 1];            // rows of the whole lattice
  const int U = k.geom.stride[DIMS - 1];       // sites of a row
  const bool per = k.geom.periodic[DIMS - 1] != 0;
  const int ncol = k.ncol, S = k.strips, tpc = k.tpc;
  const int r0 = band0(L, C, q), B = band0(L, C, q + 1) - r0;
  const int BU = k.rows * U;                   // sites of the largest band: the column stride
  constexpr int NB = 2;                        // vector buffers
  T* buf = reinterpret_cast<T*>(smem);         // [NB][ncol][BU]
  const int bufn = ncol * BU;
  T* dsm = buf + (size_t)NB * bufn;            // [BU] scaled diagonal (DS)
  unsigned char* ring =
      smem + (((size_t)NB * bufn + (DS ? BU : 0)) * sizeof(T) + 15) / 16 * 16;
  const int kb = k.batch;                      // products per batch of the dot sums

  // this thread's column, strip and plane position
  const int cc = t / tpc, tt = t - cc * tpc;
  const int strip = tt / U, u = tt - strip * U;
  const bool have = cc < ncol && strip < S;
  const int y0 = have ? (int)(((int64_t)B * strip) / S) : 0;
  const int h = have ? (int)(((int64_t)B * (strip + 1)) / S) - y0 : 0;
  const bool act = h > 0;
  const int base = have ? cc * BU + y0 * U + u : 0;
  const int col = k.col0 + cc;

  T hu, hi_, du;
  scal_from_block<T>(k.sc, hu, hi_, du);
  // in-plane neighbours: offset and coefficient, constant along the strip
  int of[DIMS - 1], ob[DIMS - 1];
  T cf[DIMS - 1], cb[DIMS - 1];
  {
    int rem = u;
#pragma unroll
    for (int d = 0; d < DIMS - 1; ++d) {
      const int Ld = k.geom.L[d], st = k.geom.stride[d];
      const int x = rem % Ld;
      rem /= Ld;
      const bool p = k.geom.periodic[d] != 0;
      of[d] = (x + 1 < Ld) ? st : (p ? -(Ld - 1) * st : 0);
      ob[d] = (x > 0) ? -st : (p ? (Ld - 1) * st : 0);
      cf[d] = (x + 1 < Ld) || p ? hu : T(0);
      cb[d] = (x > 0) || p ? hu : T(0);
    }
  }
  // the rows before and after the strip: shared::cluster addresses of buffer 0
  uint32_t at = 0, ab = 0;
  T ct = T(0), cbm = T(0);
  if (act) {
    auto addr = [&](int y) {
      int r = q;
      if (y < r0 || y >= r0 + B)
        for (r = 0; r < C - 1; ++r)
          if (y < band0(L, C, r + 1)) break;
      return map_addr(buf + (size_t)cc * BU + (y - band0(L, C, r)) * U + u, (uint32_t)r);
    };
    const int yt = r0 + y0 - 1, yb = r0 + y0 + h;
    const bool ht = yt >= 0 || per, hb = yb < L || per;
    at = addr(ht ? (yt >= 0 ? yt : L - 1) : yt + 1);
    ab = addr(hb ? (yb < L ? yb : 0) : yb - 1);
    ct = ht ? hu : T(0);
    cbm = hb ? hu : T(0);
  }

  // start vectors
  T x[H], w[H];
  {
    const unsigned long long seed = k.prm ? k.prm->seed : k.seed;
    const unsigned long long s = (unsigned long long)(k.s + (k.prm ? k.prm->s0 : 0));
    const T* src = reinterpret_cast<const T*>(k.ds);
#pragma unroll
    for (int j = 0; j < H; ++j) {
      x[j] = w[j] = T(0);
      if (j < H - G ? act : j < h) {
        const int64_t i = (int64_t)(r0 + y0 + j) * U + u;
        T im;
        random_value<T, false>(k.n, k.R, seed, s, i, col, x[j], im);
        buf[base + j * U] = x[j];
        if (DS && cc == 0) dsm[base + j * U] = src[i];
      }
    }
  }
  T hh = hu;
  auto scale = [&](T f) {
    hh *= f;
    du *= f;
    ct *= f;
    cbm *= f;
#pragma unroll
    for (int d = 0; d < DIMS - 1; ++d) {
      cf[d] *= f;
      cb[d] *= f;
    }
  };
  // the first product runs with halved coefficients
  T df = T(0.5);  // scale of the diagonal in shared memory
  scale(T(0.5));
  auto sync = [&]() {
    if (C > 1) {
      arrive();
      wait();
    } else {
      __syncthreads();
    }
  };
  sync();

  const int nprod = k.M / 2;
  const int wpc = tpc >> 5;
  // the sums of `cnt` products of batch b
  auto bulk = [&](int b, int cnt) {
    const int items = cnt * 2 * ncol;
    {
      // four lanes per (product, column, dot) add the column's warps in a fixed order
      const double* rb = reinterpret_cast<const double*>(ring) + (size_t)(b & 1) * kb * NW * 2;
      const int sub = t & 3;
      for (int i0 = 0; i0 < items; i0 += BT / 4) {
        const int it = i0 + (t >> 2);
        const bool on = it < items;
        const int pi = it / (2 * ncol), r = it - pi * 2 * ncol, c = r >> 1, dot = r & 1;
        double a = 0.0;
        if (on)
          for (int v = sub; v < wpc; v += 4) a += rb[((size_t)pi * NW + c * wpc + v) * 2 + dot];
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        a += __shfl_xor_sync(0xffffffffu, a, 2);
        if (on && sub == 0) {
          const int step = b * kb + pi;
          if (C == 1) k.sums[(size_t)step * 2 * k.Rp + (size_t)dot * k.Rp + k.col0 + c] = a;
          else k.part[((size_t)q * nprod + step) * 2 * ncol + r] = a;
        }
      }
    }
  };

  const uint32_t bufb = (uint32_t)((size_t)bufn * sizeof(T));
  // product m reads buffer m % 2 and writes the other one
  int bi = 0;
#pragma unroll 1
  for (int m = 0; m < nprod; ++m) {
    const int bo = bi ^ 1;
    double a = 0.0, b = 0.0;
    if (act) {
      const T* X = buf + bi * bufn + base;
      T* Y = buf + bo * bufn + base;
      const T* D = dsm + (base - cc * BU);
      const T xt = ldc(at + bi * bufb, T(0));
      const T xb = ldc(ab + bi * bufb, T(0));
      T prev = xt;                       // v_n of the row before
      constexpr int GS = H < 4 ? H : 4;  // sites per group: their loads go out together
#pragma unroll
      for (int j0 = 0; j0 < H; j0 += GS) {
        T nf[GS][DIMS - 1], nb[GS][DIMS - 1], de[GS];
#pragma unroll
        for (int jj = 0; jj < GS; ++jj) {
          const int j = j0 + jj;
          if (j < H - G || j < h) {
#pragma unroll
            for (int d = 0; d < DIMS - 1; ++d) {
              nf[jj][d] = X[j * U + of[d]];
              nb[jj][d] = X[j * U + ob[d]];
            }
            de[jj] = DS ? df * D[j * U] : du;
          }
        }
#pragma unroll
        for (int jj = 0; jj < GS; ++jj) {
          const int j = j0 + jj;
          if (j < H - G || j < h) {
            T acc = fma(de[jj], x[j], -w[j]);
#pragma unroll
            for (int d = 0; d < DIMS - 1; ++d) {
              acc = fma(cf[d], nf[jj][d], acc);
              acc = fma(cb[d], nb[jj][d], acc);
            }
            const bool last = j == H - 1 || (j + 1 >= H - G && j + 1 == h);
            acc = fma(last ? cbm : hh, last ? xb : x[j + 1 < H ? j + 1 : j], acc);
            acc = fma(j == 0 ? ct : hh, prev, acc);
            Y[j * U] = acc;
            prev = x[j];
            a = fma(x[j], x[j], a);
            b = fma(acc, x[j], b);
            w[j] = x[j];
            x[j] = acc;
          }
        }
      }
    }
    {
      if (C > 1) arrive();
      // lanes: the upper half of the warp goes on with b, the lower with a
      const bool hi = (lane & 16) != 0;
      double keep = hi ? b : a;
      keep += __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, o);
      if ((lane & 15) == 0)
        reinterpret_cast<double*>(ring)[((size_t)((m / kb) & 1) * kb + m % kb) * NW * 2 + warp * 2 +
                                        (lane >> 4)] = keep;
      if (C > 1) wait();
      else __syncthreads();
      // the previous batch: every thread has arrived for this product, so its
      // ring entries of the last one are written (a cluster's arrive comes
      // before the entry of the same product); their half of the ring is next
      // written kb products later
      if (m > 0 && m % kb == 0) bulk(m / kb - 1, kb);
    }
    if (m == 0) {
      scale(T(2));
      df = T(1);
    }
    bi = bo;
  }
  {
    if (C > 1) __syncthreads();  // the ring entries of the last product
    const int bl = (nprod - 1) / kb;
    bulk(bl, nprod - bl * kb);
  }
}

// ------------------------------------------------------------------ FP64 in fixed point
// run_rows' task with the vectors in 64-bit fixed point (see kpm_fixed.cuh; one
// bit less here, |v| <= 2^60 units, so that the sum of six neighbours fits 64
// bits).  Integer sums are exact, so the uniform hopping multiplies the sum of
// the neighbours once: 4 multiply-adds and 2 (2D) or 4 (3D) 64-bit adds for
// the bonds of a site, where the FP64 pipe takes an FMA per bond at a 32nd of
// that rate.  The dots' lane and warp sums are integer sums too.
template <int DIMS, bool DS, int H, int G>
__device__ __noinline__ void run_fixed(const ColsTask& k, int q, int C, unsigned char* smem) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int L = k.geom.L[DIMS - 1];
  const int U = k.geom.stride[DIMS - 1];
  const bool per = k.geom.periodic[DIMS - 1] != 0;
  const int ncol = k.ncol, S = k.strips, tpc = k.tpc;
  const int r0 = band0(L, C, q), B = band0(L, C, q + 1) - r0;
  const int BU = k.rows * U;
  long long* buf = reinterpret_cast<long long*>(smem);  // [2][ncol][BU]
  const int bufn = ncol * BU;
  Fix* dsm = reinterpret_cast<Fix*>(buf + 2 * (size_t)bufn);  // [BU] scaled diagonal (DS)
  longlong2* ring = reinterpret_cast<longlong2*>(
      smem + (((size_t)2 * bufn + (DS ? BU : 0)) * 8 + 15) / 16 * 16);  // [2][kb][NW][2] (hi, lo)
  const int kb = k.batch;

  const int cc = t / tpc, tt = t - cc * tpc;
  const int strip = tt / U, u = tt - strip * U;
  const bool have = cc < ncol && strip < S;
  const int y0 = have ? (int)(((int64_t)B * strip) / S) : 0;
  const int h = have ? (int)(((int64_t)B * (strip + 1)) / S) - y0 : 0;
  const bool act = h > 0;
  const int base = have ? cc * BU + y0 * U + u : 0;
  const int col = k.col0 + cc;

  const Fix hu = Fix::of(k.sc->hu_re), du = Fix::of(k.sc->du);
  int of[DIMS - 1], ob[DIMS - 1];
  bool pf[DIMS - 1], pb[DIMS - 1];  // the bond exists
  {
    int rem = u;
#pragma unroll
    for (int d = 0; d < DIMS - 1; ++d) {
      const int Ld = k.geom.L[d], st = k.geom.stride[d];
      const int x = rem % Ld;
      rem /= Ld;
      const bool p = k.geom.periodic[d] != 0;
      of[d] = (x + 1 < Ld) ? st : (p ? -(Ld - 1) * st : 0);
      ob[d] = (x > 0) ? -st : (p ? (Ld - 1) * st : 0);
      pf[d] = (x + 1 < Ld) || p;
      pb[d] = (x > 0) || p;
    }
  }
  uint32_t at = 0, ab = 0;
  bool pt = false, pe = false;
  if (act) {
    auto addr = [&](int y) {
      int r = q;
      if (y < r0 || y >= r0 + B)
        for (r = 0; r < C - 1; ++r)
          if (y < band0(L, C, r + 1)) break;
      return map_addr(buf + (size_t)cc * BU + (y - band0(L, C, r)) * U + u, (uint32_t)r);
    };
    const int yt = r0 + y0 - 1, yb = r0 + y0 + h;
    pt = yt >= 0 || per;
    pe = yb < L || per;
    if (pt) at = addr(yt >= 0 ? yt : L - 1);
    if (pe) ab = addr(yb < L ? yb : 0);
  }

  long long x[H], w[H];
  {
    const unsigned long long seed = k.prm ? k.prm->seed : k.seed;
    const unsigned long long s = (unsigned long long)(k.s + (k.prm ? k.prm->s0 : 0));
    const Fix* src = reinterpret_cast<const Fix*>(k.ds);
#pragma unroll
    for (int j = 0; j < H; ++j) {
      x[j] = w[j] = 0;
      if (j < H - G ? act : j < h) {
        const int64_t i = (int64_t)(r0 + y0 + j) * U + u;
        double v, im;
        random_value<double, false>(k.n, k.R, seed, s, i, col, v, im);
        x[j] = v < 0.0 ? -(1ll << k.fixq) : 1ll << k.fixq;
        buf[base + j * U] = x[j];
        if (DS && cc == 0) dsm[base + j * U] = src[i];
      }
    }
  }
  auto sync = [&]() {
    if (C > 1) {
      arrive();
      wait();
    } else {
      __syncthreads();
    }
  };
  sync();

  const int nprod = k.M / 2;
  const int wpc = tpc >> 5;
  auto bulk = [&](int b, int cnt) {
    const int items = cnt * 2 * ncol;
    // four lanes per (product, column, dot) add the column's warps (exact sums)
    const longlong2* rb = ring + (size_t)(b & 1) * kb * NW * 2;
    const int sub = t & 3;
    for (int i0 = 0; i0 < items; i0 += BT / 4) {
      const int it = i0 + (t >> 2);
      const bool on = it < items;
      const int pi = it / (2 * ncol), r = it - pi * 2 * ncol, c = r >> 1, dot = r & 1;
      long long hi = 0, lo = 0;
      if (on)
        for (int v = sub; v < wpc; v += 4) {
          const longlong2 e = rb[((size_t)pi * NW + c * wpc + v) * 2 + dot];
          hi += e.x;
          lo += e.y;
        }
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        hi += __shfl_xor_sync(0xffffffffu, hi, o);
        lo += __shfl_xor_sync(0xffffffffu, lo, o);
      }
      if (on && sub == 0) {
        const double unit = __longlong_as_double((long long)(1023 + 64 - 2 * k.fixq) << 52);
        const double a = fma((double)lo, 0x1p-32, (double)hi) * unit;
        const int step = b * kb + pi;
        if (C == 1) k.sums[(size_t)step * 2 * k.Rp + (size_t)dot * k.Rp + k.col0 + c] = a;
        else k.part[((size_t)q * nprod + step) * 2 * ncol + r] = a;
      }
    }
  };

  const uint32_t bufb = (uint32_t)((size_t)bufn * 8);
  unsigned bad = 0;
  int bad_from = nprod;  // the first product whose result left the range
  int bi = 0;
#pragma unroll 1
  for (int m = 0; m < nprod; ++m) {
    const int bo = bi ^ 1;
    long long ah = 0, ac = 0, bh = 0, bc = 0;
    if (act) {
      const long long* X = buf + bi * bufn + base;
      long long* Y = buf + bo * bufn + base;
      const Fix* D = dsm + (base - cc * BU);
      const long long xt = pt ? ldc(at + bi * bufb, 0ll) : 0;
      const long long xb = pe ? ldc(ab + bi * bufb, 0ll) : 0;
      constexpr int GS = H < 4 ? H : 4;
#pragma unroll
      for (int j0 = 0; j0 < H; j0 += GS) {
        long long sum[GS];
        Fix de[GS];
#pragma unroll
        for (int jj = 0; jj < GS; ++jj) {
          const int j = j0 + jj;
          sum[jj] = 0;
          de[jj] = du;
          if (j < H - G || j < h) {
#pragma unroll
            for (int d = 0; d < DIMS - 1; ++d) {
              if (pf[d]) sum[jj] += X[j * U + of[d]];
              if (pb[d]) sum[jj] += X[j * U + ob[d]];
            }
            if (DS) de[jj] = D[j * U];
          }
        }
#pragma unroll
        for (int jj = 0; jj < GS; ++jj) {
          const int j = j0 + jj;
          if (j < H - G || j < h) {
            const bool last = j == H - 1 || (j + 1 >= H - G && j + 1 == h);
            const long long s =
                sum[jj] + (last ? xb : x[j + 1 < H ? j + 1 : j]) + (j == 0 ? xt : w[j > 0 ? j - 1 : 0]);
            const int s0 = (int)s, s1 = (int)((s - s0) >> 32);
            const int u0 = (int)x[j], u1 = (int)((x[j] - u0) >> 32);
            long long a11 = mad64(hu.hi, s1, 0), a10 = mad64(hu.hi, s0, 0);
            long long a01 = mad64(hu.lo, s1, 0), a00 = mad64(hu.lo, s0, 0);
            if (DS || (du.hi | du.lo) != 0) {
              a11 = mad64(de[jj].hi, u1, a11);
              a10 = mad64(de[jj].hi, u0, a10);
              a01 = mad64(de[jj].lo, u1, a01);
              a00 = mad64(de[jj].lo, u0, a00);
            }
            const long long tt2 = a01 + (a10 >> 4) + (a00 >> 32);
            long long v = m == 0 ? (a11 << 3) + ((tt2 + (1ll << 24)) >> 25)
                                 : (a11 << 4) + ((tt2 + (1ll << 23)) >> 24);
            v -= w[j];
            // (with a 64th to spare, as in kpm_fixed.cuh)
            constexpr unsigned TOP = (1u << 25) + (1u << 19), X1 = (1u << 28) + (1u << 22);
            bad |= (unsigned)(a11 >> 32) + TOP > 2 * TOP;
            const int v0 = (int)v, v1 = (int)((v - v0) >> 32);
            bad |= (unsigned)v1 + X1 > 2 * X1;
            Y[j * U] = v;
            ah = mad64(u1, u1, ah);
            bh = mad64(v1, u1, bh);
            dot_low(ac, bc, u1, u0, v1, v0);
            w[j] = x[j];
            x[j] = v;
          }
        }
        // at most 4 x 2^60: carried before it could overflow
        ah += ac >> 32;
        ac &= 0xffffffffll;
        bh += bc >> 32;
        bc &= 0xffffffffll;
      }
    }
    if (C > 1) arrive();
    // lanes: the upper half of the warp goes on with b, the lower with a
    const bool up = (lane & 16) != 0;
    long long kh = up ? bh : ah, kc = up ? bc : ac;
    kh += __shfl_xor_sync(0xffffffffu, up ? ah : bh, 16);
    kc += __shfl_xor_sync(0xffffffffu, up ? ac : bc, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      kh += __shfl_xor_sync(0xffffffffu, kh, o);
      kc += __shfl_xor_sync(0xffffffffu, kc, o);
    }
    if ((lane & 15) == 0)
      ring[((size_t)((m / kb) & 1) * kb + m % kb) * NW * 2 + warp * 2 + (lane >> 4)] =
          make_longlong2(kh, kc);
    if (C > 1) wait();
    else __syncthreads();
    if (m > 0 && m % kb == 0) bulk(m / kb - 1, kb);  // as in run_rows
    if (bad) bad_from = min(bad_from, m);
    bi = bo;
  }
  if (C > 1) __syncthreads();
  const int bl = (nprod - 1) / kb;
  bulk(bl, nprod - bl * kb);
  if (bad && k.prm) {
    RunParams* prm = const_cast<RunParams*>(k.prm);
    atomicOr(&prm->flags, 8);
    atomicMin(&prm->bad_from, bad_from);
  }
}

// ------------------------------------------------------------------ FP32, slots
// The same task with the vectors in thread-major slots: site j of thread t at
// j * SLOT + t, so that every access of the recursion is a per-thread base and
// a compile-time offset (in lattice order 21 of 43 instructions per site went
// into addresses).  A thread's in-plane neighbours are
// other threads' slots of the same j.  The dot sweep, whose chains run in
// lattice order, finds its rows' slots in a table built once per task (four
// 16-bit slots of a chunk in one 8-byte load); the line traversal needs only
// the slot of each line's first site, its sites being consecutive.  SLOT is
// odd so that adjacent lines fall on different banks.
constexpr int SLOT = BT + 1;

struct SlotLayout {
  int U, S, B, spi, lg, NR, nchains, nc4, n, lines, passes;
  __device__ __forceinline__ int strip0(int s) const { return (int)(((int64_t)B * s) / S); }
  // slot of plane position u of row y, for column 0
  __device__ __forceinline__ int slot(int y, int u) const {
    const int s = ((y + 1) * S - 1) / B;
    return (y - strip0(s)) * SLOT + s * U + u;
  }
};

__device__ __forceinline__ Pair2 slot_chain(const SlotLayout& o, const uint2* tab,
                                            const unsigned short* ltab, int Lx, const float* X,
                                            const float* Y, int chain) {
  Pair2 a;
  a.s = a.c = f2(0.0f);
  const int rank = chain >> o.lg, q = chain & (o.spi - 1);
  if (o.lines == 0) {
    const uint2* e = tab + chain;
    int left = o.n - (rank * 4 * o.spi + q);  // rows of this chain lie at steps of spi below n
#pragma unroll 2
    for (; left > 3 * o.spi; left -= 16 * o.spi, e += o.nchains) {
      const uint2 v = *e;
      const int i0 = v.x & 0xffff, i1 = v.x >> 16, i2 = v.y & 0xffff, i3 = v.y >> 16;
      const float x0 = X[i0], x1 = X[i1], x2 = X[i2], x3 = X[i3];
      const float y0 = Y[i0], y1 = Y[i1], y2 = Y[i2], y3 = Y[i3];
      dot1(a, x0, y0);
      dot1(a, x1, y1);
      dot1(a, x2, y2);
      dot1(a, x3, y3);
    }
    if (left > 0) {  // a last, partly filled chunk (none of this chain follows it)
      const uint2 v = *e;
      const int i0 = v.x & 0xffff, i1 = v.x >> 16, i2 = v.y & 0xffff;
      dot1(a, X[i0], Y[i0]);
      if (left > o.spi) dot1(a, X[i1], Y[i1]);
      if (left > 2 * o.spi) dot1(a, X[i2], Y[i2]);
    }
  } else {
    int cx = rank * 4, blk = 0;
    for (int p = rank * 4; p < o.passes; p += 16) {
      while (cx >= Lx) {
        cx -= Lx;
        ++blk;
      }
      int line = (blk << o.lg) + q;
      if (cx + 4 <= Lx) {
        if (line < o.lines) {
          const int i = ltab[line] + cx;
          float x[4], y[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            x[j] = X[i + j];
            y[j] = Y[i + j];
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) dot1(a, x[j], y[j]);
        }
      } else {
        int c2 = cx;
        for (int j = 0; j < 4 && p + j < o.passes; ++j, ++c2) {
          if (c2 == Lx) {
            c2 = 0;
            line += o.spi;
          }
          if (line < o.lines) {
            const int i = ltab[line] + c2;
            dot1(a, X[i], Y[i]);
          }
        }
      }
      cx += 16;
    }
  }
  return a;
}

// (product, column, dot) total of the NR CTAs of the global-memory form that
// have rows: eight groups each in compensated pairs, their totals in FP64.
__device__ __forceinline__ double slot_total(const float2* ring, int NR, int dot) {
  double total = 0.0;
#pragma unroll 1
  for (int r = 0; r < NR; ++r) {
    float s = 0.0f, c = 0.0f;
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      const float2 e = ring[(r * 8 + g) * 2 + dot];
      pair_add(s, c, e.x, e.y);
    }
    total += (double)s - (double)c;
  }
  return total;
}

template <int DIMS, bool DS, int H, int G>
__device__ __noinline__ void run_slots(const ColsTask& k, unsigned char* smem) {
  const int t = threadIdx.x, lane = t & 31;
  const int B = k.geom.L[DIMS - 1], Ur = k.geom.stride[DIMS - 1], L0 = k.geom.L[0];
  const bool per = k.geom.periodic[DIMS - 1] != 0;
  const int ncol = k.ncol, S = k.strips, tpc = k.tpc, kb = k.batch, kl = 31 - __clz(k.batch);  // kb a power of two
  SlotLayout o;
  o.U = DIMS == 2 ? k.pitch : k.pitch * k.geom.L[1];  // thread positions of a row
  o.S = S;
  o.B = B;
  o.n = (int)k.n;
  o.spi = k.spi;
  o.lg = 31 - __clz(k.spi);
  o.lines = k.lines;
  o.passes = k.lines > 0 ? (k.lines + k.spi - 1) / k.spi * L0 : (o.n + k.spi - 1) / k.spi;
  o.NR = min(4, (o.passes + 3) / 4);
  o.nchains = o.NR * o.spi;
  o.nc4 = (o.passes + 15) / 16;
  const int bufn = (k.height * SLOT + 3) / 4 * 4;
  float* buf = reinterpret_cast<float*>(smem);  // [3][height][SLOT]
  float2* ring = reinterpret_cast<float2*>(smem + (size_t)3 * bufn * 4);  // [2][kb][ncol][NR * 8][2]
  const int rentry = o.NR * 16;
  uint2* tab = reinterpret_cast<uint2*>(ring + 2 * kb * ncol * rentry);  // [nc4][nchains]
  unsigned short* ltab = reinterpret_cast<unsigned short*>(tab);         // [lines]

  // this thread's column, strip and plane position
  const int cc = t / tpc, tt = t - cc * tpc;
  const int strip = tt / o.U, u = tt - strip * o.U;
  const int x0 = DIMS == 2 ? u : u % k.pitch, yy = DIMS == 2 ? 0 : u / k.pitch;
  const bool act = cc < ncol && strip < S && x0 < L0;
  const int y0 = act ? o.strip0(strip) : 0;
  const int h = act ? o.strip0(strip + 1) - y0 : 0;
  const int col = k.col0 + cc;

  float hu, hi_, du;
  scal_from_block<float>(k.sc, hu, hi_, du);
  int of[DIMS - 1], ob[DIMS - 1];
  float cf[DIMS - 1], cb[DIMS - 1];
#pragma unroll
  for (int d = 0; d < DIMS - 1; ++d) {
    const int Ld = k.geom.L[d], st = d == 0 ? 1 : k.pitch, x = d == 0 ? x0 : yy;
    const bool p = k.geom.periodic[d] != 0;
    of[d] = (x + 1 < Ld) ? st : (p ? -(Ld - 1) * st : 0);
    ob[d] = (x > 0) ? -st : (p ? (Ld - 1) * st : 0);
    cf[d] = (x + 1 < Ld) || p ? hu : 0.0f;
    cb[d] = (x > 0) || p ? hu : 0.0f;
  }
  // slots of the rows before and after the strip
  int at = t, ab = t;
  float ct = 0.0f, cbm = 0.0f;
  if (act) {
    const bool ht = strip > 0 || per, hb = strip + 1 < S || per;
    const int st = strip > 0 ? strip - 1 : S - 1;
    if (ht) at = (o.strip0(st + 1) - o.strip0(st) - 1) * SLOT + t + (st - strip) * o.U;
    const int sb = strip + 1 < S ? strip + 1 : 0;
    if (hb) ab = t + (sb - strip) * o.U;
    ct = ht ? hu : 0.0f;
    cbm = hb ? hu : 0.0f;
  }

  // start vectors
  float x[H], dd[DS ? H : 1];
  {
    const unsigned long long seed = k.prm ? k.prm->seed : k.seed;
    const unsigned long long s = (unsigned long long)(k.s + (k.prm ? k.prm->s0 : 0));
    const float* src = reinterpret_cast<const float*>(k.ds);
#pragma unroll
    for (int j = 0; j < H; ++j) {
      x[j] = 0.0f;
      if (DS) dd[j] = 0.0f;
      if (j < H - G ? act : j < h) {
        const int64_t i = (int64_t)(y0 + j) * Ur + (x0 + yy * L0);
        if (DS) dd[j] = src[i];
        float im;
        random_value<float, false>(k.n, k.R, seed, s, i, col, x[j], im);
        buf[j * SLOT + t] = x[j];
        buf[2 * bufn + j * SLOT + t] = 0.0f;
      }
    }
  }
  // the dot sweep's slots
  if (o.lines == 0) {
    for (int e = t; e < o.nc4 * o.nchains; e += BT) {
      const int c4 = e / o.nchains, chain = e - c4 * o.nchains;
      const int rank = chain >> o.lg, q = chain & (o.spi - 1);
      unsigned v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = ((rank + 4 * c4) * 4 + j) * o.spi + q;
        const int y = i / Ur, ur = i - y * Ur;
        v[j] = i < o.n ? o.slot(y, ur) : 0;
      }
      tab[e] = make_uint2(v[0] | v[1] << 16, v[2] | v[3] << 16);
    }
  } else {
    const int per_row = DIMS == 2 ? 1 : k.geom.L[1];
    for (int e = t; e < o.lines; e += BT) ltab[e] = (unsigned short)o.slot(e / per_row, e % per_row * k.pitch);
  }
  float hh = hu;
  auto scale = [&](float f) {
    hh *= f;
    du *= f;
    ct *= f;
    cbm *= f;
#pragma unroll
    for (int d = 0; d < DIMS - 1; ++d) {
      cf[d] *= f;
      cb[d] *= f;
    }
    if (DS) {
#pragma unroll
      for (int j = 0; j < H; ++j) dd[j] *= f;
    }
  };
  scale(0.5f);  // the first product runs with halved coefficients
  __syncthreads();

  const int nprod = k.M / 2;
  const int gl = 1 << (o.lg - 3);  // chains per group
  auto bulk = [&](int b, int cnt) {
    const int items = cnt * 2 * ncol;
    const float2* rb = ring + (b & 1) * kb * ncol * rentry;
    for (int it = t; it < items; it += BT) {
      const int pi = it / (2 * ncol), r = it - pi * 2 * ncol, c = r >> 1, dot = r & 1;
      k.sums[(size_t)(b * kb + pi) * 2 * k.Rp + (size_t)dot * k.Rp + k.col0 + c] =
          slot_total(rb + (pi * ncol + c) * rentry, o.NR, dot);
    }
  };
  // Product m reads buffer m % 3 and writes buffer (m + 1) % 3; the dots of
  // product m - 1 are swept in the same phase (v_{m-1} and v_m stay in place),
  // so one barrier per product serves both; the last phase only sweeps.
  int bi = 0;
#pragma unroll 1
  for (int m = 0; m <= nprod; ++m) {
    const int bo = bi == 2 ? 0 : bi + 1, bp = bi == 0 ? 2 : bi - 1;
    if (act && m < nprod) {
      const float* X = buf + bi * bufn;
      const float* Xo = X + t;
      const float* W = buf + bp * bufn + t;
      float* Y = buf + bo * bufn + t;
      const float* Xf[DIMS - 1];
      const float* Xb[DIMS - 1];
#pragma unroll
      for (int d = 0; d < DIMS - 1; ++d) {
        Xf[d] = Xo + of[d];
        Xb[d] = Xo + ob[d];
      }
      const float xb = X[ab];
      float prev = X[at];                // v_n of the row before
      constexpr int GS = H < 4 ? H : 4;  // sites per group: their loads go out together
#pragma unroll
      for (int j0 = 0; j0 < H; j0 += GS) {
        float nf[GS][DIMS - 1], nb[GS][DIMS - 1], ww[GS];
#pragma unroll
        for (int jj = 0; jj < GS; ++jj) {
          const int j = j0 + jj;
          if (j < H - G || j < h) {
#pragma unroll
            for (int d = 0; d < DIMS - 1; ++d) {
              nf[jj][d] = Xf[d][j * SLOT];
              nb[jj][d] = Xb[d][j * SLOT];
            }
            ww[jj] = W[j * SLOT];
          }
        }
#pragma unroll
        for (int jj = 0; jj < GS; ++jj) {
          const int j = j0 + jj;
          if (j < H - G || j < h) {
            float acc = fmaf(DS ? dd[j] : du, x[j], -ww[jj]);
#pragma unroll
            for (int d = 0; d < DIMS - 1; ++d) {
              acc = fmaf(cf[d], nf[jj][d], acc);
              acc = fmaf(cb[d], nb[jj][d], acc);
            }
            const bool last = j == H - 1 || (j + 1 >= H - G && j + 1 == h);
            acc = fmaf(last ? cbm : hh, last ? xb : x[j + 1 < H ? j + 1 : j], acc);
            acc = fmaf(j == 0 ? ct : hh, prev, acc);
            Y[j * SLOT] = acc;
            prev = x[j];
            x[j] = acc;
          }
        }
      }
    }
    if (m > 0) {
      float2* rg = ring + ((m - 1) & (2 * kb - 1)) * ncol * rentry;
      const float* X = buf + bp * bufn;
      const float* Y = buf + bi * bufn;
#pragma unroll 1
      for (int ch = t, c = 0, chain = t; ch < ncol * o.nchains; ch += BT, chain += BT) {
        while (chain >= o.nchains) {
          chain -= o.nchains;
          ++c;
        }
        const int lanes = min(32, ncol * o.nchains - (ch - lane));  // of this warp's, with a chain
        const unsigned mask = 0xffffffffu >> (32 - lanes);
        const Pair2 a = slot_chain(o, tab, ltab, L0, X + c * tpc, Y + c * tpc, chain);
        float2* out = rg + c * rentry + (chain >> (o.lg - 3)) * 2;
        if (gl == 1) {
          out[0] = make_float2(a.s.x, a.c.x);
          out[1] = make_float2(a.s.y, a.c.y);
        } else {
          // neighbours first: even lanes go on with the first dot, odd with the second
          const bool odd = lane & 1;
          float ks = odd ? a.s.y : a.s.x, kc = odd ? a.c.y : a.c.x;
          const float gs = odd ? a.s.x : a.s.y, gc = odd ? a.c.x : a.c.y;
          pair_add(ks, kc, __shfl_xor_sync(mask, gs, 1), __shfl_xor_sync(mask, gc, 1));
#pragma unroll 1
          for (int off = 2; off < gl; off <<= 1)
            pair_add(ks, kc, __shfl_xor_sync(mask, ks, off), __shfl_xor_sync(mask, kc, off));
          if ((lane & (gl - 1)) < 2) out[lane & 1] = make_float2(ks, kc);
        }
      }
      // batch b: its last sweep ran in the phase of product (b + 1) kb, one
      // barrier ago; its half of the ring is next written kb phases later
      if (m > kb && ((m - 1) & (kb - 1)) == 0) bulk(((m - 1) >> kl) - 1, kb);
    }
    __syncthreads();
    if (m == 0) scale(2.0f);
    bi = bo;
  }
  // the batch not summed in the loop (its last phase is that of product nprod)
  const int bl = (nprod - 1) / kb;
  bulk(bl, nprod - bl * kb);
}

template <typename T, int DIMS, bool DS>
__global__ void __launch_bounds__(BT, 1)
    cols_kernel(const ColsTask* __restrict__ tasks, int ntasks, int* queue, int C) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_task, s_last;
  __shared__ ColsTask s_k;
  const int t = threadIdx.x;
  const int q = C > 1 ? (int)(blockIdx.x % C) : 0;
  for (;;) {
    // the cluster's next task (every CTA has read rank 0's word before it is
    // written again or rank 0 exits)
    int task;
    if (C > 1) {
      if (q == 0 && t == 0) s_task = atomicAdd(queue, 1);
      arrive();
      wait();
      uint32_t a = map_addr(&s_task, 0);
      asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(task) : "r"(a) : "memory");
      arrive();
      wait();
    } else {
      if (t == 0) s_task = atomicAdd(queue, 1);
      __syncthreads();
      task = s_task;
      __syncthreads();
    }
    if (task >= ntasks) break;
    {
      const int* src = reinterpret_cast<const int*>(tasks + task);
      int* dst = reinterpret_cast<int*>(&s_k);
      for (int e = t; e < (int)(sizeof(ColsTask) / 4); e += BT) dst[e] = src[e];
    }
    __syncthreads();
    const ColsTask& k = s_k;
    const int hm = k.height;
    if constexpr (sizeof(T) == 4) {
      if (hm <= 2) run_slots<DIMS, DS, 2, 2>(k, smem);
      else if (hm <= 4) run_slots<DIMS, DS, 4, 2>(k, smem);
      else if (hm <= 8) run_slots<DIMS, DS, 8, 4>(k, smem);
      else if (hm <= 12) run_slots<DIMS, DS, 12, 4>(k, smem);
      else if (hm <= 16) run_slots<DIMS, DS, 16, 4>(k, smem);
      else if (hm <= 20) run_slots<DIMS, DS, 20, 4>(k, smem);
      else if (hm <= 24) run_slots<DIMS, DS, 24, 4>(k, smem);
      else if (hm <= 28) run_slots<DIMS, DS, 28, 4>(k, smem);
      else run_slots<DIMS, DS, 32, 4>(k, smem);
    } else if (k.fixq > 0) {
      if (hm <= 2) run_fixed<DIMS, DS, 2, 2>(k, q, C, smem);
      else if (hm <= 4) run_fixed<DIMS, DS, 4, 2>(k, q, C, smem);
      else if (hm <= 8) run_fixed<DIMS, DS, 8, 4>(k, q, C, smem);
      else if (hm <= 12) run_fixed<DIMS, DS, 12, 4>(k, q, C, smem);
      else run_fixed<DIMS, DS, 16, 4>(k, q, C, smem);
    } else {
      if (hm <= 2) run_rows<DIMS, DS, 2, 2>(k, q, C, smem);
      else if (hm <= 4) run_rows<DIMS, DS, 4, 2>(k, q, C, smem);
      else if (hm <= 8) run_rows<DIMS, DS, 8, 4>(k, q, C, smem);
      else if (hm <= 12) run_rows<DIMS, DS, 12, 4>(k, q, C, smem);
      else run_rows<DIMS, DS, 16, 4>(k, q, C, smem);
    }
    const int nprod = k.M / 2, ncol = k.ncol;
    if (C > 1) {
      // the CTAs' partials, added in rank order
      arrive();
      wait();
      const int total = nprod * 2 * ncol;
      for (int e = q * BT + t; e < total; e += C * BT) {
        const int step = e / (2 * ncol), r = e - step * 2 * ncol;
        double s = 0.0;
        for (int p = 0; p < C; ++p) s += k.part[(size_t)p * total + e];
        k.sums[(size_t)step * 2 * k.Rp + (size_t)(r & 1) * k.Rp + k.col0 + (r >> 1)] = s;
      }
      arrive();
      wait();
    }
    __syncthreads();  // the sums of this task (C == 1: written by this CTA)
    if (k.per_vec && q == 0) {
      const int M = k.M, R = k.R, Rp = k.Rp;
      const double inv_n = 1.0 / (double)k.n;
      for (int e = t; e < ncol * nprod; e += BT) {
        const int r = k.col0 + e / nprod, step = e % nprod;
        const double mu0 = k.sums[r] * inv_n, mu1 = k.sums[Rp + r] * inv_n;
        double me = mu0, mo = mu1;
        if (step > 0) {
          me = 2.0 * k.sums[(size_t)step * 2 * Rp + r] * inv_n - mu0;
          mo = 2.0 * k.sums[(size_t)step * 2 * Rp + Rp + r] * inv_n - mu1;
        }
        k.per_vec[(size_t)r * M + 2 * step] = me;
        k.per_vec[(size_t)r * M + 2 * step + 1] = mo;
        if (!(fabs(me) <= 1.0 + 1e-6) || !(fabs(mo) <= 1.0 + 1e-6)) atomicOr(k.flags, 1);
      }
      __syncthreads();
      // the other tasks' per-vector moments: published by their fence before
      // their count, read through L2
      __threadfence();
      if (t == 0) s_last = atomicAdd(k.tiles_done, 1) == k.ntiles - 1;
      __syncthreads();
      if (s_last) {
        __threadfence();
        for (int m = t; m < M; m += BT) {
          double acc = 0.0;
          for (int r = 0; r < R; ++r) acc += __ldcg(k.per_vec + (size_t)r * M + m);
          k.mu[m] = acc / (double)R;
        }
      }
    }
    if (C > 1) {
      arrive();
      wait();
    } else {
      __syncthreads();  // s_k and the buffers are free
    }
  }
}

// Once per kernel and device: 16-CTA clusters (a non-portable size) and
// dynamic shared memory up to COLS_MAX_SMEM.
template <typename T, int DIMS, bool DS>
bool configure() {
  static std::atomic<unsigned long long> done{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const unsigned long long bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return true;
  auto kern = cols_kernel<T, DIMS, DS>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)COLS_MAX_SMEM) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  done.fetch_or(bit, std::memory_order_acq_rel);
  return true;
}

inline void fill(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int clusters, int C,
                 size_t smem, cudaStream_t st) {
  cfg.gridDim = dim3((unsigned)(clusters * C));
  cfg.blockDim = dim3(BT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

template <typename T, int DIMS, bool DS>
cudaError_t launch(const ColsTask* tasks, int ntasks, int* queue, int clusters, int C, size_t smem,
                   cudaStream_t st) {
  if (!configure<T, DIMS, DS>()) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  fill(cfg, attr, clusters, C, smem, st);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaLaunchKernelEx(&cfg, cols_kernel<T, DIMS, DS>, tasks, ntasks, queue, C);
}

template <typename T, int DIMS, bool DS>
int max_clusters(int C, size_t smem) {
  if (!configure<T, DIMS, DS>()) return 0;
  auto kern = cols_kernel<T, DIMS, DS>;
  int n = 0;
  if (C == 1) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, BT, smem) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return n * sms;
  }
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  fill(cfg, attr, 1, C, smem, nullptr);
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

}  // namespace cols
}  // namespace kpm
