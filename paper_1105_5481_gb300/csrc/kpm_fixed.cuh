// FP64 vectors in 64-bit fixed point: the chunk policy of the fused step that
// takes the recursion off GB300's FP64 pipe.
//
// That pipe retires 2 FMAs per SM and clock, a 64th of the FP32 rate, so the
// FP64 step of a complex 3D lattice (30 FP64 instructions per element) ran at
// 89 % of its peak with HBM at 13 %.  The entries of a Chebyshev vector are
// bounded by its start vector's norm (|v_n,i| <= |v_n| <= |v_0| = sqrt(N) while
// the spectrum is enclosed), so a 64-bit integer of unit 2^-q,
// q = 61 - ceil(log2(N) / 2), holds them with at least FP64's absolute
// resolution of entries of order one while q >= 51, and integer multiply-adds
// (32 x 32 + 64 bits, 32 times the FP64 rate) do the products:
//
//   x = (x1 2^32 + x0) 2^-q     x0 signed 32 bits, |x1| <= 2^29
//   h = (h1 2^28 + h0) 2^-56    h0 signed 28 bits, |h| <= 7
//   h x: h1 x1 2^60 + h1 x0 2^28 + h0 x1 2^32 + h0 x0, each class summed exactly
//   in 64 bits over the row's bonds, then one rounding to the unit.
//
// The sums fit: sum |h| <= 15 over a row, which the host checks, bounds h1 x1 and
// h1 x0 by 2^63 for any number of entries.  h0 does not shrink with h (|h0| <= 2^27,
// |x0| <= 2^31), so h0 x0 holds 31 products and h0 x1 127: stencil rows have at most
// 13 of each per component, padded rows 17, and the entries of a CSR row beyond 30
// (15 in complex fields) are followed, four by four, by carries of the upper parts to
// the next class (Row::fold).  (Carries within every row, each 8 or 16 entries, cost
// rows of up to 19 entries 2 to 5 %.)
//
// Measured (3D L = 64 spin lattice, 64 complex vectors): 374 us per step against
// 939 on the FP64 pipe.  Bound by issue at 16 warps per SM (math-pipe throttle
// and fixed latency the largest stalls): about 500 instructions per element, 110
// of them 32 x 32 + 64 multiply-adds at two cycles each.  On the way: 489 us with
// the accumulations written as C products (they became separate 64-bit adds),
// 407 before the open-edge selects were skipped on periodic lattices and four
// positions of a line were unrolled.  CSR operators (3D, 10 % dilution, N =
// 305,000, 14 columns): 13.0 -> 7.3 ms real, 32.3 -> 16.1 ms complex (M = 256).
//
// An element takes one rounding of 2^-q / 2 per product where FP64 takes one of
// about 2^-54 relative per term.  Error of the moments against 113-bit arithmetic,
// over the FP64 pipe's: 0.91 to 0.98 on 2,000 to 16,000 sites (M = 256), 0.93 to 1.02
// up to 2^20 complex and 2^18 real sites (FIXED_MAX_N_REAL in kpm_api.cu), where an
// FP64 result's own rounding shows.  Coefficients have the absolute unit 2^-56: one
// far below the largest keeps fewer bits than in FP64, but moves H by no more than
// the FP64 rounding of the largest does.  The dots are sums of exact
// products likewise (<v_n|v_n> <= N bounds them), converted to FP64 once per
// thread group.  A value past 2^61 by a 64th (the spectrum is not enclosed: then a
// moment has left [-1, 1] as well) sets bit 3 of the call's flags; the moments that
// such a product enters become NaN.
#pragma once

#include "kpm_step.cuh"

namespace kpm {

struct Fix {  // (hi 2^28 + lo) 2^-56
  int hi, lo;
  __device__ __forceinline__ Fix() {}
  __device__ __forceinline__ Fix(int h, int l) : hi(h), lo(l) {}
  __device__ __forceinline__ explicit Fix(int z) : hi(z), lo(0) {}  // of 0 alone
  __device__ __forceinline__ Fix operator-() const { return Fix(-hi, -lo); }
  static __device__ __forceinline__ Fix of(double v) {
    const long long L = __double2ll_rn(v * 0x1p56);
    const int l = (int)((unsigned)L << 4) >> 4;
    return Fix((int)((L - l) >> 28), l);
  }
};
__device__ __forceinline__ Fix ldg_scal(const Fix* p, size_t i) {
  const int2 v = __ldg(reinterpret_cast<const int2*>(p) + i);
  return Fix(v.x, v.y);
}
__device__ __forceinline__ ScalPair<Fix> ldg_pair(const Fix* p, size_t i) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p) + i);
  return {Fix(v.x, v.y), Fix(v.z, v.w)};
}
template <>
__device__ __forceinline__ void scal_from_block<Fix>(const ScalarBlock* sc, Fix& hr, Fix& hi, Fix& du) {
  hr = Fix::of(sc->hu_re);
  hi = Fix::of(sc->hu_im);
  du = Fix::of(sc->du);
}

__device__ __forceinline__ long long mad64(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

// The classes of weight 2^32 of the dots x x and y x.  Of the products of the
// low words 16 leading bits each are enough: their error, 2^47 at random of
// either sign, is far below the unit of a sum of order 2^(2 q).
__device__ __forceinline__ void dot_low(long long& ac, long long& bc, int x1, int x0, int y1, int y0) {
  const int xh = x0 >> 16;
  ac = mad64(xh, xh, mad64(2 * x1, x0, ac));
  bc = mad64(y0 >> 16, xh, mad64(y1, x0, mad64(y0, x1, bc)));
}

// 16 bytes: two scalars (x1, x0); 2 real columns or 1 complex column (re, im).
template <bool CPLX_>
struct ChunkI64 {
  using T = Fix;
  static constexpr bool CPLX = CPLX_;
  static constexpr bool NC = true;
  static constexpr int SC = 2;
  static constexpr int VEC = CPLX ? 1 : 2;
  int x1[2], x0[2];

  __device__ __forceinline__ void set(const int4& q) {
    x1[0] = q.x; x0[0] = q.y; x1[1] = q.z; x0[1] = q.w;
  }
  __device__ __forceinline__ void ld_x(const Fix* p) { set(__ldg(reinterpret_cast<const int4*>(p))); }
  __device__ __forceinline__ void ld_cs(const Fix* p) { set(__ldcs(reinterpret_cast<const int4*>(p))); }
  __device__ __forceinline__ void st(Fix* p) const {
    *reinterpret_cast<int4*>(p) = make_int4(x1[0], x0[0], x1[1], x0[1]);
  }

  // Dots: class sums of weight 2^64 (h) and 2^32 (c, kept below 2^32 between rows).
  struct Acc {
    long long ah[VEC], ac[VEC], bh[VEC], bc[VEC];
  };
  static __device__ __forceinline__ void acc_zero(Acc& s) {
#pragma unroll
    for (int k = 0; k < VEC; ++k) s.ah[k] = s.ac[k] = s.bh[k] = s.bc[k] = 0;
  }
  static __device__ __forceinline__ void carry(long long& h, long long& c) {
    h += c >> 32;
    c &= 0xffffffffll;
  }
  static __device__ __forceinline__ void acc_add(Acc& s, const ChunkI64& x, const ChunkI64& y) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int k = CPLX ? 0 : q;
      s.ah[k] = mad64(x.x1[q], x.x1[q], s.ah[k]);
      s.bh[k] = mad64(y.x1[q], x.x1[q], s.bh[k]);
      dot_low(s.ac[k], s.bc[k], x.x1[q], x.x0[q], y.x1[q], y.x0[q]);
    }
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
      carry(s.ah[k], s.ac[k]);
      carry(s.bh[k], s.bc[k]);
    }
  }
  static __device__ __forceinline__ void warp_reduce(Acc& s, int Gt) {
    for (int off = Gt; off < 32; off <<= 1) {
#pragma unroll
      for (int k = 0; k < VEC; ++k) {
        s.ah[k] += __shfl_xor_sync(0xffffffffu, s.ah[k], off);
        s.ac[k] += __shfl_xor_sync(0xffffffffu, s.ac[k], off);
        s.bh[k] += __shfl_xor_sync(0xffffffffu, s.bh[k], off);
        s.bc[k] += __shfl_xor_sync(0xffffffffu, s.bc[k], off);
      }
    }
  }
  // in units of 2^(64 - 2 q) (RowAcc::dot_scale)
  static __device__ __forceinline__ void acc_out(const Acc& s, double (&A)[VEC], double (&B)[VEC]) {
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
      A[k] = fma((double)s.ac[k], 0x1p-32, (double)s.ah[k]);
      B[k] = fma((double)s.bc[k], 0x1p-32, (double)s.bh[k]);
    }
  }

  // One row: the class sums of its products, and v_{n-1}.
  struct Row {
    long long a11[2], a10[2], a01[2], a00[2];
    int w1[2], w0[2];
    int sh;  // 24: the step; 25: the first product, half of it
    __device__ __forceinline__ void zero() {
      sh = 24;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        a11[q] = a10[q] = a01[q] = a00[q] = 0;
        w1[q] = w0[q] = 0;
      }
    }
    __device__ __forceinline__ void set_neg(const ChunkI64& w) {
      zero();
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        w1[q] = w.x1[q];
        w0[q] = w.x0[q];
      }
    }
    __device__ __forceinline__ void half() { sh = 25; }
    __device__ __forceinline__ void mac(int q, const Fix& h, int u1, int u0) {
      a11[q] = mad64(h.hi, u1, a11[q]);
      a10[q] = mad64(h.hi, u0, a10[q]);
      a01[q] = mad64(h.lo, u1, a01[q]);
      a00[q] = mad64(h.lo, u0, a00[q]);
    }
    // carries of h0 x0 (weight 1) into h0 x1 (2^32), and of that into h1 x1 (2^60)
    __device__ __forceinline__ void fold() {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        a01[q] += a00[q] >> 32;
        a00[q] &= 0xffffffffll;
        a11[q] += a01[q] >> 28;
        a01[q] &= 0xfffffffll;
      }
    }
    // the diagonal (often zero: no on-site terms and symmetric bounds)
    __device__ __forceinline__ void axpy(const Fix& d, const ChunkI64& x) {
      if ((d.hi | d.lo) == 0) return;
      mac(0, d, x.x1[0], x.x0[0]);
      mac(1, d, x.x1[1], x.x0[1]);
    }
    __device__ __forceinline__ void cmac(const Fix& hr, const Fix& hi, const ChunkI64& x) {
      mac(0, hr, x.x1[0], x.x0[0]);
      mac(1, hr, x.x1[1], x.x0[1]);
      if constexpr (CPLX) {
        mac(0, -hi, x.x1[1], x.x0[1]);
        mac(1, hi, x.x1[0], x.x0[0]);
      }
    }
  };
};

template <bool CPLX>
struct RowAcc<ChunkI64<CPLX>> {
  using CH = ChunkI64<CPLX>;
  using type = typename CH::Row;
  static constexpr bool kIssueBound = true;
  // (31 products, the diagonal's among them)
  static constexpr int kFold = CPLX ? 15 : 30;
  static __device__ __forceinline__ void fold(type& r) { r.fold(); }
  // The sums rounded to the unit, less v_{n-1}.  `bad` is set when a value
  // leaves +-2^61 by more than a 64th: |a11| bounds the sum before its shift can
  // overflow.  (The start block of one site of N = 4^k lies on 2^61, and a spectrum
  // outside the bounds by less than KPM_EDIVERGE allows for passes it by 2.5e-7.)
  static __device__ __forceinline__ CH done(const type& r, unsigned& bad) {
    CH y;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      // in units of 2^32 (2^-24 of the result's); folded or not, the same result
      const long long t = r.a01[q] + (r.a10[q] >> 4) + (r.a00[q] >> 32);
      long long v;
      if (r.sh == 24) v = (r.a11[q] << 4) + ((t + (1ll << 23)) >> 24);
      else v = (r.a11[q] << 3) + ((t + (1ll << 24)) >> 25);
      const int top = (int)(r.a11[q] >> 32);
      v -= ((long long)r.w1[q] << 32) + r.w0[q];
      const int lo = (int)v;
      y.x0[q] = lo;
      y.x1[q] = (int)((v - lo) >> 32);
      constexpr unsigned TOP = (1u << 26) + (1u << 20), X1 = (1u << 29) + (1u << 23);
      bad |= (unsigned)top + TOP > 2 * TOP;
      bad |= (unsigned)y.x1[q] + X1 > 2 * X1;
    }
    return y;
  }
  static __device__ __forceinline__ double dot_scale(const StepArgs& a) {
    return __longlong_as_double((long long)(1023 + 64 - 2 * a.fixq) << 52);
  }
  static __device__ __forceinline__ void report(const StepArgs& a, unsigned bad) {
    if (bad && a.err) {
      atomicOr(a.err, 8);
      atomicMin(a.err + 1, a.step);
    }
  }
};

}  // namespace kpm
