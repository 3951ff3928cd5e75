// The dense products of the Hutch++ split (Y^T Y, A^T G, Y R^{-1}, G - A B)
// in fixed point.
//
// An FP64 instruction takes a sub-partition 64 clocks and more on this GPU (78
// measured), a 32 x 32 + 64-bit integer multiply-add 4.7, an FP32 one 1, so
// n s^2 FP64 multiply-adds took the time (93 % FP64 pipe) of products that
// read and write a few n s numbers.  A column is scaled by the power of two
// 2^f above its largest entry and held as integers of 60 bits in two limbs.
//
// Sums over rows: X = xh + 2^-32 xl, xh an integer of H bits and xl the 32 bits
// that follow (signed, rounded to FP32's 24), and
//
//   X Y = xh yh + 2^-32 (xh yl + xl yh)    (+ 2^-64 xl yl)
//
// takes one integer multiply-add, summed exactly, and two FP32 ones, whose sum
// is H bits smaller and joins the integers every fourth row.  A^T G adds
// 56-bit entries.  Applies: two limbs of 30 bits and three integer products.
//
// How exact: with a typical entry 2^f / rho (rho is about 10 for Gaussian
// columns), Gram entries err by 1e-17 to 3e-17 on the diagonal and 3e-18 to
// 1e-17 of the norms off it (NumPy replay against exact sums, rho = 8 to 16, n =
// 4,883; FP64 sums 0.7e-16 to 1.6e-16 and 1e-17).  Orthonormal columns are off
// the exact factor by 0.85e-16 to 1.03e-16 of their norm, by the FP64 kernels
// 0.85e-16 to 0.92e-16 (rms; 13,007 and 24,001 x 64, 20,011 x 32, 50,021 x 20).  Blocks with
// rho above 16 (the entries of one heavy row, say), infinities or NaN are
// flagged, and the FP64 kernels, launched after each of these, run instead.
// With FP32 cross terms in the applies too, and sums rounded at each fold,
// columns were off by 1.1e-15 at rho = 8 and 1.3e-14 at 31 (4,883 x 64).
//
// FP32 blocks (mixed solves) take the two sums over rows as well, in place of
// compensated FP32 dots of 17 operations (which err by 2^-48): H = 28, cross
// terms folded every 64th row, up to rho = 64.
//
// One GB300, us a launch before -> after (the FP64 or compensated FP32 kernel
// against this one; column_scales adds 34 + 8 us at 1M x 20):
//                            Y^T Y        Y R^-1       A^T G         G - A B
//   1M x 20 FP64             415 -> 150   436 -> 242
//   2.1M x 20 FP64           850 -> 303   911 -> 500   1689 -> 341   1531 -> 652
//   1M x 40 FP32             610 -> 445                1174 -> 626
// The integer multiply-adds' pipe bounds the applies (with FP32 cross terms 163,
// 335 and 421 us), it and the conversions of the cross terms the sums (131 us
// with those once in 64 rows).
#include "densefix.cuh"
#include "dense.cuh"
#include "krylov.cuh"

#include <algorithm>
#include <type_traits>

namespace ld {

namespace {

constexpr int kFT = 256;         // threads of the sums over rows
// Gram sums: H, the rows a thread sums before it folds (2^62 at most) and those
// whose FP32 cross terms it sums (below 2^31 units).  An FP32 block's entries
// have 24 bits, and the compensated sums before erred by 2^-48.
template <typename TY> struct Gram;
template <> struct Gram<double> { static constexpr int kBits = 29, kFold = 16, kCross = 4; };
template <> struct Gram<float> { static constexpr int kBits = 28, kFold = 64, kCross = 64; };
constexpr int kAtgFold = 64;     // A^T G: 64 2^56 = 2^62
// 2^f above this many times a column's mean magnitude flags the block.  (Gaussian
// columns reach 12 at a million rows and 16 at 2^31.)
template <typename TY> constexpr float max_over_mean() { return std::is_same<TY, double>::value ? 16.f : 64.f; }
constexpr int kAtgBits = 24;     // A^T G: entries as 24 + 32-bit integers
constexpr int kSlotRowsMax = 16384;
// Folded sums are kept in units of 2^fold_shift, so that a slot's stay below 2^62.
inline int fold_shift(int rows_slot, int bits) {
  int lg = 0;
  while ((1 << lg) < rows_slot) ++lg;
  return std::max(0, lg + bits - 62);
}
// Shared memory over all shapes (launch limits): sums (staged chunks of at most
// 2048 column slots, 8 bytes and A^T G's 4) and applies (64 columns).
constexpr int kSumsSmem = 16 * kFT * 8 + 2 * 2048 * (8 + 4);
constexpr int kAppRows = 128;                 // rows of an apply's chunk: four a lane
constexpr int kAppStride = kAppRows + 2;      // staged column stride: 16-byte steps, banks spread
constexpr int kAppSmem = kMaxSketch * kMaxSketch * 8 + 2 * kMaxSketch * kAppStride * 8;

// Elements of 2^f > |x| from the bits: the exponent of one above it.
__device__ __forceinline__ unsigned abs_word(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ unsigned abs_word(float x) { return __float_as_uint(x) & 0x7fffffff; }
template <typename TY> struct Bits;
template <> struct Bits<double> {
  static constexpr unsigned kInf = 0x7ff00000u;
  static __device__ __forceinline__ int exp(unsigned w) { return (int)(w >> 20) - 1022; }
  // |x| to 20 bits as FP32 (the conversion instruction runs on the FP64 pipe).
  static __device__ __forceinline__ float mag(unsigned w) {
    return w < (897u << 20) ? 0.f : w >= (1150u << 20) ? __uint_as_float(0x7f800000u)
                                                       : __uint_as_float((w - (896u << 20)) << 3);
  }
};
template <> struct Bits<float> {
  static constexpr unsigned kInf = 0x7f800000u;
  static __device__ __forceinline__ int exp(unsigned w) { return (int)(w >> 23) - 126; }
  static __device__ __forceinline__ float mag(unsigned w) { return __uint_as_float(w); }
};

// |x| 2^(H + 32 - f), truncated, and the sign as a mask; |x| < 2^f.
template <int H>
__device__ __forceinline__ unsigned long long to_fixed(double x, int f, int& m) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  unsigned long long w =
      ((unsigned long long)(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) | ((unsigned)lo << 11);
  asm("shr.b64 %0, %0, %1;" : "+l"(w) : "r"(1054 - H + f - ((hi >> 20) & 0x7ff)));  // (64 and more: 0)
  m = hi >> 31;
  return w;
}
template <int H>
__device__ __forceinline__ unsigned long long to_fixed(float x, int f, int& m) {
  const int b = __float_as_int(x);
  unsigned long long w = (unsigned long long)(((unsigned)b << 8) | 0x80000000u) << 32;
  asm("shr.b64 %0, %0, %1;" : "+l"(w) : "r"(158 - H + f - ((b >> 23) & 0xff)));
  m = b >> 31;
  return w;
}
// xh and the bits of xl.
template <int H, typename TY>
__device__ __forceinline__ int2 to_limbs(TY x, int f) {
  int m;
  const unsigned long long w = to_fixed<H>(x, f, m);
  const int lo = (int)(unsigned)w, hi = (int)(w >> 32) - (lo >> 31);
  return make_int2((hi ^ m) - m, __float_as_int((float)lo) ^ (m & 0x80000000));
}
// 30-bit limbs: X = xh 2^30 + xl below 2^60, 0 <= xl < 2^30 (rounded down).
__device__ __forceinline__ int2 to_limbs30(double x, int f) {
  int m;
  const unsigned long long w = to_fixed<28>(x, f, m);
  return make_int2((int)__funnelshift_r((unsigned)w, (unsigned)(w >> 32), 30) ^ m,
                   ((int)(unsigned)w ^ m) & 0x3fffffff);
}
// v 2^ex (|ex| far from the exponent's limits).
__device__ __forceinline__ double scaled(long long v, int ex) {
  const double d = (double)v;
  return v ? __hiloint2double(__double2hiint(d) + (ex << 20), __double2loint(d)) : 0.0;
}

template <typename TY>
__device__ __forceinline__ void copy_async(void* dst, const TY* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)), "l"(src), "n"((int)sizeof(TY))
               : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The elements (row, column) of a rows x s chunk that a thread takes, in
// steps of the CTA size without divisions in the loop.
struct Walk {
  int r, i, dr, di, s;
  __device__ __forceinline__ Walk(int s_)
      : r(threadIdx.x / s_), i(threadIdx.x % s_), dr(blockDim.x / s_), di(blockDim.x % s_), s(s_) {}
  __device__ __forceinline__ void next() {
    r += dr;
    i += di;
    if (i >= s) {
      i -= s;
      ++r;
    }
  }
};

// Largest |x| (its leading word) and sum of |x| per column: [s][CTA].
template <typename TY>
__global__ void __launch_bounds__(256) k_col_stats(const TY* __restrict__ Y, int ldy, int n, int s,
                                                   unsigned* __restrict__ mx, float* __restrict__ sum) {
  __shared__ unsigned sm[256];
  __shared__ float ss[256];
  const int R = 256 / s, r = threadIdx.x / s, i = threadIdx.x - r * s;
  unsigned m = 0;
  float a = 0.f;
  if (r < R) {
    const int step = gridDim.x * R;
    int row = blockIdx.x * R + r;
    for (; row + 3LL * step < n; row += 4 * step) {
      TY v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = __ldg(Y + (size_t)(row + u * step) * ldy + i);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const unsigned w = abs_word(v[u]);
        m = max(m, w);
        a += Bits<TY>::mag(w);
      }
    }
    for (; row < n; row += step) {
      const unsigned w = abs_word(__ldg(Y + (size_t)row * ldy + i));
      m = max(m, w);
      a += Bits<TY>::mag(w);
    }
  }
  sm[threadIdx.x] = m;
  ss[threadIdx.x] = a;
  __syncthreads();
  if (threadIdx.x < s) {
    for (int q = 1; q < R; ++q) {
      m = max(m, sm[q * s + threadIdx.x]);
      a += ss[q * s + threadIdx.x];
    }
    mx[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = m;
    sum[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = a;
  }
}

template <typename TY>
__global__ void __launch_bounds__(1024) k_col_exps(const unsigned* __restrict__ mx,
                                                   const float* __restrict__ sum, int cnt, int n,
                                                   int s, int* __restrict__ ex, int* __restrict__ bad) {
  __shared__ int any;
  if (threadIdx.x == 0) any = 0;
  __syncthreads();
  for (int c = threadIdx.x >> 5; c < s; c += 32) {
    unsigned m = 0;
    float a = 0.f;
    for (int q = threadIdx.x & 31; q < cnt; q += 32) {
      m = max(m, mx[(size_t)c * cnt + q]);
      a += sum[(size_t)c * cnt + q];
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      m = max(m, __shfl_xor_sync(~0u, m, o));
      a += __shfl_xor_sync(~0u, a, o);
    }
    if ((threadIdx.x & 31) == 0) {
      const int f = m ? Bits<TY>::exp(m) : 0;
      // (a column outside FP32's range has an infinite or zero sum)
      const bool ok = m < Bits<TY>::kInf && (m == 0 || (f > -100 && f < 100 && a < 3e38f &&
                                                        ldexpf(1.f, f) <= max_over_mean<TY>() * (a / (float)n)));
      ex[c] = ok ? f : 0;
      if (!ok) any = 1;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) *bad = any;
}

__device__ __forceinline__ void unrank_tile(int q, int s, int& i, int& j) {
  i = 0;
  while (q >= s - i) {
    q -= s - i;
    ++i;
  }
  j = i + q;
}

// Sums over rows: a thread owns a 4 x 4 tile of column pairs (of the upper
// triangle for the Gram matrix, of A x G for A^T G) and every RS-th row of the
// staged chunks, so that eight column loads feed 16 products; the
// tiles times the row subsets fill the CTA.  A chunk is copied in while the
// one before it is summed and converted in place by the threads that copied
// it.  The integer sums are exact for Gram::kFold (kAtgFold) rows, then whole
// units of 2^shift go to shared memory and the remainder stays, so that a slot
// rounds once, at its end: by 2^-63 rows 2^2f at most.  The product xl yl is left
// out but on the diagonal of FP64 blocks, where it is never negative: it would sum to
// 2^-2H / 12 a row.
template <typename TY, bool ATG>
__global__ void __launch_bounds__(kFT, 2)
    k_sums_fix(const TY* __restrict__ Y, int ldy, int n, int s, int r, uint64_t key,
               const uint64_t* __restrict__ keyp, const int* __restrict__ ex,
               const int* __restrict__ bad, int rows_slot, int nslots, int RS, int chunk,
               int shift, double* __restrict__ part) {
  if (*bad) return;
  if constexpr (ATG)
    if (keyp) key = *keyp;
  constexpr bool kExact = !ATG && std::is_same<TY, double>::value;
  extern __shared__ __align__(16) unsigned char smem_df[];
  const int s4 = (s + 3) / 4, r4 = (r + 3) / 4, SP = 4 * s4, GP = 4 * r4;
  const int nt = ATG ? s4 * r4 : s4 * (s4 + 1) / 2;
  long long* T = reinterpret_cast<long long*>(smem_df);                // [16][kFT]
  int2* buf = reinterpret_cast<int2*>(T + 16 * kFT);                   // [2][chunk][SP]
  int* gbuf = reinterpret_cast<int*>(buf + 2 * (size_t)chunk * SP);    // [2][chunk][GP]
  __shared__ int se[kMaxSketch];
  for (int c = threadIdx.x; c < s; c += kFT) se[c] = ex[c];
  if (SP > s || (ATG && GP > r)) {  // columns past the last are zero
    for (int e = threadIdx.x; e < 2 * chunk * SP; e += kFT) buf[e] = make_int2(0, 0);
    if (ATG)
      for (int e = threadIdx.x; e < 2 * chunk * GP; e += kFT) gbuf[e] = 0;
  }
  const int rs = threadIdx.x / nt, t = threadIdx.x - rs * nt;
  const bool live = rs < RS;
  int ti, tj;
  if constexpr (ATG) {
    ti = t / r4;
    tj = t - ti * r4;
  } else {
    unrank_tile(t, s4, ti, tj);
  }
  __syncthreads();

  for (int slot = blockIdx.x; slot < nslots; slot += gridDim.x) {
    const int row0 = slot * rows_slot;
    const int row1 = (int)min((long long)row0 + rows_slot, (long long)n);
    auto stage = [&](int c0, int2* dst) {
      const int rows = min(chunk, row1 - c0);
      const TY* src = Y + (size_t)c0 * ldy;
      for (Walk w(s); w.r < rows; w.next())
        copy_async(dst + w.r * SP + w.i, src + (size_t)w.r * ldy + w.i);
    };
    long long hh[16], all[4] = {0, 0, 0, 0};
    float cr[16], sq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int v = 0; v < 16; ++v) {
      hh[v] = 0;
      cr[v] = 0.f;
      T[v * kFT + threadIdx.x] = 0;
    }
    // half: 0 (the remainder is kept), or at a slot's end half a unit.
    auto fold = [&](long long half) {
      const long long mask = (1LL << shift) - 1;
#pragma unroll
      for (int v = 0; v < 16; ++v) {
        const long long S = ATG ? (long long)((unsigned long long)all[v >> 2] - 2ULL * (unsigned long long)hh[v])
                                : hh[v] + __float2ll_rn(cr[v] * 0x1p-32f);
        T[v * kFT + threadIdx.x] += (S + half) >> shift;
        // A^T G: the remainder as all - 2 hh again, all its parity (that of every
        // S of the column).
        hh[v] = ATG ? ((all[v >> 2] & mask & 1) - (S & mask)) >> 1 : S & mask;
        cr[v] = 0.f;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) all[q] &= mask & 1;
    };
    const int per = (chunk + RS - 1) / RS;  // rows of a chunk a thread takes
    int cnt = 0, cur = 0, it = 0;
    stage(row0, buf);
    for (int c0 = row0; c0 < row1; c0 += chunk, cur ^= 1) {
      const int rows = min(chunk, row1 - c0);
      int2* b = buf + (size_t)cur * chunk * SP;
      int* gb = gbuf + (size_t)cur * chunk * GP;
      copy_wait();
      for (Walk w(s); w.r < rows; w.next()) {
        int2* p = b + w.r * SP + w.i;
        const TY x = *reinterpret_cast<const TY*>(p);
        if constexpr (ATG) {
          int m;
          const long long X = (long long)to_fixed<kAtgBits>(x, se[w.i], m);
          *reinterpret_cast<long long*>(p) = (X ^ (long long)m) - m;
        } else {
          *p = to_limbs<Gram<TY>::kBits>(x, se[w.i]);
        }
      }
      if constexpr (ATG)
        for (Walk w(r); w.r < rows; w.next())
          gb[w.r * GP + w.i] = (int)probe_sign(key, (uint32_t)w.i, (uint32_t)(c0 + w.r));
      __syncthreads();  // the chunk is converted; the other buffer's readers are done
      if (c0 + chunk < row1) stage(c0 + chunk, buf + (size_t)(cur ^ 1) * chunk * SP);
      if (live) {
        if (cnt + per > (ATG ? kAtgFold : Gram<TY>::kFold)) {
          fold(0);
          cnt = 0;
        }
        cnt += per;
        for (int rr = rs; rr < rows; rr += RS) {
          const int4* pa = reinterpret_cast<const int4*>(b + rr * SP + 4 * ti);
          if constexpr (ATG) {
            // sum g x = sum x - 2 (sum of x where g = -1): predicated additions.
            const longlong2* px = reinterpret_cast<const longlong2*>(pa);
            const longlong2 x0 = px[0], x1 = px[1];
            const long long x[4] = {x0.x, x0.y, x1.x, x1.y};
            const int4 g4 = *reinterpret_cast<const int4*>(gb + rr * GP + 4 * tj);
            const int g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              all[q] += x[q];
              asm("{.reg .pred p;\n setp.lt.s32 p, %8, 0;\n @p add.s64 %0, %0, %4;\n @p add.s64 %1, %1, %5;\n"
                  " @p add.s64 %2, %2, %6;\n @p add.s64 %3, %3, %7;}"
                  : "+l"(hh[q]), "+l"(hh[4 + q]), "+l"(hh[8 + q]), "+l"(hh[12 + q])
                  : "l"(x[0]), "l"(x[1]), "l"(x[2]), "l"(x[3]), "r"(g[q]));
            }
          } else {
            const int4* pb = reinterpret_cast<const int4*>(b + rr * SP + 4 * tj);
            const int4 a0 = pa[0], a1 = pa[1], b0 = pb[0], b1 = pb[1];
            const int ah[4] = {a0.x, a0.z, a1.x, a1.z}, bh[4] = {b0.x, b0.z, b1.x, b1.z};
            const float al[4] = {__int_as_float(a0.y), __int_as_float(a0.w), __int_as_float(a1.y),
                                 __int_as_float(a1.w)};
            const float bl[4] = {__int_as_float(b0.y), __int_as_float(b0.w), __int_as_float(b1.y),
                                 __int_as_float(b1.w)};
            float af[4], bf[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              af[q] = (float)ah[q];
              bf[q] = (float)bh[q];
            }
#pragma unroll
            for (int v = 0; v < 16; ++v) {
              hh[v] += (long long)ah[v >> 2] * bh[v & 3];
              cr[v] = fmaf(af[v >> 2], bl[v & 3], cr[v]);
              cr[v] = fmaf(al[v >> 2], bf[v & 3], cr[v]);
            }
            if constexpr (kExact) {
              if (ti == tj) {
#pragma unroll
                for (int q = 0; q < 4; ++q) sq[q] = fmaf(al[q], bl[q], sq[q]);
              }
              if (++it == Gram<TY>::kCross) {
                it = 0;
#pragma unroll
                for (int v = 0; v < 16; ++v) {
                  hh[v] += __float2int_rn(cr[v] * 0x1p-32f);
                  cr[v] = 0.f;
                }
              }
            }
          }
        }
      }
    }
    if (live) {
      if constexpr (kExact) {
#pragma unroll
        for (int q = 0; q < 4; ++q) hh[5 * q] += __float2ll_rn(sq[q] * 0x1p-64f);
      }
      fold(shift ? 1LL << (shift - 1) : 0);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 16 * nt; e += kFT) {
      const int v = e / nt, q = e - v * nt;
      int qi, qj;
      if constexpr (ATG) {
        qi = q / r4;
        qj = q - qi * r4;
      } else {
        unrank_tile(q, s4, qi, qj);
      }
      const int i = 4 * qi + (v >> 2), j = 4 * qj + (v & 3);
      if (i >= s || j >= (ATG ? r : s) || (!ATG && i > j)) continue;
      long long a = 0;
      for (int z = 0; z < RS; ++z) a += T[v * kFT + z * nt + q];
      const int pair = ATG ? i * r + j : i * s - i * (i - 1) / 2 + (j - i);
      const int f = shift + (ATG ? se[i] - kAtgBits - 32 : se[i] + se[j] - 2 * Gram<TY>::kBits);
      part[(size_t)pair * nslots + slot] = scaled(a, f);
    }
    __syncthreads();
  }
}

// Applies: warp w owns four output columns, a lane four rows of the chunk
// (2 lane, 2 lane + 1 and the same in its second half: 16-byte reads without
// bank conflicts), so that four loads feed 16 products.  Staged by column,
// copied one chunk ahead, converted in place.  The factor's columns are scaled
// so that their absolute sums (times the block's scales) stay below one, which
// bounds sum |yh rh| by 2^60 and sum |yl rh| by 2^60; |yh rl| is below 2^59, so
// the cross terms are folded every eighth product.  All three products of the
// limbs are integer ones: with FP32 cross terms, whose sum over i is as large as
// the result's own 24 leading bits, the columns of an orthogonalised 4,883 x 64
// block were off by 6.9e-16 of their norm (FP64 kernels 0.9e-16).  The warps'
// triangular loops differ in length: the columns rotate over the warps from
// CTA to CTA, so that an SM's sub-partitions are loaded alike.
template <bool PROJ>
__global__ void __launch_bounds__(512, 1)
    k_apply_fix(const double* Y, int ldy, int n, int s, int r, const double* __restrict__ Rm,
                const int* __restrict__ ex, const int* __restrict__ bad, uint64_t key,
                const uint64_t* __restrict__ keyp, double* A, int lda) {
  if (*bad) return;
  if constexpr (PROJ)
    if (keyp) key = *keyp;
  extern __shared__ __align__(16) unsigned char smem_df[];
  const int r4 = (r + 3) / 4, rc = 4 * r4;
  int2* rt = reinterpret_cast<int2*>(smem_df);   // [s][rc]
  int2* buf = rt + s * rc;                       // [2][s][kAppStride]
  __shared__ int ke[kMaxSketch + 4], se[kMaxSketch];
  {
    double* rd = reinterpret_cast<double*>(buf);
    for (int e = threadIdx.x; e < s * r; e += blockDim.x) rd[e] = Rm[e];
    for (int c = threadIdx.x; c < s; c += blockDim.x) se[c] = ex[c];
    __syncthreads();
    // ke[l]: sum_i |R_il| 2^f_i < 2^ke, from 21-bit mantissas rounded up.
    for (int l = threadIdx.x; l < r; l += blockDim.x) {
      int km = -4000;
      for (int i = 0; i < s; ++i) {
        const unsigned w = abs_word(rd[i * r + l]);
        if (w >> 20) km = max(km, (int)(w >> 20) - 1023 + se[i]);
      }
      unsigned sum = 0;
      for (int i = 0; i < s; ++i) {
        const unsigned w = abs_word(rd[i * r + l]);
        if (w >> 20) {
          const int d = km - ((int)(w >> 20) - 1023 + se[i]);
          sum += ((((w & 0xfffffu) | 0x100000u) + 1) >> min(d, 31)) + 1;
        }
      }
      int k = sum ? km - 20 + 32 - __clz(sum) : 0;
      ke[l] = PROJ ? max(k, 0) : k;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < s * rc; e += blockDim.x) {
      const int i = e / rc, l = e - i * rc;
      int2 a = make_int2(0, 0);
      if (l < r) {
        a = to_limbs30(rd[i * r + l], ke[l] - se[i]);
        if (a.y >= 1 << 29) ++a.x, a.y -= 1 << 30;  // (|rl| <= 2^29)
      }
      rt[e] = a;
    }
    __syncthreads();
  }
  const int lane = threadIdx.x & 31;
  const int lt = (int)((threadIdx.x >> 5) + blockIdx.x) % r4;
  const int imax = PROJ ? s : min(4 * lt + 4, s);
  auto stage = [&](int c0, int2* dst) {
    const int rows = min(kAppRows, n - c0);
    const double* src = Y + (size_t)c0 * ldy;
    for (Walk w(s); w.r < rows; w.next())
      copy_async(dst + w.i * kAppStride + w.r, src + (size_t)w.r * ldy + w.i);
  };
  int cur = 0;
  const int step = gridDim.x * kAppRows;
  if (blockIdx.x * kAppRows < n) stage(blockIdx.x * kAppRows, buf);
  for (int c0 = blockIdx.x * kAppRows; c0 < n; c0 += step, cur ^= 1) {
    const int rows = min(kAppRows, n - c0);
    int2* b = buf + cur * s * kAppStride;
    copy_wait();
    for (Walk w(s); w.r < rows; w.next()) {
      int2* p = b + w.i * kAppStride + w.r;
      *p = to_limbs30(*reinterpret_cast<const double*>(p), se[w.i]);
    }
    __syncthreads();
    if (n - c0 > step) stage(c0 + step, buf + (cur ^ 1) * s * kAppStride);
    long long hh[16], cr[16];
#pragma unroll
    for (int v = 0; v < 16; ++v) hh[v] = cr[v] = 0;
    const int4* py = reinterpret_cast<const int4*>(b) + lane;
    const int4* pr = reinterpret_cast<const int4*>(rt + 4 * lt);
#pragma unroll 2
    for (int i = 0; i < imax; ++i, py += kAppStride / 2, pr += rc / 2) {
      const int4 y0 = py[0], y1 = py[kAppRows / 4], r0 = pr[0], r1 = pr[1];
      const int yh[4] = {y0.x, y0.z, y1.x, y1.z}, yl[4] = {y0.y, y0.w, y1.y, y1.w};
      const int rh[4] = {r0.x, r0.z, r1.x, r1.z}, rl[4] = {r0.y, r0.w, r1.y, r1.w};
#pragma unroll
      for (int v = 0; v < 16; ++v) {
        hh[v] += (long long)yh[v >> 2] * rh[v & 3];
        cr[v] += (long long)yh[v >> 2] * rl[v & 3];
        cr[v] += (long long)yl[v >> 2] * rh[v & 3];
      }
      if ((i & 7) == 7) {
#pragma unroll
        for (int v = 0; v < 16; ++v) {
          hh[v] += cr[v] >> 30;
          cr[v] &= 0x3fffffff;
        }
      }
    }
    const bool pairs = !((uintptr_t)A & 15) && !(lda & 1);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int row = 2 * lane + (u & 1) + (u >> 1) * (kAppRows / 2);
      if (row >= rows) continue;
      double o[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int l = 4 * lt + q, k = l < r ? ke[l] : 0;
        // In units of 2^(k - 60); g = +-1 joins the integer.
        long long V = hh[4 * u + q] + ((cr[4 * u + q] + (1 << 29)) >> 30);
        if constexpr (PROJ)
          V = (long long)probe_sign(key, (uint32_t)l, (uint32_t)(c0 + row)) * (1LL << (60 - min(k, 60))) - V;
        o[q] = scaled(V, k - 60);
      }
      double* dst = A + (size_t)(c0 + row) * lda + 4 * lt;
      if (pairs && 4 * lt + 4 <= r) {
        *reinterpret_cast<double2*>(dst) = make_double2(o[0], o[1]);
        *reinterpret_cast<double2*>(dst + 2) = make_double2(o[2], o[3]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (4 * lt + q < r) dst[q] = o[q];
      }
    }
  }
}

// Resident CTAs of a persistent grid.
template <typename K>
int resident(K kern, int threads, size_t smem) {
  int fit = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, threads, smem) != cudaSuccess || fit < 1) {
    (void)cudaGetLastError();
    fit = 1;
  }
  return fit * sm_count();
}

int slot_rows(int n) {
  const int want = div_up(div_up(n, 2 * sm_count()), 256) * 256;
  return std::max(256, std::min(want, kSlotRowsMax));
}

int stat_grid(int n, int s) { return std::max(1, std::min(4 * sm_count(), div_up(n, 256 / s * 4))); }

template <typename TY, bool ATG>
int sums_fix(const TY* Y, int ldy, int n, int s, int r, uint64_t key, const uint64_t* keyp,
             const ColScales& c, double* part, cudaStream_t st) {
  const int s4 = div_up(s, 4), r4 = div_up(r, 4);
  const int nt = ATG ? s4 * r4 : s4 * (s4 + 1) / 2;
  const int RS = kFT / nt, wide = 4 * (ATG ? std::max(s4, r4) : s4);
  const int chunk = RS * std::max(1, std::min(ATG ? 32 : std::min(32, Gram<TY>::kFold), 2048 / (RS * wide)));
  const size_t smem = 16 * kFT * 8 + 2 * (size_t)chunk * 4 * s4 * 8 + (ATG ? 2 * (size_t)chunk * 4 * r4 * 4 : 0);
  auto kern = k_sums_fix<TY, ATG>;
  LD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSumsSmem));
  const int nslots = densefix_slots(n);
  kern<<<std::min(nslots, resident(kern, kFT, smem)), kFT, smem, st>>>(
      Y, ldy, n, s, r, key, keyp, c.exp, c.bad, slot_rows(n), nslots, RS, chunk,
      fold_shift(slot_rows(n), ATG ? kAtgBits + 32 : 2 * Gram<TY>::kBits), part);
  LD_CHECK_LAUNCH();
  return LOGDET_OK;
}

template <bool PROJ>
int apply_launch(const double* Y, int ldy, int n, int s, int r, const double* Rm, const ColScales& c,
                 uint64_t key, const uint64_t* keyp, double* A, int lda, cudaStream_t st) {
  const int r4 = div_up(r, 4), threads = 32 * r4;
  const size_t smem = (size_t)s * 4 * r4 * 8 + 2 * (size_t)s * kAppStride * 8;
  auto kern = k_apply_fix<PROJ>;
  LD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kAppSmem));
  kern<<<std::min(div_up(n, kAppRows), resident(kern, threads, smem)), threads, smem, st>>>(
      Y, ldy, n, s, r, Rm, c.exp, c.bad, key, keyp, A, lda);
  LD_CHECK_LAUNCH();
  return LOGDET_OK;
}
}  // namespace

bool densefix_ok(int n, int s, bool fp32) {
  return s > 0 && (double)n * s * s >= (fp32 ? 2e8 : 2e7);
}

// Whole orthogonalisations, us, FP64 kernels / these, by n s^2: s = 7, 1e7
// 167/161, 2e7 222/199; 20, 1e7 155/179, 2e7 216/197, 4e7 285/244; 32, 2e7
// 239/234, 4e7 347/257; 40, 2e7 264/291, 3e7 279/295, 4e7 367/323; 50, 3e7
// 370/386, 4e7 390/390, 6e7 535/433; 64, 4e7 526/563, 6e7 597/565 (wide blocks
// have few slots of many column pairs).  FP32: s = 7, 1e8 526/368; 20, 1e8
// 227/248, 2e8 352/353, 4e8 679/610; 32, 4e8 622/585; 40, 4e8 574/586, 8e8
// 1043/953; 50, 8e8 972/1055, 1.6e9 1717/1792 (of 256 threads 182 have a tile).
bool densefix_orth_ok(int n, int s, bool fp32) {
  if (!densefix_ok(n, s, fp32)) return false;
  const double w = (double)n * s * s;
  return fp32 ? s <= 48 && w >= 4e7 * s - 1.08e9 : w >= 1e6 * s - 1.2e7;
}

size_t densefix_workspace_doubles(int s) { return (size_t)s * 4 * sm_count() + kMaxSketch + 2; }

int densefix_slots(int n) { return div_up(n, slot_rows(n)); }

template <typename TY>
int column_scales(const TY* Y, int ldy, int n, int s, double* ws, ColScales* out, cudaStream_t st) {
  const int grid = stat_grid(n, s);
  unsigned* mx = reinterpret_cast<unsigned*>(ws);
  float* sum = reinterpret_cast<float*>(mx + (size_t)s * grid);
  out->exp = reinterpret_cast<int*>(ws + (size_t)s * grid);
  out->bad = out->exp + kMaxSketch;
  k_col_stats<TY><<<grid, 256, 0, st>>>(Y, ldy, n, s, mx, sum);
  LD_CHECK_LAUNCH();
  k_col_exps<TY><<<1, 1024, 0, st>>>(mx, sum, grid, n, s, out->exp, out->bad);
  LD_CHECK_LAUNCH();
  return LOGDET_OK;
}
template int column_scales<double>(const double*, int, int, int, double*, ColScales*, cudaStream_t);
template int column_scales<float>(const float*, int, int, int, double*, ColScales*, cudaStream_t);

template <typename TY>
int gram_fix(const TY* Y, int ldy, int n, int s, const ColScales& c, double* part, cudaStream_t st) {
  return sums_fix<TY, false>(Y, ldy, n, s, s, 0, nullptr, c, part, st);
}
template int gram_fix<double>(const double*, int, int, int, const ColScales&, double*, cudaStream_t);
template int gram_fix<float>(const float*, int, int, int, const ColScales&, double*, cudaStream_t);

template <typename TY>
int atg_fix(const TY* A, int lda, int n, int s, int r, uint64_t key, const uint64_t* keyp,
            const ColScales& c, double* part, cudaStream_t st) {
  return sums_fix<TY, true>(A, lda, n, s, r, key, keyp, c, part, st);
}
template int atg_fix<double>(const double*, int, int, int, int, uint64_t, const uint64_t*,
                             const ColScales&, double*, cudaStream_t);
template int atg_fix<float>(const float*, int, int, int, int, uint64_t, const uint64_t*,
                            const ColScales&, double*, cudaStream_t);

int apply_fix(const double* Y, int ldy, int n, int s, const double* Rinv, double* A, int lda,
              const ColScales& c, cudaStream_t st) {
  return apply_launch<false>(Y, ldy, n, s, s, Rinv, c, 0, nullptr, A, lda, st);
}
int project_fix(const double* A, int lda, int n, int s, int r, uint64_t key, const uint64_t* keyp,
                const double* B, double* X, int ldx, const ColScales& c, cudaStream_t st) {
  return apply_launch<true>(A, lda, n, s, r, B, c, key, keyp, X, ldx, st);
}
}  // namespace ld
