// FP64 SpMM pass of grid stencil matrices in fixed point.
//
// An FP64 instruction takes a sub-partition 64 clocks and more on this GPU (78
// measured), a 32 x 32 + 64-bit integer multiply-add 4.7, so the product y = A x of an FP64 block
// is summed in integers.  Each column of x becomes X = x 2^60 / F (truncated
// to an integer below 2^60), F a power of two 32 to 128 times the column's
// root mean square (from sigma, which is 1 / |u|), and each matrix entry
// A = a 2^(60 - ka), with 2^ka above the largest absolute row sum.  With
// X = xh 2^30 + xl and A = ah 2^30 + al,
//
//   sum A X = 2^60 sum ah xh + 2^30 sum (ah xl + al xh) + sum al xl
//
// three multiply-adds a term (the last sum is below one unit of the result
// and left out); no sum overflows: |sum ah xh| <= 2^60, and the cross sum
// stays below 2^63 for up to 13 entries (longer rows fold it every eight).
// The result is rounded to FP64 once.  Its error, a few units of 2^-60 F, is
// below that of an FP64 sum, which rounds every product and addition to 2^-53
// of its size.  (x and the entries are cut at 2^-60 of F and of the largest row
// sum, so a number far below those keeps fewer bits than FP64's 53; a product's
// error is measured by the norms, as the recurrences use it.)  Quadratic forms of
// 12 Lanczos steps against extended precision, 120 probes each, rms error here /
// of the CSR pass: 3D Laplacian 1.25e-15 / 1.02e-15, 2D 0.90e-15 / 1.44e-15,
// Matern 0.29e-15 / 0.52e-15.  An entry of x too large for its column's F (or not finite) sets
// the job's flag; k_spmm_fix_general, launched after every product, then redoes
// it with FP64 arithmetic, and takes the job's later products alone.
//
// x arrives as in the FP32 sweeps (dia.cu): a CTA sweeps a segment of a line
// (2D) or a tile of a plane (3D) over consecutive lines or planes, keeping
// the windows that the current one needs in a ring of shared memory filled by
// TMA.  Each window is converted in place once, when it arrives, instead of
// once per diagonal; the entries' fixed-point values come by plain loads, one
// line ahead in registers.
//
// 3D Laplacian 128^3, 60 probes: 1.17 -> 0.69 ms a pass of 40 columns with one
// dot (59.6 -> 35.0 ms a solve), 123 -> 84 ms a window-4 solve; the CSR pass
// stands at 90 % of the FP64 peak there.
//
// The dot x . y is summed in integers too; the dots with other window vectors
// are FP64 multiply-adds on the rounded y.
#include "fix.cuh"
#include "profile.cuh"
#include "tma.cuh"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

namespace ld {

namespace {

// Two CTAs of 256 threads per SM, so that one converts while the other sums.
// One of 512 (larger tiles, fewer converted points) gains 5 % with one dot and
// loses 8 % with four; 320 threads, three CTAs of 160, and two windows ahead
// of the line instead of one (smaller tiles) all lose 1 to 8 %: the time is
// the instructions' (of a 128^3 single-dot pass 0.35 ms in the sums, 0.1 in
// the conversions, the rest waits and barriers).
constexpr int kFixThreads = 256;
constexpr int kFixSmem = 112 * 1024;           // per CTA
constexpr int kFixValRegs = 4;                 // values a thread loads ahead
constexpr int kFixPoints = 4;                  // points of a line or plane a thread takes
constexpr int kFixMaxWindows = 15;              // ring slots: a barrier each, in 128 bytes with `skip`
constexpr int kFixAhead = 1;                    // windows loaded ahead of the current line's
constexpr int kFixMaxWidth = 128;              // TMA box: 256 words

__host__ __device__ inline int fix_win_points(const DiaInfo& d, int T, int tx, int ty) {
  return d.dim == 3 ? (tx + 2 * d.Ax) * (ty + 2 * d.Ay) : T + d.cw;
}
__host__ __device__ inline int round128(int bytes) { return (bytes + 127) / 128 * 128; }

// Shared memory of a CTA: barriers, window offsets, dot reduction, two lines
// of values, the ring.
struct FixSmem {
  int tab, red, vals, ring, slot, total;
};
__host__ __device__ inline FixSmem fix_smem(const DiaInfo& d, int T, int tx, int ty, int width) {
  FixSmem s;
  const int nr = 2 * d.A + 1 + kFixAhead;
  s.tab = 128;
  s.red = s.tab + round128(nr * kMaxDiags * 4);
  s.vals = s.red + round128(kFixThreads * 16);
  s.ring = s.vals + 2 * round128(T * d.ndiag * 8);
  s.slot = round128(fix_win_points(d, T, tx, ty) * width * 8);
  s.total = s.ring + nr * s.slot;
  return s;
}

struct FixUnit {
  int gu, jb, seg0, segT, k0, nl;  // as SwUnit in dia.cu
};
// Unit gu; with SKIP, the CTA's first one from gu on whose job is not in *skip.
template <int DIM, bool SKIP>
__device__ __forceinline__ void fix_unit(FixUnit& U, const SpmmBatch<double>& B, int gu,
                                         const volatile unsigned* skip) {
  static_assert(kMaxJobs <= 32, "one bit a job");
  if constexpr (SKIP)
    while (gu < B.total_tiles && (*skip >> find_job(B, gu) & 1u)) gu += gridDim.x;
  U.gu = gu;
  if (gu >= B.total_tiles) return;
  U.jb = find_job(B, gu);
  const SpmmJob<double>& J = B.jobs[U.jb];
  const DiaInfo& D = J.dinfo;
  const int u = gu - B.tile_start[U.jb];
  const int seg = u % J.dia_nseg, chunk = u / J.dia_nseg;
  if constexpr (DIM == 3) {
    const int nsx = (D.L + J.dia_tx - 1) >> J.dia_txs;
    U.seg0 = (seg % nsx) << J.dia_txs;
    U.segT = seg / nsx * J.dia_ty;
  } else {
    U.seg0 = seg * J.dia_T;
    U.segT = min(J.dia_T, D.L - U.seg0);
  }
  U.k0 = chunk * J.dia_kc;
  U.nl = min(J.dia_kc, J.dia_nlines - U.k0);
}

// One warp: the jobs whose flag is set, a bit each.
__device__ __forceinline__ unsigned jobs_out_of_range(const SpmmBatch<double>& B) {
  const int j = threadIdx.x & 31;
  return __ballot_sync(~0u, j < B.njobs && __ldcg(B.jobs[j].bad) != 0);
}

// Row of point p of a unit's line or plane k, or -1 outside the grid.
template <int DIM>
__device__ __forceinline__ int fix_row(const SpmmJob<double>& J, const FixUnit& U, int k, int p) {
  const DiaInfo& D = J.dinfo;
  if constexpr (DIM == 3) {
    const int x = U.seg0 + (p & (J.dia_tx - 1)), y = U.segT + (p >> J.dia_txs);
    return p < J.dia_T && x < D.L && y < D.ny ? k * D.P + y * D.L + x : -1;
  } else {
    const int row = U.seg0 + p + k * D.L;
    return p < U.segT && row < J.n ? row : -1;
  }
}

// Thread 0: arm the barrier and copy window q (line or plane k0 - A + q).
template <int DIM>
__device__ __forceinline__ void fix_issue(const SpmmJob<double>& J, const FixUnit& U, int q,
                                          uint32_t dst, uint32_t bar, unsigned extra_tx) {
  const DiaInfo& D = J.dinfo;
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  mbar_expect_tx(bar, (uint32_t)fix_win_points(D, J.dia_T, J.dia_tx, J.dia_ty) * J.width * 8 + extra_tx);
  if constexpr (DIM == 3)
    tma_load_4d(dst, &J.tmap, 2 * J.col_off, U.seg0 - D.Ax, U.segT - D.Ay, U.k0 - D.A + q, bar);
  else
    tma_load_2d(dst, &J.tmap, 2 * J.col_off, U.seg0 + (U.k0 - D.A + q) * D.L + D.cmin, bar);
}

// x = +-M 2^(e - 1075) to X = xh 2^30 + xl, 0 <= xl < 2^30: M << 11 is
// shifted right by K - e, K = 1026 + log2 F; 4 is the least shift that keeps
// the magnitude below 2^60 (a smaller one is reported through rmin).  A
// negative number is complemented, which is one unit below its negation.
__device__ __forceinline__ void to_fixed(int lo, int hi, int K, int& xh, int& xl, int& rmin) {
  const int r = K - ((hi >> 20) & 0x7ff);
  rmin = min(rmin, r);
  const unsigned wh = __funnelshift_l(lo, hi, 11) | 0x80000000u, wl = (unsigned)lo << 11;
  unsigned long long w = ((unsigned long long)wh << 32) | wl;
  asm("shr.b64 %0, %0, %1;" : "+l"(w) : "r"(r));  // (shifts of 64 and more give 0)
  const int m = hi >> 31;
  xl = ((int)(unsigned)w ^ m) & 0x3fffffff;
  xh = (int)__funnelshift_r((unsigned)w, (unsigned)(w >> 32), 30) ^ m;
}

// v 2^ex rounded to FP64: the conversion runs on the FP64 pipe, 64 clocks; in
// integers (magnitude, leading one, shifts, rounding: about 20 instructions)
// it was slower, 88 ms against 84 for the passes of a window-4 solve.
__device__ __forceinline__ double from_fixed(long long v, int ex) {
  const double d = (double)v;
  return v ? __hiloint2double(__double2hiint(d) + (ex << 20), __double2loint(d)) : 0.0;
}

// log2 F of column p of a job.
__device__ __forceinline__ int fix_exp(const SpmmJob<double>& J, int p) {
  if (!J.sig) return J.xexp;
  const int e = ((__double2hiint(__ldcg(J.sig + (size_t)p * J.sig_stride)) >> 20) & 0x7ff) - 1023;
  return 5 - e - J.hn;
}

// NOTH: window vectors other than x itself, dotted in FP64 (a conversion and
// three multiply-adds a term would cost more).  SELF: the last dot is x . y,
// summed in integers from the window's converted x and the unrounded y:
// about 11 instructions against a load and a 64-clock DFMA (window-4 solve:
// 98 -> 84 ms with the conversion above; a single dot: unchanged).
// MANY: several jobs a launch.  Jobs whose flag is set already are the general
// kernel's alone (their vectors have left the range, mostly for good): a lone
// one ends the launch at once, of several the units are skipped.  Either reads
// the flags once for the whole CTA, since another CTA may be setting one.  (The
// skipping cost a lone 128^3 single-dot pass 1 to 2 %, through the compiler's
// schedule of the sums: 683 us against 695.)
template <int NOTH, bool SELF, int NDC, int DIM, bool MANY>
__global__ void __launch_bounds__(kFixThreads, 2)
    k_spmm_fix(const __grid_constant__ SpmmBatch<double> B, unsigned extra_tx,
               unsigned long long wait_ns) {
  constexpr int kDiags = NDC > 0 ? NDC : kMaxDiags;
  constexpr int V = 2;
  constexpr bool kEarly = NOTH <= 3;  // window vectors loaded before the sums
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const uint32_t bar0 = smem_addr(smem_raw);
  int* xo_tab = reinterpret_cast<int*>(smem_raw + 128);
  volatile unsigned* skip = reinterpret_cast<unsigned*>(smem_raw + 8 * kFixMaxWindows);
  if constexpr (MANY) {
    if (threadIdx.x < 32) {
      const unsigned out = jobs_out_of_range(B);
      if (threadIdx.x == 0) *skip = out;
    }
    __syncthreads();
  } else {
    if (__syncthreads_or(threadIdx.x == 0 && __ldcg(B.jobs[0].bad))) return;
  }
  FixUnit C;
  fix_unit<DIM, MANY>(C, B, blockIdx.x, skip);
  if (C.gu >= B.total_tiles) return;
  // Every job of a launch has the same matrix structure constants up to its
  // sizes; the ring is laid out per job, so a CTA drains before it changes.
  int cur_jb = -1;
  int nr = 0;
  FixSmem M{};
  double acc_s[NOTH > 0 ? NOTH : 1][V];
  __int128 self[V] = {0, 0};  // sum of X Y / 2^30
  int G = 1, R = 1, r = 0, g = 0, nd = 0, width = 0, A = 0, col0 = 0, ldy = 0, noth = 0, dself = 0;
  int K[V], ex[V], rmin = 1 << 20;
  bool live = false;
  if (threadIdx.x == 0) {
    for (int q = 0; q < kFixMaxWindows; ++q) mbar_init(bar0 + 8 * q, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  FixUnit P = C;
  int pq = 0, issued = 0, pslot = 0;              // producer (thread 0 issues)
  int t0 = 0, wnext = 0, wslot = 0, rslot = 0;    // consumer, as in dia.cu
  uint32_t phases = 0;
#pragma unroll
  for (int d = 0; d < (NOTH > 0 ? NOTH : 1); ++d) acc_s[d][0] = acc_s[d][1] = 0.0;

  // Loads up to nr windows past `released`, of units of the current job.
  auto produce = [&](int released) {
    while (P.gu < B.total_tiles && P.jb == cur_jb && issued < released + nr) {
      const SpmmJob<double>& J = B.jobs[P.jb];
      if (threadIdx.x == 0)
        fix_issue<DIM>(J, P, pq, bar0 + M.ring + pslot * M.slot, bar0 + 8 * pslot, extra_tx);
      ++issued;
      if (++pslot == nr) pslot = 0;
      if (++pq == P.nl + 2 * J.dinfo.A) {
        fix_unit<DIM, MANY>(P, B, P.gu + gridDim.x, skip);
        pq = 0;
      }
    }
  };

  while (C.gu < B.total_tiles) {
    const SpmmJob<double>& J = B.jobs[C.jb];
    const DiaInfo& D = J.dinfo;
    if (C.jb != cur_jb) {
      // (the last unit's reads ended at a barrier, every load was waited for)
      cur_jb = C.jb;
      nd = NDC > 0 ? NDC : D.ndiag;
      A = D.A;
      nr = 2 * A + 1 + kFixAhead;
      width = J.width;
      M = fix_smem(D, J.dia_T, J.dia_tx, J.dia_ty, width);
      G = width / V;
      R = kFixThreads / G;
      r = threadIdx.x / G;
      g = threadIdx.x - r * G;
      live = r < R;
      col0 = J.col_off + g * V;
      ldy = J.ld;
      noth = J.ndots - (SELF ? 1 : 0);
      if constexpr (NDC == 0)
        for (int d = 0; d < nd; ++d)
          if (D.off[d] == 0) dself = d;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int f = live ? fix_exp(J, col0 + v) : 0;
        K[v] = 1026 + f;
        ex[v] = J.ka - 60 + f;
      }
      // Slots are numbered from 0 again; a barrier's parity goes on.
      pslot = wslot = rslot = 0;
      for (int e = threadIdx.x; e < nr * kMaxDiags; e += kFixThreads) {
        const int rot = e / kMaxDiags, d = e - rot * kMaxDiags;
        const int pos = DIM == 3 ? (D.dy[d] + D.Ay) * (J.dia_tx + 2 * D.Ax) + D.dx[d] + D.Ax : D.cpos[d];
        xo_tab[e] = d < nd ? M.ring + ((rot + A + D.line[d]) % nr) * M.slot + pos * width * 8 : 0;
      }
      __syncthreads();
      produce(issued);
    }
    const int nwin = C.nl + 2 * A, T = J.dia_T, vbytes = round128(T * nd * 8);
    const int wp = fix_win_points(D, T, J.dia_tx, J.dia_ty);
    // What stays the same on every line or plane of the unit: where the
    // thread's points lie in the block (elements from the line's first row of
    // the unit's origin; -1: none), in the windows and among the values, and
    // where the values it loads lie.
    const int line_rows = DIM == 3 ? D.P : D.L;
    const int row0 = C.k0 * line_rows + (DIM == 3 ? C.segT * D.L + C.seg0 : C.seg0);
    int oo[kFixPoints], xb[kFixPoints], ev[kFixValRegs];
#pragma unroll
    for (int q = 0; q < kFixPoints; ++q) {
      const int p = r + q * R;
      const int row = live ? fix_row<DIM>(J, C, C.k0, p) : -1;
      oo[q] = row >= 0 ? (row - row0) * ldy + col0 : -1;
      const int pos = DIM == 3 ? (p >> J.dia_txs) * (J.dia_tx + 2 * D.Ax) + (p & (J.dia_tx - 1)) : p;
      xb[q] = pos * width * 8 + g * 16;
    }
#pragma unroll
    for (int q = 0; q < kFixValRegs; ++q) {
      const int e = threadIdx.x + q * kFixThreads, p = e / nd;
      const int row = e < T * nd ? fix_row<DIM>(J, C, C.k0, p) : -1;
      ev[q] = row >= 0 ? (row - row0) * nd + (e - p * nd) : -1;
    }
    const int2* fx = J.fix + (size_t)row0 * nd;
    // (2D: the last line may be short; n - row0 rows are left at the origin)
    auto load_vals = [&](int j, int2 (&v)[kFixValRegs]) {
      const int2* f = fx + (size_t)j * line_rows * nd;
      const long long left = DIM == 2 ? (long long)(J.n - row0 - j * line_rows) * nd : 1LL << 40;
#pragma unroll
      for (int q = 0; q < kFixValRegs; ++q)
        v[q] = ev[q] >= 0 && ev[q] < left ? __ldg(f + ev[q]) : make_int2(0, 0);
    };
    auto store_vals = [&](int buf, const int2 (&v)[kFixValRegs]) {
#pragma unroll
      for (int q = 0; q < kFixValRegs; ++q) {
        const int e = threadIdx.x + q * kFixThreads;
        if (e < T * nd) *reinterpret_cast<int2*>(smem_raw + M.vals + buf * vbytes + e * 8) = v[q];
      }
    };
    int2 vr[kFixValRegs];
    load_vals(0, vr);
    store_vals(0, vr);
    for (int j = 0; j < C.nl; ++j) {
      // Wait for the windows of line k0 + j and convert the new ones (the
      // others' readers are past the previous line's barrier only for the
      // window that line released, which is none of these).
      const int tw = t0 + j + 2 * A;
      bool ok = true;
      while (ok && wnext <= tw) {
        ok = mbar_wait_bounded(bar0 + 8 * wslot, (phases >> wslot) & 1u, wait_ns);
        if (!ok) break;
        phases ^= 1u << wslot;
        if (live) {
          unsigned char* w = smem_raw + M.ring + wslot * M.slot + g * 16;
#pragma unroll 2
          for (int p = r; p < wp; p += R) {
            int4* c = reinterpret_cast<int4*>(w + p * width * 8);
            const int4 b = *c;
            int4 f;
            to_fixed(b.x, b.y, K[0], f.x, f.y, rmin);
            to_fixed(b.z, b.w, K[1], f.z, f.w, rmin);
            *c = f;
          }
        }
        ++wnext;
        if (++wslot == nr) wslot = 0;
      }
      if (__syncthreads_or(!ok)) {
        for (int t = wnext, sl = wslot; t < issued; ++t) {  // copies still in flight
          mbar_wait_bounded(bar0 + 8 * sl, (phases >> sl) & 1u, wait_ns);
          if (++sl == nr) sl = 0;
        }
        if (threadIdx.x == 0) atomicExch(J.err, 1);
        return;
      }
      produce(t0 + j);  // window t0 + j - 1 was read last on the line before
      const bool more = j + 1 < C.nl;
      if (more) load_vals(j + 1, vr);
      if (live) {
        const int* xt = xo_tab + rslot * kMaxDiags;
        int xo[kDiags];
#pragma unroll
        for (int d = 0; d < kDiags; ++d) xo[d] = xt[d];
        const unsigned char* vb = smem_raw + M.vals + (j & 1) * vbytes;
        const size_t lo = (size_t)(row0 + j * line_rows) * ldy;
        double* yline = J.y + lo;
        // (2D: the short last line, in elements from its first row here)
        const long long left = DIM == 2 ? (long long)(J.n - row0 - j * line_rows) * ldy : 0;
        // x . y of the line's points: |sum xh yh| <= 4 2^60, cross sums below 2^63.
        long long sh[V] = {0, 0}, sc[V] = {0, 0};
#pragma unroll
        for (int q = 0; q < kFixPoints; ++q) {
          if (oo[q] < 0 || (DIM == 2 && oo[q] >= left)) continue;
          double2 u[kEarly && NOTH > 0 ? NOTH : 1];
          if constexpr (kEarly) {
#pragma unroll
            for (int d = 0; d < NOTH; ++d)
              if (d < noth) u[d] = __ldg(reinterpret_cast<const double2*>(J.dotv[d] + lo + oo[q]));
          }
          const unsigned char* xq = smem_raw + xb[q];
          const int2* av = reinterpret_cast<const int2*>(vb + (r + q * R) * nd * 8);
          long long H[V] = {0, 0}, X[V] = {0, 0};
          int4 xc;
#pragma unroll
          for (int d = 0; d < kDiags; ++d) {
            if (NDC > 0 || d < nd) {
              const int2 a = av[d];
              const int4 x = *reinterpret_cast<const int4*>(xq + xo[d]);
              if (NDC > 0 && d == NDC / 2) xc = x;  // (5, 7 and 13 points: symmetric stencils)
              H[0] += (long long)a.x * x.x;
              X[0] += (long long)a.x * x.y;
              X[0] += (long long)a.y * x.x;
              H[1] += (long long)a.x * x.z;
              X[1] += (long long)a.x * x.w;
              X[1] += (long long)a.y * x.z;
              if (NDC == 0 && d == 7) {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                  H[v] += X[v] >> 30;
                  X[v] &= 0x3fffffff;
                }
              }
            }
          }
          if constexpr (SELF && NDC == 0) xc = *reinterpret_cast<const int4*>(xq + xt[dself]);
          double yv[V];
#pragma unroll
          for (int v = 0; v < V; ++v) {
            const long long Y = H[v] + ((X[v] + (1 << 29)) >> 30);
            yv[v] = from_fixed(Y, ex[v]);
            if constexpr (SELF) {
              // Y = yh 2^30 + yl, |yl| <= 2^29 (so the dropped xl yl has mean 0)
              const int yl = (int)((unsigned)Y << 2) >> 2, yh = (int)((Y - yl) >> 30);
              const int xh = v ? xc.z : xc.x, xl = v ? xc.w : xc.y;
              sh[v] += (long long)xh * yh;
              sc[v] += (long long)xh * yl;
              sc[v] += (long long)xl * yh;
            }
          }
          *reinterpret_cast<double2*>(yline + oo[q]) = make_double2(yv[0], yv[1]);
#pragma unroll
          for (int d = 0; d < NOTH; ++d) {
            if (d < noth) {
              const double2 w = kEarly ? u[kEarly ? d : 0]
                                       : __ldg(reinterpret_cast<const double2*>(J.dotv[d] + lo + oo[q]));
              acc_s[d][0] = fma(w.x, yv[0], acc_s[d][0]);
              acc_s[d][1] = fma(w.y, yv[1], acc_s[d][1]);
            }
          }
        }
        if constexpr (SELF) {
#pragma unroll
          for (int v = 0; v < V; ++v) self[v] += ((__int128)sh[v] << 30) + sc[v];
        }
      }
      if (more) store_vals((j + 1) & 1, vr);
      if (++rslot == nr) rslot = 0;
    }
    const int unit = C.gu - B.tile_start[C.jb];
    AccD* red = reinterpret_cast<AccD*>(smem_raw + M.red);
#pragma unroll
    for (int d = 0; d < NOTH; ++d) {
      if (d < noth) {
        const AccD a2[V] = {{acc_s[d][0]}, {acc_s[d][1]}};
        cta_reduce_write<double, AccD>(red, a2, live, G, R, J.col_off, J.width,
                                       J.part + (size_t)d * ldy * J.ntiles, J.ntiles, unit);
      }
      acc_s[d][0] = acc_s[d][1] = 0.0;
    }
    if constexpr (SELF) {
      AccD a2[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int f = ex[v] - (J.ka - 60);  // X = x 2^(60 - f), Y = y 2^-ex
        const double t = fma((double)(long long)(self[v] >> 64), 0x1p64,
                             (double)(unsigned long long)self[v]);
        a2[v].s = ldexp(t, f - 30 + ex[v]);
        self[v] = 0;
      }
      cta_reduce_write<double, AccD>(red, a2, live, G, R, J.col_off, J.width,
                                     J.part + (size_t)noth * ldy * J.ntiles, J.ntiles, unit);
    }
    if (rmin < 4) {
      atomicOr(J.bad, 1);
      rmin = 1 << 20;
    }
    __syncthreads();  // every read of the unit's windows and values is done
    rslot += 2 * A;
    if (rslot >= nr) rslot -= nr;
    t0 += nwin;
    produce(t0);
    fix_unit<DIM, MANY>(C, B, C.gu + gridDim.x, skip);
  }
}

// A 2^(ka - 60), A = a.x 2^30 + a.y, in FP64: leading one, shift and rounding
// in integers, where the conversion and its scaling would take the FP64 pipe as
// long as the entry's two multiply-adds.
__device__ __forceinline__ double fix_entry(int2 a, int ka) {
  const long long A = ((long long)a.x << 30) + a.y;
  if (A == 0) return 0.0;
  const unsigned long long m = A < 0 ? -(unsigned long long)A : (unsigned long long)A;
  const int lz = __clzll((long long)m);
  const unsigned long long f = m << lz;
  const unsigned long long r = (f >> 11) + ((f >> 10) & 1);  // 2^52 <= r <= 2^53
  const long long bits = ((long long)(1025 + ka - lz) << 52) + (long long)r;
  return __longlong_as_double(A < 0 ? bits | (1LL << 63) : bits);
}

// The same product, y and partials with FP64 arithmetic, for jobs whose flag
// is set (x outside its column's range); a read of the flag otherwise.  ND:
// bound of the jobs' dots (their sums stay in registers).  The FP64 pipe
// bounds it like the CSR pass: 64 x 63 x 61 Laplacian with one entry raised by
// 8, 60 probes, 30 steps, all but the first few beyond the range, the SpMM
// passes of a solve 5.9 ms (CSR pass 6.1), window 4 11.7 (12.9); 15.1 and 30.2
// with the dots' sums in local memory, the conversions on the FP64 pipe and the
// fixed-point pass run as well in every step.
template <int ND, int DIM>
__global__ void __launch_bounds__(kFixThreads, ND > 4 ? 2 : ND > 2 ? 3 : 4)
    k_spmm_fix_general(const __grid_constant__ SpmmBatch<double> B) {
  __shared__ AccD red[kFixThreads * 2];
  const unsigned in_range = ~jobs_out_of_range(B);
  if (in_range == ~0u) return;
  FixUnit U;
  for (fix_unit<DIM, true>(U, B, blockIdx.x, &in_range); U.gu < B.total_tiles;
       fix_unit<DIM, true>(U, B, U.gu + gridDim.x, &in_range)) {
    const SpmmJob<double>& J = B.jobs[U.jb];
    const DiaInfo& D = J.dinfo;
    const int nd = D.ndiag, G = J.width / 2, R = kFixThreads / G;
    const int r = threadIdx.x / G, g = threadIdx.x - r * G, col0 = J.col_off + g * 2;
    const bool live = r < R;
    AccD acc[ND > 0 ? ND : 1][2];
#pragma unroll
    for (int d = 0; d < ND; ++d) acc[d][0].zero(), acc[d][1].zero();
    for (int k = U.k0; live && k < U.k0 + U.nl; ++k)
      for (int p = r; p < J.dia_T; p += R) {
        const int row = fix_row<DIM>(J, U, k, p);
        if (row < 0) continue;
        const int2* fa = J.fix + (size_t)row * nd;
        double s0 = 0.0, s1 = 0.0;
        for (int d0 = 0; d0 < nd; d0 += 4) {
          int2 a[4];
          double2 x[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) a[q] = d0 + q < nd ? __ldg(fa + d0 + q) : make_int2(0, 0);
#pragma unroll
          for (int q = 0; q < 4; ++q)  // (no entry: the neighbour may not exist)
            x[q] = a[q].x | a[q].y ? __ldg(reinterpret_cast<const double2*>(
                                         J.x + (size_t)(row + D.off[d0 + q]) * J.ld + col0))
                                   : make_double2(0.0, 0.0);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (d0 + q < nd) {
              const double av = fix_entry(a[q], J.ka);
              s0 = fma(av, x[q].x, s0);
              s1 = fma(av, x[q].y, s1);
            }
        }
        const size_t off = (size_t)row * J.ld + col0;
        *reinterpret_cast<double2*>(J.y + off) = make_double2(s0, s1);
#pragma unroll
        for (int d = 0; d < ND; ++d) {
          if (d < J.ndots) {
            const double2 u = __ldg(reinterpret_cast<const double2*>(J.dotv[d] + off));
            acc[d][0].fma(u.x, s0);
            acc[d][1].fma(u.y, s1);
          }
        }
      }
#pragma unroll
    for (int d = 0; d < ND; ++d)
      if (d < J.ndots)
        cta_reduce_write<double, AccD>(red, acc[d], live, G, R, J.col_off, J.width,
                                       J.part + (size_t)d * J.ld * J.ntiles, J.ntiles,
                                       U.gu - B.tile_start[U.jb]);
    __syncthreads();
  }
}

template <typename Vin>
__global__ void k_fix_values(const int* __restrict__ rowptr, const int* __restrict__ colind,
                             const int* __restrict__ slot, const Vin* __restrict__ vals, int n, int nd,
                             double c, double shift, int k, int2* __restrict__ out) {
  const double up = ldexp(1.0, k);
  for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < n; row += gridDim.x * blockDim.x)
    for (int q = rowptr[row]; q < rowptr[row + 1]; ++q) {
      long long a = __double2ll_rn((double)vals[q] / c * up);
      if (colind[q] == row) a += __double2ll_rn(shift / c * up);
      const long long hi = (a + (1 << 29)) >> 30;
      out[(size_t)row * nd + slot[q]] = make_int2((int)hi, (int)(a - (hi << 30)));
    }
}

}  // namespace

bool fix_geom(const logdet_ctx* h, int width, int ld, FixGeom* out) {
  const DiaInfo& d = h->dia;
  if (h->kind != 0 || d.ndiag == 0 || !h->dia_slot || width % 2 || width < 2 || width > kFixMaxWidth ||
      2 * d.A + 1 + kFixAhead > kFixMaxWindows || (d.dim == 3 && (long long)d.P * ld >= (1LL << 30)))
    return false;
  const int R = kFixThreads / (width / 2);
  FixGeom g;
  memset(&g, 0, sizeof g);
  auto fits = [&](int T, int tx, int ty) {
    return T <= kFixPoints * R && T * d.ndiag <= kFixValRegs * kFixThreads && fix_smem(d, T, tx, ty, width).total <= kFixSmem;
  };
  if (d.dim == 3) {
    // The tile with the fewest converted points per result that fits.
    double best = 1e30;
    for (int txs = 5; txs >= 2; --txs) {
      const int tx = 1 << txs;
      if (tx > 4 && tx / 2 >= d.L) continue;
      for (int ty = 1; ty <= 32 && ty <= d.ny; ++ty) {
        const int T = tx * ty;
        if (T < R || tx + 2 * d.Ax > 256 || ty + 2 * d.Ay > 256 || !fits(T, tx, ty)) continue;
        const double over = (double)((d.L + tx - 1) / tx * tx) / d.L *
                            ((double)((d.ny + ty - 1) / ty * ty) / d.ny) *
                            ((double)((T + R - 1) / R * R) / T);
        const double cost = ((double)(tx + 2 * d.Ax) * (ty + 2 * d.Ay) / T + 2.0) * over;
        if (cost < best) {
          best = cost;
          g.T = T;
          g.tx = tx;
          g.ty = ty;
          g.txs = txs;
        }
      }
    }
    if (g.T == 0) return false;
    g.nseg = (d.L + g.tx - 1) / g.tx * ((d.ny + g.ty - 1) / g.ty);
    g.nlines = d.nz;
  } else {
    for (int t = R; t + d.cw <= 256 && (t == R || t - R < d.L) && fits(t, 0, 0); t += R) g.T = t;
    if (g.T == 0) return false;
    g.nseg = (d.L + g.T - 1) / g.T;
    g.nlines = (h->n + d.L - 1) / d.L;
  }
  const int chunks = std::max(1, 8 * sm_count() / g.nseg);
  g.kc = (g.nlines + chunks - 1) / chunks;
  g.kc = std::min(g.nlines, std::max(g.kc, 8 * d.A));
  g.units = g.nseg * ((g.nlines + g.kc - 1) / g.kc);
  *out = g;
  return true;
}

int fix_scale(const logdet_ctx* h, double c, double shift) {
  // |Q|_inf <= max(d + r, r - d) over the rows, the Gershgorin ends.
  const double b = (std::max(h->g_hi, -h->g_lo) + shift) / c;
  return std::ilogb(b) + 1;
}

int fix_values(const logdet_ctx* h, double c, double shift, int ka, int2* out, cudaStream_t st) {
  const int n = h->n, nd = h->dia.ndiag;
  LD_CUDA(cudaMemsetAsync(out, 0, sizeof(int2) * (size_t)nd * n, st));
  ProfScope prof(KC_OTHER, st);
  const int blocks = std::max(1, std::min(div_up(n, 256), 8 * sm_count()));
  if (h->vals_dtype == LOGDET_VALS_F64)
    k_fix_values<double><<<blocks, 256, 0, st>>>(h->rowptr, h->colind, h->dia_slot,
                                                 (const double*)h->vals, n, nd, c, shift, 60 - ka, out);
  else
    k_fix_values<float><<<blocks, 256, 0, st>>>(h->rowptr, h->colind, h->dia_slot,
                                                (const float*)h->vals, n, nd, c, shift, 60 - ka, out);
  LD_CHECK_LAUNCH();
  return LOGDET_OK;
}

int fix_job(SpmmJob<double>& J, const logdet_ctx* h, const FixGeom& g, const int2* fix, int ka,
            int* err, int* bad) {
  const DiaInfo& d = h->dia;
  J.dinfo = d;
  J.fix = fix;
  J.ka = ka;
  J.hn = std::ilogb((double)J.n) / 2;
  J.err = err;
  J.bad = bad;
  J.dia_T = g.T;
  J.dia_kc = g.kc;
  J.dia_nseg = g.nseg;
  J.dia_nlines = g.nlines;
  J.dia_tx = g.tx;
  J.dia_ty = g.ty;
  J.dia_txs = g.txs;
  J.ntiles = g.units;
  LD_TRY(tma_encode_ready());
  // TMA over 4-byte words: 16-byte bases, pitches and innermost coordinates.
  if (((uintptr_t)J.x & 15) || J.ld % 2 || J.width % 2 || J.col_off % 2 || J.width > kFixMaxWidth) {
    set_error("fixed-point sweep: block not aligned for TMA");
    return LOGDET_EINVAL;
  }
  const float* x = reinterpret_cast<const float*>(J.x);
  if (d.dim == 3)
    return tma_encode_grid(&J.tmap, x, d, 2 * J.ld, 2 * J.ld, 2 * J.width, g.tx + 2 * d.Ax,
                           g.ty + 2 * d.Ay);
  return tma_encode_2d(&J.tmap, x, 2 * J.ld, J.n, 2 * J.ld, 2 * J.width, g.T + d.cw);
}

int launch_spmm_fix(const SpmmBatch<double>& b, cudaStream_t s) {
  int nd = 0, smem = 0;
  double flops = 0.0, bytes = 0.0;
  int ndc = b.jobs[0].dinfo.ndiag;
  const int dim = b.jobs[0].dinfo.dim;
  for (int j = 0; j < b.njobs; ++j) {
    const SpmmJob<double>& J = b.jobs[j];
    nd = std::max(nd, J.ndots);
    if (J.dinfo.ndiag != ndc) ndc = 0;
    if (J.ndots > 0 && J.dotv[J.ndots - 1] != J.x) {
      set_error("fixed-point sweep: the last dot vector must be x");
      return LOGDET_EINVAL;
    }
    smem = std::max(smem, fix_smem(J.dinfo, J.dia_T, J.dia_tx, J.dia_ty, J.width).total);
    const double vb = (double)J.n * J.b * 8;
    const int extra_reads = J.ndots - ((J.ndots > 0 && J.dotv[0] == J.x) ? 1 : 0);
    flops += 2.0 * (double)J.nnz * J.b + 2.0 * (double)J.n * J.b * J.ndots;
    bytes += (double)J.nnz * 8 + vb * (2 + extra_reads);
  }
  if (dim == 3 ? ndc != 7 : (ndc != 5 && ndc != 13)) ndc = 0;
  for (int j = 0; j < b.njobs; ++j)  // (compiled counts: the middle entry is the diagonal)
    if (ndc && b.jobs[j].dinfo.off[ndc / 2] != 0) ndc = 0;
  // Test hook: see launch_spmm_dia; "sketch" stalls the products without dots
  // alone (the sketch's).
  const char* stall_env = getenv("LOGDET_TEST_SWEEP_STALL");
  const bool stall = stall_env && (stall_env[0] == '1' || (nd == 0 && !strcmp(stall_env, "sketch")));
  const unsigned extra_tx = stall ? 16u : 0u;
  const unsigned long long wait_ns = stall ? 20000000ull : kDiaWaitNs;
  const int grid = std::max(1, std::min(b.total_tiles, 2 * sm_count()));
  ProfScope prof(KC_SPMM, s, flops, bytes);  // (one pass: both launches)
#define LD_FIX_KERN(NO, SELF, NC, DM) \
  (b.njobs > 1 ? k_spmm_fix<NO, SELF, NC, DM, true> : k_spmm_fix<NO, SELF, NC, DM, false>)
#define LD_FIX_CASE(NO, SELF)                                                                  \
  {                                                                                            \
    auto kern = dim == 3 ? (ndc == 7 ? LD_FIX_KERN(NO, SELF, 7, 3) : LD_FIX_KERN(NO, SELF, 0, 3)) \
                         : ndc == 13 ? LD_FIX_KERN(NO, SELF, 13, 2)                            \
                         : ndc == 5  ? LD_FIX_KERN(NO, SELF, 5, 2)                             \
                                     : LD_FIX_KERN(NO, SELF, 0, 2);                            \
    LD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kFixSmem)); \
    kern<<<grid, kFixThreads, smem, s>>>(b, extra_tx, wait_ns);                                \
    break;                                                                                     \
  }
  do {
    if (nd == 0) LD_FIX_CASE(0, false)
    if (nd == 1) LD_FIX_CASE(0, true)
    if (nd == 2) LD_FIX_CASE(1, true)
    if (nd <= 4) LD_FIX_CASE(3, true)
    LD_FIX_CASE(kMaxWin - 1, true)
  } while (0);
#undef LD_FIX_CASE
#undef LD_FIX_KERN
  LD_CHECK_LAUNCH();
  // Four CTAs per SM: the FP64 pipe is full from two.
  const int ggrid = std::max(1, std::min(b.total_tiles, 4 * sm_count()));
  prof_count();
#define LD_FIX_GENERAL(ND)                                                       \
  {                                                                              \
    if (dim == 3) k_spmm_fix_general<ND, 3><<<ggrid, kFixThreads, 0, s>>>(b);    \
    else k_spmm_fix_general<ND, 2><<<ggrid, kFixThreads, 0, s>>>(b);             \
    break;                                                                       \
  }
  do {
    if (nd == 0) LD_FIX_GENERAL(0)
    if (nd == 1) LD_FIX_GENERAL(1)
    if (nd == 2) LD_FIX_GENERAL(2)
    if (nd <= 4) LD_FIX_GENERAL(4)
    LD_FIX_GENERAL(kMaxWin)
  } while (0);
#undef LD_FIX_GENERAL
  LD_CHECK_LAUNCH();
  return LOGDET_OK;
}

int fix_spmm_block(const logdet_ctx* h, const int2* fix, int ka, const double* x, double* y, int ld,
                   int xexp, int* err_host, cudaStream_t st) {
  DevBuf<int> flags(st);
  LD_TRY(flags.alloc(2));
  LD_TRY(flags.zero());
  FixGeom g;
  if (!fix_geom(h, ld, ld, &g)) {
    set_error("fixed-point sweep: block of %d columns does not fit", ld);
    return LOGDET_EINVAL;
  }
  SpmmBatch<double> B;
  memset(&B, 0, sizeof B);
  B.njobs = 1;
  SpmmJob<double>& J = B.jobs[0];
  J.x = x;
  J.y = y;
  J.n = h->n;
  J.ld = J.width = J.b = ld;
  J.nnz = h->nnz;
  J.xexp = xexp;
  LD_TRY(fix_job(J, h, g, fix, ka, flags.p, flags.p + 1));
  B.tile_start[1] = B.total_tiles = J.ntiles;
  LD_TRY(launch_spmm_fix(B, st));
  LD_CUDA(cudaMemcpyAsync(err_host, flags.p, sizeof(int), cudaMemcpyDeviceToHost, st));
  return LOGDET_OK;
}

}  // namespace ld
