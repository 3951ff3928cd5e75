// Fast convolution for the matrix-free gridded operators (see grid.cuh): y =
// Q x by 2D Fourier transforms, for supports whose (2 R + 1)^2 taps cost more
// than the transforms do.
//
// The grid is covered by tx x ty windows of Nx x Ny points (powers of two;
// overlap-save, or one zero-padded window along an axis where n + R <= N).
// The stencil is even in both offsets, so its symbol (the DFT of the table)
// is real, and one complex transform convolves two real fields at once: one
// window is the real part, the next window of the same block column the
// imaginary part.  Both come from one column, so their magnitudes are alike
// and neither loses accuracy to the other.
//
//   k_fft_rows   transforms along x of each window row, into the workspace
//   k_fft_cols   transforms along y, times the symbol, and back
//   k_fft_back   inverse transforms along x, valid points into y (+ shift)
//
// Transforms run in registers (8 or 16 points per thread) with two or three
// passes exchanged through shared memory; forward transforms leave their
// output in digit-permuted order, the symbol is stored in that order and the
// inverse takes it back, so nothing is ever reordered.
//
// Against the direct convolution, which the FMA pipes bound (48 % of the FP32
// peak, 40 % of the FP64 one): Wendland support 50 on 1200 x 900, 16 FP32
// columns 6.6 -> 0.24 ms an application (17.6 us rows, 33 us columns, 22 us
// back per four columns: 2 TB/s through L2, the exchanges and twiddles issue
// more than they move); support 20 on 301 x 240, 20 FP64 columns 6.3 -> 0.38
// ms, bound by the FP64 pipe (about 130 operations a point and column).
#include "grid.cuh"
#include "profile.cuh"

#include <cmath>

namespace ld {

namespace {

template <typename CT> struct CplxOf;
template <> struct CplxOf<float> { using type = float2; };
template <> struct CplxOf<double> { using type = double2; };

// Radices of a transform of 2^LN points: R1 R2 R3 = N, E = R1 points a thread.
template <int LN> struct Shape;
template <> struct Shape<6> { static constexpr int R1 = 8, R2 = 8, R3 = 1; };
template <> struct Shape<7> { static constexpr int R1 = 16, R2 = 8, R3 = 1; };
template <> struct Shape<8> { static constexpr int R1 = 16, R2 = 16, R3 = 1; };
template <> struct Shape<9> { static constexpr int R1 = 8, R2 = 8, R3 = 8; };
template <> struct Shape<10> { static constexpr int R1 = 16, R2 = 8, R3 = 8; };
template <> struct Shape<11> { static constexpr int R1 = 16, R2 = 16, R3 = 8; };

// Frequency of slot s of a transform of 2^ln points: s = (k1 R2 + k2) R3 + k3
// holds frequency k1 + R1 (k2 + R2 k3).
__host__ __device__ __forceinline__ int slot_freq(int ln, int s) {
  const int b1 = (ln == 6 || ln == 9) ? 3 : 4;
  const int b2 = (ln == 8 || ln == 11) ? 4 : 3;
  const int b3 = ln - b1 - b2;
  const int k3 = s & ((1 << b3) - 1), k2 = (s >> b3) & ((1 << b2) - 1), k1 = s >> (b2 + b3);
  return k1 + (k2 << b1) + (k3 << (b1 + b2));
}

template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return {a.x + b.x, a.y + b.y}; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return {a.x - b.x, a.y - b.y}; }
template <bool INV, typename C> __device__ __forceinline__ C cmul(C a, C w) {  // a w, or a conj(w)
  if constexpr (INV) return {fma(a.y, w.y, a.x * w.x), fma(-a.x, w.y, a.y * w.x)};
  else return {fma(-a.y, w.y, a.x * w.x), fma(a.x, w.y, a.y * w.x)};
}
template <bool INV, typename C> __device__ __forceinline__ C mul_mi(C a) {  // -i a, or i a
  if constexpr (INV) return {-a.y, a.x};
  else return {a.y, -a.x};
}

// DFT of R points in registers, natural order, by halving (Cooley and Tukey
// 1965): even and odd points, twiddles exp(-+ 2 pi i k / R).
template <int R, bool INV, typename C>
__device__ __forceinline__ void dft(C (&v)[R]) {
  if constexpr (R == 2) {
    const C a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
  } else if constexpr (R > 2) {
    using CT = decltype(v[0].x);
    C e[R / 2], o[R / 2];
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      e[k] = v[2 * k];
      o[k] = v[2 * k + 1];
    }
    dft<R / 2, INV>(e);
    dft<R / 2, INV>(o);
    constexpr double kC[8] = {1.0, 0.92387953251128675613, 0.70710678118654752440,
                              0.38268343236508977173, 0.0, -0.38268343236508977173,
                              -0.70710678118654752440, -0.92387953251128675613};
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      constexpr int step = 16 / R;
      C w;
      if (k == 0) w = o[k];
      else if (2 * k == R / 2) w = mul_mi<INV>(o[k]);
      else if (4 * k == R / 2 || 4 * k == 3 * (R / 2)) {  // +-sqrt(1/2) -+ i sqrt(1/2)
        const CT h = (CT)kC[2];
        const C r = mul_mi<INV>(o[k]);
        w = 4 * k == R / 2 ? C{(o[k].x + r.x) * h, (o[k].y + r.y) * h}
                           : C{(r.x - o[k].x) * h, (r.y - o[k].y) * h};
      } else {
        const int q = k * step;  // angle 2 pi q / 16, 0 < q < 8
        const C t = {(CT)kC[q], (CT)(q <= 4 ? -kC[4 - q] : -kC[q - 4])};
        w = cmul<INV>(o[k], t);
      }
      v[k] = cadd(e[k], w);
      v[k + R / 2] = csub(e[k], w);
    }
  }
}

// Slot idx of line c among C interleaved lines; one slot in nine is skipped
// so that threads eight slots apart fall on different banks.
__device__ __forceinline__ int at(int idx, int C, int c) { return (idx + (idx >> 3)) * C + c; }

template <int LN>
struct Fft {
  static constexpr int N = 1 << LN, R1 = Shape<LN>::R1, R2 = Shape<LN>::R2, R3 = Shape<LN>::R3;
  static constexpr int E = R1, TL = N / E;                // points a thread, threads a line
  static constexpr int L1 = N / R1, L2 = L1 / R2;         // lengths left after passes 1 and 2
  static constexpr int RL = R3 > 1 ? R3 : R2;             // the last pass's radix
  static constexpr size_t slots = N + N / 8;

  // The slot of register q after forward().
  __device__ __forceinline__ static int slot(int t, int q) { return (t + TL * (q / RL)) * RL + q % RL; }

  // v[j] = point t + TL j on entry; v[q] = slot(t, q) on return.  tw: roots
  // exp(-2 pi i k / (N tws)).
  template <typename C>
  __device__ __forceinline__ static void forward(C (&v)[E], C* sm, int t, int c, int nl,
                                                 const C* __restrict__ tw, int tws) {
    dft<R1, false>(v);
#pragma unroll
    for (int k = 0; k < R1; ++k) {
      if (k) v[k] = cmul<false>(v[k], __ldg(tw + t * k * tws));
      sm[at(k * TL + t, nl, c)] = v[k];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < E / R2; ++i) {
      const int bi = t + TL * i, sub = bi / L2, pos = bi % L2;
      C u[R2];
#pragma unroll
      for (int j = 0; j < R2; ++j) u[j] = sm[at(sub * L1 + pos + L2 * j, nl, c)];
      dft<R2, false>(u);
#pragma unroll
      for (int k = 0; k < R2; ++k) {
        if constexpr (R3 > 1) {
          if (k) u[k] = cmul<false>(u[k], __ldg(tw + pos * k * R1 * tws));
          sm[at(sub * L1 + pos + L2 * k, nl, c)] = u[k];
        } else {
          v[i * R2 + k] = u[k];
        }
      }
    }
    if constexpr (R3 > 1) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < E / R3; ++i) {
        C u[R3];
#pragma unroll
        for (int j = 0; j < R3; ++j) u[j] = sm[at((t + TL * i) * R3 + j, nl, c)];
        dft<R3, false>(u);
#pragma unroll
        for (int k = 0; k < R3; ++k) v[i * R3 + k] = u[k];
      }
    }
  }

  // The unscaled inverse: slots in, points t + TL j out.  Every pass writes
  // the slots it has read, so one barrier separates two passes.
  template <typename C>
  __device__ __forceinline__ static void inverse(C (&v)[E], C* sm, int t, int c, int nl,
                                                 const C* __restrict__ tw, int tws) {
    if constexpr (R3 > 1) {
#pragma unroll
      for (int i = 0; i < E / R3; ++i) {
        C u[R3];
#pragma unroll
        for (int k = 0; k < R3; ++k) u[k] = v[i * R3 + k];
        dft<R3, true>(u);
#pragma unroll
        for (int j = 0; j < R3; ++j) sm[at((t + TL * i) * R3 + j, nl, c)] = u[j];
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < E / R2; ++i) {
      const int bi = t + TL * i, sub = bi / L2, pos = bi % L2;
      C u[R2];
#pragma unroll
      for (int k = 0; k < R2; ++k) {
        if constexpr (R3 > 1) {
          u[k] = sm[at(sub * L1 + pos + L2 * k, nl, c)];
          if (k) u[k] = cmul<true>(u[k], __ldg(tw + pos * k * R1 * tws));
        } else {
          u[k] = v[i * R2 + k];
        }
      }
      dft<R2, true>(u);
#pragma unroll
      for (int j = 0; j < R2; ++j) sm[at(sub * L1 + pos + L2 * j, nl, c)] = u[j];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < R1; ++k) {
      v[k] = sm[at(k * TL + t, nl, c)];
      if (k) v[k] = cmul<true>(v[k], __ldg(tw + t * k * tws));
    }
    dft<R1, true>(v);
  }
};

// One launch's arguments.  A unit is a vector chunk of V block columns of one
// pair of windows; units u0, u0 + 1, ... of the launch own consecutive
// Nx x Ny x V complex pieces of the workspace, [y][slot of x][column].
template <typename T>
struct FftArgs {
  GridFft p;
  int nx, ny, ld, u0;
  const T* x;
  T* y;
  const double* colshift;
  typename CplxOf<T>::type* ws;
  const typename CplxOf<T>::type* tw;  // exp(-2 pi i k / max(Nx, Ny))
  const T* sym;                        // [Nx / 2 + 1][slot of y], divided by Nx Ny
};

struct Window {  // one window of the cover, and the points of it that are results
  int x0, y0, vx0, vx1, vy0, vy1;
};
__device__ __forceinline__ Window window_of(const GridFft& p, int tile, int nx, int ny) {
  Window w;
  if (tile >= p.tx * p.ty) return {0, ny, 0, 0, 0, 0};  // no such window: rows past the grid
  const int ix = tile % p.tx, iy = tile / p.tx;
  w.x0 = ix * p.bx - p.hx;
  w.y0 = iy * p.by - p.hy;
  w.vx0 = p.hx;
  w.vx1 = min(p.hx + p.bx, nx - w.x0);
  w.vy0 = p.hy;
  w.vy1 = min(p.hy + p.by, ny - w.y0);
  return w;
}
__device__ __forceinline__ bool row_in(const Window& w, int yy, int ny) {
  return w.y0 + yy >= 0 && w.y0 + yy < ny;
}
__device__ __forceinline__ bool row_out(const Window& w, int yy) { return yy >= w.vy0 && yy < w.vy1; }

// Lines a CTA of the row kernels takes (columns of a chunk x rows), and lines
// of the column kernel: at least 256 threads, 64-byte runs in k_fft_cols.
template <typename T, int LN> constexpr int row_lines() {
  constexpr int want = 256 / Fft<LN>::TL;
  return want > Vec16<T>::N ? want : Vec16<T>::N;
}
template <typename T, int LN> constexpr int col_lines() {
  constexpr int want = 256 / Fft<LN>::TL, run = 64 / (2 * (int)sizeof(T));
  return want > run ? want : run;
}

template <typename T, int LN>
__global__ void __launch_bounds__(Fft<LN>::TL* row_lines<T, LN>()) k_fft_rows(const FftArgs<T> A) {
  using F = Fft<LN>;
  using C = typename CplxOf<T>::type;
  constexpr int V = Vec16<T>::N, NL = row_lines<T, LN>(), RP = NL / V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sm = reinterpret_cast<C*>(smem_raw);
  const int c = threadIdx.x % NL, t = threadIdx.x / NL, v = c % V;
  const int unit = A.u0 + blockIdx.y, pair = unit % A.p.pairs, col = unit / A.p.pairs * V + v;
  const int Ny = 1 << A.p.lny, yy0 = blockIdx.x * RP, yy = yy0 + c / V;
  const Window a = window_of(A.p, 2 * pair, A.nx, A.ny), b = window_of(A.p, 2 * pair + 1, A.nx, A.ny);
  bool any = false;  // (the same for the whole CTA)
  for (int r = 0; r < RP; ++r) any = any || row_in(a, yy0 + r, A.ny) || row_in(b, yy0 + r, A.ny);
  if (!any) return;
  const bool ia = row_in(a, yy, A.ny), ib = row_in(b, yy, A.ny);
  C r[F::E];
#pragma unroll
  for (int j = 0; j < F::E; ++j) {
    const int xx = t + F::TL * j;
    const int ga = a.x0 + xx, gb = b.x0 + xx;
    r[j].x = ia && ga >= 0 && ga < A.nx ? __ldg(A.x + ((size_t)(a.y0 + yy) * A.nx + ga) * A.ld + col) : T(0);
    r[j].y = ib && gb >= 0 && gb < A.nx ? __ldg(A.x + ((size_t)(b.y0 + yy) * A.nx + gb) * A.ld + col) : T(0);
  }
  F::forward(r, sm, t, c, NL, A.tw, 1 << (A.p.lnt - LN));
  if (!ia && !ib) return;
  C* out = A.ws + ((size_t)blockIdx.y * Ny + yy) * ((size_t)F::N * V) + v;
#pragma unroll
  for (int q = 0; q < F::E; ++q) out[F::slot(t, q) * V] = r[q];
}

template <typename T, int LN>
__global__ void __launch_bounds__(Fft<LN>::TL* col_lines<T, LN>(),
                                  Fft<LN>::TL* col_lines<T, LN>() * (int)sizeof(T) > 2048 ? 1 : 2)
    k_fft_cols(const FftArgs<T> A) {
  using F = Fft<LN>;
  using C = typename CplxOf<T>::type;
  constexpr int V = Vec16<T>::N, NL = col_lines<T, LN>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sm = reinterpret_cast<C*>(smem_raw);
  const int c = threadIdx.x % NL, t = threadIdx.x / NL;
  const int pair = (A.u0 + blockIdx.y) % A.p.pairs;
  const int Nx = 1 << A.p.lnx, ci = blockIdx.x * NL + c;
  const Window a = window_of(A.p, 2 * pair, A.nx, A.ny), b = window_of(A.p, 2 * pair + 1, A.nx, A.ny);
  C* line = A.ws + (size_t)blockIdx.y * F::N * ((size_t)Nx * V) + ci;
  const size_t pitch = (size_t)Nx * V;
  const int tws = 1 << (A.p.lnt - LN);
  C r[F::E];
#pragma unroll
  for (int j = 0; j < F::E; ++j) {
    const int yy = t + F::TL * j;
    r[j] = row_in(a, yy, A.ny) || row_in(b, yy, A.ny) ? line[yy * pitch] : C{T(0), T(0)};
  }
  F::forward(r, sm, t, c, NL, A.tw, tws);
  const int kx = slot_freq(A.p.lnx, ci / V);
  const T* sym = A.sym + (size_t)min(kx, Nx - kx) * F::N;
#pragma unroll
  for (int q = 0; q < F::E; ++q) {
    const T s = __ldg(sym + F::slot(t, q));
    r[q].x *= s;
    r[q].y *= s;
  }
  // The inverse works out its addresses and roots anew: carried over from the
  // forward transform they cost the 1024-point FP64 instance 255 registers
  // and the 2048-point one a 1.9 KB spill.
  int ti = t;
  const C* tw = A.tw;
  asm volatile("" : "+r"(ti), "+l"(tw), "+l"(line));
  F::inverse(r, sm, ti, c, NL, tw, tws);
#pragma unroll
  for (int j = 0; j < F::E; ++j) {
    const int yy = ti + F::TL * j;
    if (row_out(a, yy) || row_out(b, yy)) line[yy * pitch] = r[j];
  }
}

template <typename T, int LN>
__global__ void __launch_bounds__(Fft<LN>::TL* row_lines<T, LN>()) k_fft_back(const FftArgs<T> A) {
  using F = Fft<LN>;
  using C = typename CplxOf<T>::type;
  constexpr int V = Vec16<T>::N, NL = row_lines<T, LN>(), RP = NL / V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sm = reinterpret_cast<C*>(smem_raw);
  const int c = threadIdx.x % NL, t = threadIdx.x / NL, v = c % V;
  const int unit = A.u0 + blockIdx.y, pair = unit % A.p.pairs, col = unit / A.p.pairs * V + v;
  const int Ny = 1 << A.p.lny, yy0 = blockIdx.x * RP, yy = yy0 + c / V;
  const Window a = window_of(A.p, 2 * pair, A.nx, A.ny), b = window_of(A.p, 2 * pair + 1, A.nx, A.ny);
  bool any = false;  // (the same for the whole CTA)
  for (int r = 0; r < RP; ++r) any = any || row_out(a, yy0 + r) || row_out(b, yy0 + r);
  if (!any) return;
  const bool oa = row_out(a, yy), ob = row_out(b, yy);
  const C* in = A.ws + ((size_t)blockIdx.y * Ny + yy) * ((size_t)F::N * V) + v;
  C r[F::E];
#pragma unroll
  for (int q = 0; q < F::E; ++q)
    r[q] = oa || ob ? in[F::slot(t, q) * V] : C{T(0), T(0)};
  F::inverse(r, sm, t, c, NL, A.tw, 1 << (A.p.lnt - LN));
  const T sh = A.colshift ? T(A.colshift[col]) : T(0);
#pragma unroll
  for (int j = 0; j < F::E; ++j) {
    const int xx = t + F::TL * j;
    if (oa && xx >= a.vx0 && xx < a.vx1) {
      const size_t o = ((size_t)(a.y0 + yy) * A.nx + a.x0 + xx) * A.ld + col;
      A.y[o] = A.colshift ? fma(sh, __ldg(A.x + o), r[j].x) : r[j].x;
    }
    if (ob && xx >= b.vx0 && xx < b.vx1) {
      const size_t o = ((size_t)(b.y0 + yy) * A.nx + b.x0 + xx) * A.ld + col;
      A.y[o] = A.colshift ? fma(sh, __ldg(A.x + o), r[j].y) : r[j].y;
    }
  }
}

// ---------------------------------------------------------------------------
// Tables of one solve: the roots of unity, and the symbol of W / c.  The
// quadrant table's evenness makes both DFTs cosine sums: A[dy][kx] over dx,
// then sym[kx][ky] over dy, in FP64, for kx <= Nx / 2 and ky in slot order.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_fft_roots(int n, double2* __restrict__ tw64, typename CplxOf<T>::type* __restrict__ tw) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    double s, co;
    sincospi(-2.0 * k / n, &s, &co);
    tw64[k] = {co, s};
    tw[k] = {(T)co, (T)s};
  }
}

__global__ void k_fft_sym_x(const double* __restrict__ tab, int R, int row_len, double c, int lnx,
                            int lnt, const double2* __restrict__ tw, double* __restrict__ out) {
  const int half = (1 << lnx) / 2 + 1, mask = (1 << lnx) - 1, dy = blockIdx.y;
  const int kx = blockIdx.x * blockDim.x + threadIdx.x;
  if (kx >= half) return;
  const double* w = tab + (size_t)dy * row_len + R;
  double s = w[0] / c;
  for (int dx = 1; dx <= R; ++dx)
    s = fma(2.0 * (w[dx] / c), tw[((dx * kx) & mask) << (lnt - lnx)].x, s);
  out[(size_t)dy * half + kx] = s;
}

template <typename T>
__global__ void k_fft_sym_y(const double* __restrict__ a, int R, int lnx, int lny, int lnt,
                            const double2* __restrict__ tw, T* __restrict__ sym) {
  const int half = (1 << lnx) / 2 + 1, Ny = 1 << lny;
  const int slot = blockIdx.x * blockDim.x + threadIdx.x, kx = blockIdx.y;
  if (slot >= Ny) return;
  const int ky = slot_freq(lny, slot);
  double s = a[kx];
  for (int dy = 1; dy <= R; ++dy)
    s = fma(2.0 * a[(size_t)dy * half + kx], tw[((dy * ky) & (Ny - 1)) << (lnt - lny)].x, s);
  sym[(size_t)kx * Ny + slot] = (T)(s / ((double)(1 << lnx) * Ny));
}

template <typename T, int LN, int KIND>
int launch_one(const FftArgs<T>& A, int units, cudaStream_t st) {
  using C = typename CplxOf<T>::type;
  constexpr int NL = KIND == 1 ? col_lines<T, LN>() : row_lines<T, LN>();
  constexpr size_t smem = Fft<LN>::slots * NL * sizeof(C);
  auto fn = KIND == 0 ? k_fft_rows<T, LN> : KIND == 1 ? k_fft_cols<T, LN> : k_fft_back<T, LN>;
  if constexpr (smem > 48 * 1024)
    LD_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  constexpr int V = Vec16<T>::N;
  const int gx = KIND == 1 ? ((1 << A.p.lnx) * V) / NL : div_up(1 << A.p.lny, NL / V);
  fn<<<dim3(gx, units), Fft<LN>::TL * NL, smem, st>>>(A);
  LD_CHECK_LAUNCH();
  return LOGDET_OK;
}

template <typename T, int KIND>
int launch_fft(const FftArgs<T>& A, int units, cudaStream_t st) {
  switch (KIND == 1 ? A.p.lny : A.p.lnx) {
    case 6: return launch_one<T, 6, KIND>(A, units, st);
    case 7: return launch_one<T, 7, KIND>(A, units, st);
    case 8: return launch_one<T, 8, KIND>(A, units, st);
    case 9: return launch_one<T, 9, KIND>(A, units, st);
    case 10: return launch_one<T, 10, KIND>(A, units, st);
    case 11: return launch_one<T, 11, KIND>(A, units, st);
  }
  set_error("grid operator: transform length 2^%d", KIND == 1 ? A.p.lny : A.p.lnx);
  return LOGDET_EINVAL;
}

}  // namespace

// Windows along an axis of n points for transforms of N: one zero-padded
// window where it fits (a circular wrap then only meets zeros), else
// overlap-save windows whose outer R points are discarded on both sides.
static bool axis_cover(int n, int R, int N, int* tiles, int* b, int* halo) {
  if (n + R <= N) {
    *tiles = 1;
    *b = n;
    *halo = 0;
    return true;
  }
  if (N - 2 * R < 16) return false;
  *b = N - 2 * R;
  *halo = R;
  *tiles = div_up(n, *b);
  return true;
}

template <typename T>
GridFft grid_fft_plan(const logdet_ctx* h, int ld) {
  GridFft best;
  double best_cost = 0.0;
  const size_t unit_cap = std::max((size_t)h->n * ld * sizeof(T), kGridFftFree);
  for (int lx = 6; lx <= 11; ++lx)
    for (int ly = 6; ly <= 11; ++ly) {
      GridFft p;
      p.lnx = lx;
      p.lny = ly;
      p.lnt = std::max(lx, ly);
      if (!axis_cover(h->gx, h->gr, 1 << lx, &p.tx, &p.bx, &p.hx) ||
          !axis_cover(h->gy, h->gr, 1 << ly, &p.ty, &p.by, &p.hy))
        continue;
      const long long tiles = (long long)p.tx * p.ty;
      if (tiles > (1 << 20)) continue;
      p.pairs = (int)((tiles + 1) / 2);
      if (lx + ly > 20 || grid_fft_unit_bytes<T>(p) > unit_cap) continue;
      const double cost = (double)p.pairs * std::ldexp(1.0, lx + ly) * (lx + ly);
      if (best.pairs == 0 || cost < best_cost) {
        best = p;
        best_cost = cost;
      }
    }
  if (best.pairs == 0) return best;
  constexpr GridCost g = grid_cost<T>();
  const double taps = (double)h->nnz / h->n;
  const double direct =
      g.start + std::max(g.tap * taps, (double)h->n * ld * (taps + g.stage) / g.taps_per_us);
  if (direct < kGridFftMargin * (g.start + best_cost * ld * g.unit)) best.pairs = 0;
  return best;
}
template GridFft grid_fft_plan<float>(const logdet_ctx*, int);
template GridFft grid_fft_plan<double>(const logdet_ctx*, int);

// Roots (complex), then the symbol.
template <typename T>
size_t grid_fft_table_count(const GridFft& p) {
  return ((size_t)2 << p.lnt) + (((size_t)1 << p.lnx) / 2 + 1) * ((size_t)1 << p.lny);
}
template size_t grid_fft_table_count<float>(const GridFft&);
template size_t grid_fft_table_count<double>(const GridFft&);

template <typename T>
int grid_fft_table(const logdet_ctx* h, const GridFft& p, double c, T* out, cudaStream_t st) {
  using C = typename CplxOf<T>::type;
  const int half = (1 << p.lnx) / 2 + 1, R = h->gr, nt = 1 << p.lnt;
  DevBuf<double2> tw(st);
  DevBuf<double> a(st);
  LD_TRY(tw.alloc(nt));
  LD_TRY(a.alloc((size_t)(R + 1) * half));
  prof_add_launches(2);
  ProfScope prof(KC_OTHER, st);
  k_fft_roots<T><<<div_up(nt, 128), 128, 0, st>>>(nt, tw.p, reinterpret_cast<C*>(out));
  LD_CHECK_LAUNCH();
  k_fft_sym_x<<<dim3(div_up(half, 128), R + 1), 128, 0, st>>>(h->gtab, R, grid_row_len(R), c, p.lnx,
                                                              p.lnt, tw.p, a.p);
  LD_CHECK_LAUNCH();
  k_fft_sym_y<T><<<dim3(div_up(1 << p.lny, 128), half), 128, 0, st>>>(
      a.p, R, p.lnx, p.lny, p.lnt, tw.p, out + 2 * (size_t)nt);
  LD_CHECK_LAUNCH();
  return LOGDET_OK;
}
template int grid_fft_table<float>(const logdet_ctx*, const GridFft&, double, float*, cudaStream_t);
template int grid_fft_table<double>(const logdet_ctx*, const GridFft&, double, double*, cudaStream_t);

template <typename T>
int grid_fft_apply(const logdet_ctx* h, const GridFft& p, const T* tab, const T* x, T* y, int ld,
                   const double* colshift, void* scratch, size_t scratch_bytes, cudaStream_t st) {
  using C = typename CplxOf<T>::type;
  constexpr int V = Vec16<T>::N;
  if (ld % V) {
    set_error("grid operator: leading dimension %d is not a multiple of %d", ld, V);
    return LOGDET_EINVAL;
  }
  const size_t unit = grid_fft_unit_bytes<T>(p);
  const long long units = (long long)(ld / V) * p.pairs;
  DevBuf<unsigned char> own(st);
  if (scratch_bytes < unit) {
    scratch_bytes = std::min(std::max((size_t)h->n * ld * sizeof(T), grid_fft_own_bytes<T>(p, ld)),
                             (size_t)units * unit);
    LD_TRY(own.alloc(scratch_bytes));
    scratch = own.p;
  }
  // Units per launch group: what the workspace holds, and no more than stays
  // in L2 between the three kernels.
  const long long fit = (long long)(std::min(scratch_bytes, std::max(unit, kGridFftGroup)) / unit);
  const int group = (int)std::min<long long>(std::min(units, fit), 32768);
  FftArgs<T> A;
  A.p = p;
  A.nx = h->gx;
  A.ny = h->gy;
  A.ld = ld;
  A.x = x;
  A.y = y;
  A.colshift = colshift;
  A.ws = static_cast<C*>(scratch);
  A.tw = reinterpret_cast<const C*>(tab);
  A.sym = tab + ((size_t)2 << p.lnt);
  // Accounting: the transforms' operations (5 N log2 N each way) and the
  // block read and written once.
  const double pts = (double)units * V * std::ldexp(1.0, p.lnx + p.lny);
  prof_add_launches(3 * ((units + group - 1) / group) - 1);  // (the scope counts one)
  ProfScope prof(KC_GRID, st, 10.0 * pts * (p.lnx + p.lny), 2.0 * (double)h->n * ld * sizeof(T));
  for (long long u0 = 0; u0 < units; u0 += group) {
    const int nu = (int)std::min<long long>(group, units - u0);
    A.u0 = (int)u0;
    LD_TRY((launch_fft<T, 0>(A, nu, st)));
    LD_TRY((launch_fft<T, 1>(A, nu, st)));
    LD_TRY((launch_fft<T, 2>(A, nu, st)));
  }
  return LOGDET_OK;
}
template int grid_fft_apply<float>(const logdet_ctx*, const GridFft&, const float*, const float*,
                                   float*, int, const double*, void*, size_t, cudaStream_t);
template int grid_fft_apply<double>(const logdet_ctx*, const GridFft&, const double*, const double*,
                                    double*, int, const double*, void*, size_t, cudaStream_t);

}  // namespace ld
