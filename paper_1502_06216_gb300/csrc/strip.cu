// strip.cu -- persistent CUDA-core form of a JKO step (FP32 / FP64, the separable
// Gaussian by taps, one density): one cooperative launch runs the pairs of the
// scaling loop (Prop. 3.3) with the stopping rule of Sec. 3.4 inside.
//
// Block g owns a strip of nc whole columns and a strip of nr whole rows, kept in
// shared memory for the whole step (a, p and the prox fields by columns; b and q
// by rows).  A filter pass along the owned axis is then local, and since xi is
// separable its two 1-D passes may be taken in either order, so a pair is
//     columns: T = K_y a             | exchange: T, columns -> rows
//     rows:    Y = T K_x, b = q / Y, U = b K_x
//                                    | exchange: U, rows -> columns
//     columns: s = K_y U, a = Prox(s)/s, p = a s
// with two exchanges through L2 where a kernel per pass makes four passes over
// images in L2 and four launches.
//
// Exchange: every element travels as an 8-byte word {32 bits of data, epoch}
// (two words for FP64), written and read as one access each, so a reader needs
// no barrier and no fence: it polls the word itself until the epoch of this pair
// appears (bounded).  The words for one receiver are contiguous.  One buffer per
// direction suffices: a block writes the words of pair k + 1 only after it has
// received all of pair k's of the other direction, which their senders wrote
// after reading theirs.  The residual of each block's rows travels the same way, twice
// buffered by pair parity (a block without columns may still be reading pair
// k's when pair k + 1's are written); every block adds all of them in one
// fixed order and takes the same decision.
#include <algorithm>

#include "jko_internal.cuh"
#include "jko_kernels.h"

namespace jko {

namespace {

constexpr unsigned kSpin = 1u << 22;   // polls of one word before giving up
constexpr int kStripMaxLine = 4096;

// ---- words of the exchange buffers: {data, epoch}, one 64-bit access each ----
__device__ __forceinline__ void put_word(unsigned long long* w, unsigned v, unsigned ep) {
  const unsigned long long x = (unsigned long long)ep << 32 | v;
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"(x) : "memory");
}
__device__ __forceinline__ void get_words(const unsigned long long* w, unsigned long long& x,
                                          unsigned long long& y) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
               : "=l"(x), "=l"(y) : "l"(w) : "memory");
}
template <typename T> constexpr int kWords = sizeof(T) / 4;   // words per element
__device__ __forceinline__ void put_elem(unsigned long long* w, float v, unsigned ep) {
  put_word(w, __float_as_uint(v), ep);
}
__device__ __forceinline__ void put_elem(unsigned long long* w, double v, unsigned ep) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  put_word(w, (unsigned)b, ep);
  put_word(w + 1, (unsigned)(b >> 32), ep);
}
// Both words of a pair, polled until they carry epoch ep; false: given up.
__device__ __forceinline__ bool wait_pair(const unsigned long long* w, unsigned ep,
                                          unsigned long long& x, unsigned long long& y,
                                          volatile int* fault) {
  for (unsigned i = 0; (unsigned)(x >> 32) != ep || (unsigned)(y >> 32) != ep; ++i) {
    if (i >= kSpin || *fault) return false;
    get_words(w, x, y);
  }
  return true;
}
__device__ __forceinline__ double words_double(unsigned long long lo, unsigned long long hi) {
  return __longlong_as_double((long long)((hi << 32) | (lo & 0xffffffffull)));
}

// ---- lines in shared memory ----
// Line l of an image strip starts at l * stride; its element i sits at sw(pad +
// i), zeros around it (at least as far as the windows below reach).  pad = r
// modulo 8 and the strides are multiples of 64 elements, so that every window
// of eight starts at a multiple of eight.  Eight FP32 outputs per thread: the
// 16-byte units a quarter-warp reads lie two apart, so the low bit of a unit's
// index is flipped in every second group of eight units (conflict-free).
constexpr int kPadR = 56;
__host__ __device__ __forceinline__ int line_pad(int r) { return 24 + (r & 7); }
__host__ __device__ __forceinline__ int line_stride(int n, int r) {
  return (line_pad(r) + n + kPadR + 63) & ~63;
}
constexpr int kTapPad = 32;   // zeros behind the taps
template <typename T, int RB>
__device__ __forceinline__ int sw(int i) {
  return (sizeof(T) == 4 && RB == 8) ? i ^ ((i >> 3) & 4) : i;
}

// acc[o] = sum_t k[t] x[i0 + o + t - r] over one line, t ascending, as
// filter_pass adds them (terms beyond the band or the line are products with
// zeros).  FP32, RB = 4 or 8: three register windows of RB elements rotate and
// the taps are read four ahead, so that shared-memory loads are in flight
// during the multiply-adds; the exit is tested once per 24 taps and the window
// addresses advance by immediates.  At 256^2 (one warp per scheduler) a pass
// over two lines takes 1.6k cycles against 2.8k with a test and an address
// computation per window.
__device__ __forceinline__ void lds4(uint32_t a, float* o) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3]) : "r"(a) : "memory");
}
template <int RB>
__device__ __forceinline__ void window(uint32_t b, float (&w)[RB]) {
  const uint32_t p = RB == 8 ? b ^ ((b >> 3) & 16u) : b;   // sw() on byte addresses
#pragma unroll
  for (int u = 0; u < RB / 4; ++u) lds4(p ^ (16u * u), w + 4 * u);
}
template <int RB>
__device__ __forceinline__ void line_taps(float (&acc)[RB], const float* line, int pad,
                                          const float* s_k, int n, int r, int i0) {
  static_assert(RB == 4 || RB == 8, "");
  constexpr int ST = 24 / RB;   // windows per exit test
  int t_lo = r - i0 - (RB - 1);
  if (t_lo < 0) t_lo = 0;
  t_lo &= ~(RB - 1);
  int t_hi = n - 1 - i0 + r;
  if (t_hi > 2 * r) t_hi = 2 * r;
  uint32_t xb = (uint32_t)__cvta_generic_to_shared(line + pad + i0 - r + t_lo);
  uint32_t kb = (uint32_t)__cvta_generic_to_shared(s_k + t_lo);
  float w[3][RB], k[2][4];
  window<RB>(xb, w[0]);
  lds4(kb, k[0]);
  window<RB>(xb + 4 * RB, w[1]);
  for (int t = t_lo; t <= t_hi; t += 24) {
#pragma unroll
    for (int s = 0; s < ST; ++s) {
      window<RB>(xb + 4 * RB * (s + 2), w[(s + 2) % 3]);
#pragma unroll
      for (int v = 0; v < RB; v += 4) {
        const int c = (s * (RB / 4) + v / 4) & 1;
        lds4(kb + 4 * (s * RB + v + 4), k[c ^ 1]);
#pragma unroll
        for (int d = 0; d < 4; ++d) {
#pragma unroll
          for (int o = 0; o < RB; ++o)
            acc[o] = fmaf(k[c][d], (o + v + d < RB) ? w[s % 3][o + v + d]
                                                    : w[(s + 1) % 3][o + v + d - RB], acc[o]);
        }
      }
    }
    xb += 4 * 24;
    kb += 4 * 24;
  }
}
// FP64 (RB = 1): bound by the FP64 pipe (64 cycles a warp instruction and
// scheduler); each lane runs its own taps inside the line, four per test.
template <int RB>
__device__ __forceinline__ void line_taps(double (&acc)[RB], const double* line, int pad,
                                          const double* s_k, int n, int r, int i0) {
  int t_lo = r - i0 - (RB - 1);
  if (t_lo < 0) t_lo = 0;
  int t_hi = n - 1 - i0 + r;
  if (t_hi > 2 * r) t_hi = 2 * r;
  const double* x = line + pad + i0 - r;
  for (int t = t_lo; t <= t_hi; t += 4) {
    double xx[4 + RB - 1], kk[4];
#pragma unroll
    for (int u = 0; u < 4 + RB - 1; ++u) xx[u] = x[t + u];
#pragma unroll
    for (int u = 0; u < 4; ++u) kk[u] = s_k[t + u];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
#pragma unroll
      for (int o = 0; o < RB; ++o) acc[o] = fma(kk[u], xx[u + o], acc[o]);
    }
  }
}

// The warp's sum of the residual terms: a tree in the working precision (FP32
// terms carry ~2^-24 each; the blocks and the grid are added in FP64).
__device__ __forceinline__ double warp_res(float v) { return (double)warp_sum_f(v); }
__device__ __forceinline__ double warp_res(double v) { return warp_sum(v); }

template <typename T>
struct StripArgs {
  int nx, ny, rx, ry, nc, nr, gr;   // gr: blocks that own rows
  unsigned mc, mr;               // ceil(2^32 / nc), ceil(2^32 / nr): division by multiply
  const T* taps_x;
  const T* taps_y;
  const T* q;
  T* a;
  T* p;
  unsigned long long* x1;        // T: [row block][x][nr], even words per block
  unsigned long long* x2;        // U: [column block][y][nc]
  unsigned long long* xres;      // residuals of the blocks' rows, 2 words each, [2][gr]
  unsigned* epoch;
  Ctrl* ctrl;
  int pairs;
};

// w / d for w < 2^16 d with m = ceil(2^32 / d) (d = 1: m wraps to 0)
__device__ __forceinline__ int div_by(int w, int d, unsigned m) {
  return d == 1 ? w : (int)__umulhi((unsigned)w, m);
}

// Shared memory of a block, in elements of T behind the taps.
template <typename T>
struct StripSmem {
  int sc, sr;          // line strides of columns and rows
  size_t kx, ky, a, c2, b, r2, q, p, E, sw, c, kap, m1f, mask, total;   // byte offsets
};
template <typename T>
__host__ __device__ inline StripSmem<T> strip_smem(int nx, int ny, int rx, int ry, int nc, int nr,
                                                   bool hE, bool hsw, bool hc, bool hkap,
                                                   bool hm1f, bool hmask) {
  StripSmem<T> S;
  S.sc = line_stride(ny, ry);
  S.sr = line_stride(nx, rx);
  size_t o = 0;
  auto take = [&](size_t n) { const size_t at = o; o += (n * sizeof(T) + 255) / 256 * 256; return at; };
  S.kx = take(2 * rx + 1 + kTapPad);
  S.ky = take(2 * ry + 1 + kTapPad);
  S.a = take((size_t)nc * S.sc);
  S.c2 = take((size_t)nc * S.sc);
  S.b = take((size_t)nr * S.sr);
  S.r2 = take((size_t)nr * S.sr);
  S.q = take((size_t)nr * nx);
  const size_t cc = (size_t)nc * ny;
  S.p = take(cc);
  S.E = take(hE ? cc : 0);
  S.sw = take(hsw ? cc : 0);
  S.c = take(hc ? cc : 0);
  S.kap = take(hkap ? cc : 0);
  S.m1f = take(hm1f ? cc : 0);
  S.mask = o;
  if (hmask) o += (cc + 127) / 128 * 128;
  S.total = o + 256;   // (the base is rounded up)
  return S;
}

template <typename T, int EK, int RB, int NT>
__global__ void __launch_bounds__(NT, 1) strip_kernel(StripArgs<T> A, ProxArgs<T> P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // 256-byte aligned: window() applies sw() to absolute shared addresses
  unsigned char* smem = smem_raw + (-(int)__cvta_generic_to_shared(smem_raw) & 255);
  __shared__ int s_bad, s_fault, s_dec;
  __shared__ double s_wres[NT / 32];
  constexpr int KW = kWords<T>;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nthreads = blockDim.x, nwarps = nthreads >> 5;
  const int nx = A.nx, ny = A.ny;
  const StripSmem<T> S = strip_smem<T>(nx, ny, A.rx, A.ry, A.nc, A.nr, EK == EK_CROWD,
                                       P.sw != nullptr, P.c != nullptr, P.kappa != nullptr,
                                       P.m1f != nullptr, P.mask != nullptr);
  T* s_kx = (T*)(smem + S.kx);
  T* s_ky = (T*)(smem + S.ky);
  T* s_a = (T*)(smem + S.a);     // a by columns
  T* s_c2 = (T*)(smem + S.c2);   // U received / T to send, by columns
  T* s_b = (T*)(smem + S.b);     // b by rows
  T* s_r2 = (T*)(smem + S.r2);   // T received / U to send, by rows
  T* s_q = (T*)(smem + S.q);
  T* s_p = (T*)(smem + S.p);
  const int padc = line_pad(A.ry), padr = line_pad(A.rx);
  Ctrl* ctrl = A.ctrl;
  // this block's columns [x0, x0 + ncg) and rows [y0, y0 + nrg)
  const int x0 = blockIdx.x * A.nc, y0 = blockIdx.x * A.nr;
  const int ncg = max(0, min(A.nc, nx - x0)), nrg = max(0, min(A.nr, ny - y0));
  const int done0 = *(volatile int*)&ctrl->done, bad0 = *(volatile int*)&ctrl->nonfinite;
  if (done0 != RUNNING || bad0) {   // the same state for every block: none waits for this one
    if (done0 == RUNNING && tid == 0 && blockIdx.x == 0) ctrl->done = NONFINITE;
    return;
  }
  const int maxit = ctrl->max_iter, stall = ctrl->stall;
  const double tol = ctrl->tol;
  const unsigned ep0 = *(volatile unsigned*)A.epoch;
  if (tid == 0) {
    s_bad = 0;
    s_fault = 0;
    s_dec = 0;
  }

  // taps, zeros around the lines, a = 1 (Sec. 3.4), q and the prox fields
  for (int t = tid; t < 2 * A.rx + 1 + kTapPad; t += nthreads)
    s_kx[t] = t <= 2 * A.rx ? A.taps_x[t] : T(0);
  for (int t = tid; t < 2 * A.ry + 1 + kTapPad; t += nthreads)
    s_ky[t] = t <= 2 * A.ry ? A.taps_y[t] : T(0);
  for (int l = wid; l < A.nc; l += nwarps)
    for (int i = lane; i < S.sc; i += 32) {
      s_c2[l * S.sc + i] = T(0);
      s_a[l * S.sc + sw<T, RB>(i)] = (i >= padc && i < padc + ny) ? T(1) : T(0);
    }
  for (int l = wid; l < A.nr; l += nwarps)
    for (int i = lane; i < S.sr; i += 32) {
      s_b[l * S.sr + i] = T(0);
      s_r2[l * S.sr + i] = T(0);
    }
  for (int l = wid; l < nrg; l += nwarps)
    for (int i = lane; i < nx; i += 32) s_q[l * nx + i] = A.q[(size_t)(y0 + l) * nx + i];
  // the prox fields by columns: element xl * ny + y of the block's copy
  ProxArgs<T> L = P;
  auto field = [&](const T* g, size_t at) -> const T* {
    T* s = (T*)(smem + at);
    for (int e = tid; e < ny * ncg; e += nthreads) {
      const int y = e / ncg, xl = e - y * ncg;
      s[xl * ny + y] = g[(size_t)y * nx + x0 + xl];
    }
    return s;
  };
  if (EK == EK_CROWD) L.E = field(P.E, S.E);
  if (P.sw != nullptr) L.sw = field(P.sw, S.sw);
  if (P.c != nullptr) L.c = field(P.c, S.c);
  if (P.kappa != nullptr) L.kappa = field(P.kappa, S.kap);
  if (P.m1f != nullptr) L.m1f = field(P.m1f, S.m1f);
  if (P.mask != nullptr) {
    uint8_t* s = (uint8_t*)(smem + S.mask);
    for (int e = tid; e < ny * ncg; e += nthreads) {
      const int y = e / ncg, xl = e - y * ncg;
      s[xl * ny + y] = P.mask[(size_t)y * nx + x0 + xl];
    }
    L.mask = s;
  }
  for (int e = tid; e < ny * A.nc; e += nthreads) s_p[e] = T(0);
  __syncthreads();

  // The filter along the owned axis: lines of n elements in `src`, RB outputs
  // per work item, op(line, first output, outputs).
  auto filter = [&](const T* src, int stride, int pad, int lines, int n, int r, const T* s_k,
                    auto&& op) {
    const int nseg = (n + RB - 1) / RB;
    for (int item = tid; item < lines * nseg; item += nthreads) {
      const int l = item / nseg, i0 = (item - l * nseg) * RB;
      T acc[RB];
#pragma unroll
      for (int o = 0; o < RB; ++o) acc[o] = T(0);
      line_taps<RB>(acc, src + l * stride, pad, s_k, n, r, i0);
      op(l, i0, acc);
    }
  };
  // outputs of a filter into the lines of dst (what lies there has been sent or read)
  auto to_lines = [&](T* dst, int stride, int pad, int n) {
    return [=](int l, int i0, T (&acc)[RB]) {
#pragma unroll
      for (int o = 0; o < RB; ++o)
        if (i0 + o < n) dst[l * stride + sw<T, RB>(pad + i0 + o)] = acc[o];
    };
  };
  // Sends the lines of src (n elements each, the block's lines [l0, l0 + lines) of
  // `total`): element i goes to block i / d of the other axis, its words at
  // [i / d][line][i mod d].
  auto send = [&](unsigned long long* X, const T* src, int stride, int pad, int l0, int lines,
                  int total, int n, int d, unsigned m, unsigned ep) {
    const size_t region = ((size_t)total * d * KW + 1) & ~(size_t)1;
    for (int i = tid; i < n; i += nthreads) {
      const int g = div_by(i, d, m), il = i - g * d;
      unsigned long long* w = X + g * region + ((size_t)l0 * d + il) * KW;
      const T* s = src + sw<T, RB>(pad + i);
      for (int l = 0; l < lines; ++l) put_elem(w + (size_t)l * d * KW, s[l * stride], ep);
    }
  };
  // Receives this block's lines (d per block, `lines` of them in use, n elements
  // each) into dst: the words [block][element][line].
  auto receive = [&](const unsigned long long* X, T* dst, int stride, int pad, int lines, int n,
                     int d, unsigned m, unsigned ep) {
    if (lines == 0) return;
    const size_t region = ((size_t)n * d * KW + 1) & ~(size_t)1;
    const unsigned long long* w0 = X + blockIdx.x * region;
    constexpr int UN = 4;   // pairs of words in flight per thread
    const int npair = (n * d * KW + 1) >> 1;
    for (int k0 = tid; k0 < npair; k0 += nthreads * UN) {
      unsigned long long x[UN], y[UN];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int k = k0 + u * nthreads;
        x[u] = y[u] = (unsigned long long)ep << 32;
        if (k < npair) get_words(w0 + 2 * (size_t)k, x[u], y[u]);
      }
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int k = k0 + u * nthreads;
        if (k >= npair) continue;
        if (KW == 2) {
          const int i = div_by(k, d, m), l = k - i * d;
          if (l >= lines) continue;
          if (!wait_pair(w0 + 2 * (size_t)k, ep, x[u], y[u], &s_fault)) s_fault = 1;
          dst[l * stride + sw<T, RB>(pad + i)] = (T)words_double(x[u], y[u]);
        } else {
          // elements 2k and 2k + 1; the last block of a ragged grid has lines
          // that nobody sends, and an odd region ends in an unused word
          const int e0 = 2 * k, e1 = 2 * k + 1;
          const int i0 = div_by(e0, d, m), l0 = e0 - i0 * d;
          const int i1 = div_by(e1, d, m), l1 = e1 - i1 * d;
          const bool u0 = l0 < lines, u1 = i1 < n && l1 < lines;
          for (unsigned t = 0; (u0 && (unsigned)(x[u] >> 32) != ep) ||
                               (u1 && (unsigned)(y[u] >> 32) != ep); ++t) {
            if (t >= kSpin || *(volatile int*)&s_fault) {
              s_fault = 1;
              break;
            }
            get_words(w0 + 2 * (size_t)k, x[u], y[u]);
          }
          if (u0) dst[l0 * stride + sw<T, RB>(pad + i0)] = (T)__uint_as_float((unsigned)x[u]);
          if (u1) dst[l1 * stride + sw<T, RB>(pad + i1)] = (T)__uint_as_float((unsigned)y[u]);
        }
      }
    }
  };

  int it = 0, pair = 0, since = 0;
  double best = INFINITY;
  for (; pair < A.pairs; ++pair) {
    const unsigned ep = ep0 + 1u + (unsigned)pair;
    // columns: T = K_y a
    filter(s_a, S.sc, padc, ncg, ny, A.ry, s_ky, to_lines(s_c2, S.sc, padc, ny));
    __syncthreads();
    send(A.x1, s_c2, S.sc, padc, x0, ncg, nx, ny, A.nr, A.mr, ep);
    receive(A.x1, s_r2, S.sr, padr, nrg, nx, A.nr, A.mr, ep);
    __syncthreads();
    // rows: Y = T K_x, the residual |b_old Y - q| and b = q / Y
    const bool have_prev = it > 0;
    int bad = 0;
    T res = T(0);
    filter(s_r2, S.sr, padr, nrg, nx, A.rx, s_kx, [&](int l, int i0, T (&acc)[RB]) {
#pragma unroll
      for (int o = 0; o < RB; ++o) {
        if (i0 + o >= nx) continue;
        const T qv = s_q[l * nx + i0 + o];
        T* bp = s_b + l * S.sr + sw<T, RB>(padr + i0 + o);
        if (have_prev) res += abs_residual<T>(*bp, acc[o], qv);
        const T bn = b_update<T>(qv, acc[o]);
        bad |= !dev_finite(bn);
        *bp = bn;
      }
    });
    // the warps' residuals in the working precision, the block's and the grid's in FP64
    const double wres = warp_res(res);
    if (lane == 0) s_wres[wid] = wres;
    if (bad) s_bad = 1;
    __syncthreads();
    // the block's residual (NaN where it met a non-finite scaling) to every block
    unsigned long long* xr = A.xres + (size_t)(pair & 1) * A.gr * 2;
    if (wid == 0 && nrg > 0) {
      const double v = warp_sum(lane < nwarps ? s_wres[lane] : 0.0);
      if (lane == 0) put_elem(xr + 2 * blockIdx.x, s_bad ? (double)NAN : v, ep);
    }
    // U = b K_x, rows -> columns
    filter(s_b, S.sr, padr, nrg, nx, A.rx, s_kx, to_lines(s_r2, S.sr, padr, nx));
    __syncthreads();
    send(A.x2, s_r2, S.sr, padr, y0, nrg, ny, nx, A.nc, A.mc, ep);
    if (wid == nwarps - 1) {
      // the stop rule (Sec. 3.4) on the sum over the blocks, in one order everywhere
      constexpr int UN = 5;   // blocks per lane whose words are in flight at once
      double v = 0.0;
      for (int g0 = lane; g0 < A.gr; g0 += 32 * UN) {
        unsigned long long lo[UN], hi[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u)
          if (g0 + 32 * u < A.gr) get_words(xr + 2 * (g0 + 32 * u), lo[u], hi[u]);
#pragma unroll
        for (int u = 0; u < UN; ++u)
          if (g0 + 32 * u < A.gr) {
            if (!wait_pair(xr + 2 * (g0 + 32 * u), ep, lo[u], hi[u], &s_fault)) s_fault = 1;
            v += words_double(lo[u], hi[u]);
          }
      }
      v = warp_sum(v);
      const bool first = lane == 0 && blockIdx.x == 0;
      int d = RUNNING;
      if (!isfinite(v)) d = NONFINITE;
      else if (it > 0 && v <= tol) d = CONVERGED;
      else if (it >= maxit) d = MAX_ITER;
      else if (stall > 0 && it >= 1) {
        // the stall rule (stall_rule), its state in this warp: every block keeps the same
        since = (it == 1 || v < best) ? 0 : since + 1;
        best = it == 1 ? v : fmin(best, v);
        if (since >= stall) d = STALLED;
      }
      if (first) {
        if (it > 0) ctrl->res_last = v;
        if (d != RUNNING) ctrl->done = d;
      }
      if (lane == 0) s_dec = d != RUNNING;
    }
    receive(A.x2, s_c2, S.sc, padc, ncg, ny, A.nc, A.mc, ep);
    __syncthreads();
    if (s_dec || s_fault) break;
    // columns: s = K_y U, a = Prox(s) / s, p = a s
    bad = 0;
    filter(s_c2, S.sc, padc, ncg, ny, A.ry, s_ky, [&](int l, int i0, T (&acc)[RB]) {
#pragma unroll
      for (int o = 0; o < RB; ++o) {
        if (i0 + o >= ny) continue;
        const int idx = l * ny + i0 + o;
        const T a = prox_ratio<T, EK>(L, idx, acc[o]);
        bad |= !dev_finite(a);
        s_a[l * S.sc + sw<T, RB>(padc + i0 + o)] = a;
        s_p[idx] = a * acc[o];
      }
    });
    if (bad) s_bad = 1;
    ++it;
    __syncthreads();
  }

  // the final a and p (p of the pair the last residual belongs to)
  for (int e = tid; e < ny * ncg; e += nthreads) {
    const int y = e / ncg, xl = e - y * ncg;
    A.a[(size_t)y * nx + x0 + xl] = s_a[xl * S.sc + sw<T, RB>(padc + y)];
    A.p[(size_t)y * nx + x0 + xl] = s_p[xl * ny + y];
  }
  if (tid == 0) {
    if (s_fault) atomicOr(&ctrl->nonfinite, 2);
    if (blockIdx.x == 0) {
      ctrl->it = it;
      *A.epoch = ep0 + 1u + (unsigned)pair;
    }
  }
}

// ---- host ----
template <typename T, int RB, int NT>
void* strip_fn_ek(int ek) {
  if (ek == EK_CROWD) return (void*)strip_kernel<T, EK_CROWD, RB, NT>;
  if (ek == EK_ENTROPY) return (void*)strip_kernel<T, EK_ENTROPY, RB, NT>;
  return (void*)strip_kernel<T, EK_POWER, RB, NT>;
}
template <typename T>
void* strip_fn(int rb, int ek);
template <>
void* strip_fn<float>(int rb, int ek) {
  return rb == 8 ? strip_fn_ek<float, 8, 512>(ek) : strip_fn_ek<float, 4, 512>(ek);
}
template <>
void* strip_fn<double>(int, int ek) { return strip_fn_ek<double, 1, 512>(ek); }

int ceil_div(int a, int b) { return (a + b - 1) / b; }
unsigned magic(int d) { return (unsigned)((0x100000000ull + (unsigned)d - 1) / (unsigned)d); }

}  // namespace

// The rule for the persistent form, on the grid, the band and the precision.
// Both sides measured on a GB300 (us a pair, this form / a kernel per pass, flows
// to tol with their launches and finalisations): FP32 128^2 8.4 / 21.4, 201 x 149
// 9.8 / 26, 256^2 10.8 / 26, 512^2 porous 42 / 56 (three pairs a step), 700^2
// 31 / 52, 1024^2 64 / 81; FP64 128^2 36 / 111, 201 x 149 57 / 132, 256^2 162 /
// 197, 512^2 1253 / 1124.  FP64 is bound by its pipe, so whole lines per block
// (4 against 3.4 on average at 512^2) cost what the launches save: up to two
// lines a block.  FP32: wherever the strips fit the shared memory of one block
// per SM (about 1060 cells a side).  Long thin grids, whose short side has too
// few lines for the blocks, keep the per-pass form unless a block's line is
// short work anyway.
template <typename T>
StripPlan strip_plan(int nx, int ny, int rx, int ry, int ek, const ProxArgs<T>& P, int max_blocks) {
  StripPlan sp;
  int dev = 0, coop = 0, sms = 0, smem_max = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return sp;
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (!coop || sms < 1 || nx > kStripMaxLine || ny > kStripMaxLine) return sp;
  const int G = max_blocks > 0 ? std::min(max_blocks, sms) : sms;
  sp.nc = ceil_div(nx, G);
  sp.nr = ceil_div(ny, G);
  if (sizeof(T) == 8 && std::max(sp.nc, sp.nr) > 2 && max_blocks <= 0) return StripPlan{};
  const double most = std::max((double)sp.nc * ny, (double)sp.nr * nx);
  const double work = std::max((double)sp.nc * ny * (2 * ry + 1), (double)sp.nr * nx * (2 * rx + 1));
  if (most * G > 4.0 * nx * ny && work > (sizeof(T) == 8 ? 4e4 : 5e5)) return StripPlan{};
  sp.G = std::max(ceil_div(nx, sp.nc), ceil_div(ny, sp.nr));
  // eight outputs per work item where that leaves every scheduler two warps, else four
  // (256^2: 8.8 us a pair with four, 11.4 with eight; 1024^2 72 and 64); FP64: one
  auto items = [&](int rb) {
    return std::max(sp.nc * ceil_div(ny, rb), sp.nr * ceil_div(nx, rb));
  };
  sp.rb = sizeof(T) == 8 ? 1 : items(8) >= 256 ? 8 : 4;
  sp.threads = std::min(512, std::max(256, ceil_div(items(sp.rb), 32) * 32));
  const auto S = strip_smem<T>(nx, ny, rx, ry, sp.nc, sp.nr, ek == EK_CROWD,
                               P.sw != nullptr, P.c != nullptr, P.kappa != nullptr,
                               P.m1f != nullptr, P.mask != nullptr);
  sp.smem = S.total;
  if (S.total + 1024 > (size_t)smem_max) return StripPlan{};
  void* fn = strip_fn<T>(sp.rb, ek);
  int per_sm = 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S.total) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, sp.threads, S.total) !=
          cudaSuccess ||
      per_sm * sms < sp.G) {
    cudaGetLastError();
    return StripPlan{};
  }
  const size_t kw = sizeof(T) / 4;
  const size_t r1 = ((size_t)nx * sp.nr * kw + 1) & ~(size_t)1;
  const size_t r2 = ((size_t)ny * sp.nc * kw + 1) & ~(size_t)1;
  sp.x1_words = r1 * ceil_div(ny, sp.nr);
  sp.x2_words = r2 * ceil_div(nx, sp.nc);
  sp.words = sp.x1_words + sp.x2_words + 4 * (size_t)sp.G + 2;
  return sp;
}

template <typename T>
cudaError_t strip_launch(const StripPlan& sp, int ek, int nx, int ny, int rx, int ry,
                         const T* taps_x, const T* taps_y, const T* q, T* a, T* p,
                         const ProxArgs<T>& P, Ctrl* ctrl, unsigned long long* words, int pairs,
                         cudaStream_t st) {
  StripArgs<T> A{nx, ny, rx, ry, sp.nc, sp.nr, ceil_div(ny, sp.nr), magic(sp.nc), magic(sp.nr), taps_x, taps_y, q, a, p,
                 words, words + sp.x1_words, words + sp.x1_words + sp.x2_words,
                 (unsigned*)(words + sp.words - 2), ctrl, pairs};
  ProxArgs<T> Pc = P;
  void* args[] = {&A, &Pc};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)sp.G);
  cfg.blockDim = dim3((unsigned)sp.threads);
  cfg.dynamicSmemBytes = sp.smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  void* fn = strip_fn<T>(sp.rb, ek);
  // another handle of the same kernel may have set a smaller limit
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sp.smem);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

#define JKO_STRIP_INST(T)                                                                      \
  template StripPlan strip_plan<T>(int, int, int, int, int, const ProxArgs<T>&, int);       \
  template cudaError_t strip_launch<T>(const StripPlan&, int, int, int, int, int, const T*,    \
                                       const T*, const T*, T*, T*, const ProxArgs<T>&, Ctrl*,  \
                                       unsigned long long*, int, cudaStream_t);
JKO_STRIP_INST(float)
JKO_STRIP_INST(double)
#undef JKO_STRIP_INST

}  // namespace jko
