// strip.cuh -- device pieces of the persistent CUDA-core kernels (strip.cu: a
// step; strip_adjoint.cu: a step of the reverse pass): images owned by strips
// of columns and rows in shared memory, and their exchange.
//
// Block g owns nc whole columns and nr whole rows of each of NI images.  A filter
// along the owned axis is local; between the two axes every element travels as
// an 8-byte word {32 bits of data, epoch} (two words for FP64), written and read
// as one access each, so a reader needs no barrier and no fence: it polls the
// word itself until the epoch of this round appears (bounded).  The words for
// one receiver are contiguous: [receiver][image][sender's line][receiver's line].
// One buffer per direction suffices: a block writes the words of round k + 1
// only after it has received all of round k's of the other direction, which their
// senders wrote after reading theirs.
#pragma once

#include "jko_internal.cuh"

namespace jko {
namespace strip {

constexpr unsigned kSpin = 1u << 22;   // polls of one word before giving up

// ---- words of the exchange buffers: {data, epoch}, one 64-bit access each ----
__device__ __forceinline__ void put_word(unsigned long long* w, unsigned v, unsigned ep) {
  const unsigned long long x = (unsigned long long)ep << 32 | v;
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"(x) : "memory");
}
__device__ __forceinline__ unsigned long long get_word(const unsigned long long* w) {
  unsigned long long x;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(w) : "memory");
  return x;
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
// FP64 (one output): bound by the FP64 pipe (64 cycles a warp instruction and
// scheduler); each lane runs its own taps inside the line, four per test, those of part
// `part` of its range (parts of len taps each).
__device__ __forceinline__ void line_taps_part(double (&acc)[1], const double* line, int pad,
                                               const double* s_k, int n, int r, int i0, int part,
                                               int len) {
  int t = r - i0;
  if (t < 0) t = 0;
  t += part * len;
  int t_hi = n - 1 - i0 + r;
  if (t_hi > 2 * r) t_hi = 2 * r;
  if (t_hi > t + len - 1) t_hi = t + len - 1;
  const double* x = line + pad + i0 - r;
  for (; t + 3 <= t_hi; t += 4) {
    double xx[4], kk[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) xx[u] = x[t + u];
#pragma unroll
    for (int u = 0; u < 4; ++u) kk[u] = s_k[t + u];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[0] = fma(kk[u], xx[u], acc[0]);
  }
  for (; t <= t_hi; ++t) acc[0] = fma(s_k[t], x[t], acc[0]);
}

// w / d for w < 2^16 d with m = ceil(2^32 / d) (d = 1: m wraps to 0)
__device__ __forceinline__ int div_by(int w, int d, unsigned m) {
  return d == 1 ? w : (int)__umulhi((unsigned)w, m);
}
// quotient of small non-negative integers (exact below 2^20)
__device__ __forceinline__ int quot(int i, float inv) { return (int)(((float)i + 0.5f) * inv); }
inline unsigned magic(int d) {
  return (unsigned)((0x100000000ull + (unsigned)d - 1) / (unsigned)d);
}
inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Grid, band and split of a launch, and its exchange buffers.
struct Geo {
  int nx, ny, rx, ry, nc, nr, gr, gc;   // gr, gc: blocks that own rows, columns
  unsigned mc, mr;                      // magic of nc, nr
  int parts, len_c, len_r;              // FP64: parts of an output's taps, taps of each by axis
  const void* taps_x;
  const void* taps_y;
  unsigned long long* x1;        // columns -> rows
  unsigned long long* x2;        // rows -> columns
  unsigned long long* xres;      // sums of the blocks, 2 words each, [2][max(gr, gc)]
  unsigned* epoch;
};

// Shared memory of a block (byte offsets from its 256-byte aligned base): the
// taps, NI images by columns and by rows twice (zero-padded lines), then `rows`
// and `cols` plain images of nr nx and nc ny elements, and the mask.
struct Smem {
  int sc, sr;          // line strides of columns and rows
  size_t kx, ky, a, c2, b, r2, part, row, col, row_b, col_b, mask, total;
};
template <typename T>
__host__ __device__ inline Smem smem_of(int nx, int ny, int rx, int ry, int nc, int nr, int ni,
                                        int parts, int rows, int cols, bool mask) {
  Smem S;
  S.sc = line_stride(ny, ry);
  S.sr = line_stride(nx, rx);
  size_t o = 0;
  auto take = [&](size_t n) { const size_t at = o; o += (n * sizeof(T) + 255) / 256 * 256; return at; };
  S.kx = take(2 * rx + 1 + kTapPad);
  S.ky = take(2 * ry + 1 + kTapPad);
  S.a = take((size_t)ni * nc * S.sc);
  S.c2 = take((size_t)ni * nc * S.sc);
  S.b = take((size_t)ni * nr * S.sr);
  S.r2 = take((size_t)ni * nr * S.sr);
  S.part = take(parts > 1 ? (size_t)parts * ni * (nc * ny > nr * nx ? nc * ny : nr * nx) : 0);
  S.row_b = ((size_t)nr * nx * sizeof(T) + 255) / 256 * 256;
  S.col_b = ((size_t)nc * ny * sizeof(T) + 255) / 256 * 256;
  S.row = o;
  S.col = S.row + rows * S.row_b;
  S.mask = S.col + cols * S.col_b;
  S.total = S.mask + (mask ? ((size_t)nc * ny + 127) / 128 * 128 : 0) + 256;   // (the base is rounded up)
  return S;
}

// This block's strips of NI images and the four moves of a round.
template <typename T, int NI, int RB>
struct Strips {
  static constexpr int KW = kWords<T>;
  const Geo& G;
  int x0, y0, ncg, nrg;          // columns [x0, x0 + ncg), rows [y0, y0 + nrg)
  int sc, sr, padc, padr;
  T *kx, *ky, *a, *c2, *b, *r2, *part;
  int* fault;

  __device__ __forceinline__ Strips(const Geo& g, const Smem& S, unsigned char* smem, int* s_fault)
      : G(g), sc(S.sc), sr(S.sr), fault(s_fault) {
    kx = (T*)(smem + S.kx);
    ky = (T*)(smem + S.ky);
    a = (T*)(smem + S.a);
    c2 = (T*)(smem + S.c2);
    b = (T*)(smem + S.b);
    r2 = (T*)(smem + S.r2);
    part = (T*)(smem + S.part);
    x0 = blockIdx.x * g.nc;
    y0 = blockIdx.x * g.nr;
    ncg = max(0, min(g.nc, g.nx - x0));
    nrg = max(0, min(g.nr, g.ny - y0));
    padc = line_pad(g.ry);
    padr = line_pad(g.rx);
  }
  // element i of line l of image m, by columns (pointers a, c2) or rows (b, r2)
  __device__ __forceinline__ int at_c(int m, int l, int i) const {
    return (m * G.nc + l) * sc + sw<T, RB>(padc + i);
  }
  __device__ __forceinline__ int at_r(int m, int l, int i) const {
    return (m * G.nr + l) * sr + sw<T, RB>(padr + i);
  }

  // taps and zeros around (and in) all lines
  __device__ __forceinline__ void load_taps() {
    for (int t = threadIdx.x; t < 2 * G.rx + 1 + kTapPad; t += blockDim.x)
      kx[t] = t <= 2 * G.rx ? ((const T*)G.taps_x)[t] : T(0);
    for (int t = threadIdx.x; t < 2 * G.ry + 1 + kTapPad; t += blockDim.x)
      ky[t] = t <= 2 * G.ry ? ((const T*)G.taps_y)[t] : T(0);
    for (int i = threadIdx.x; i < NI * G.nc * sc; i += blockDim.x) a[i] = c2[i] = T(0);
    for (int i = threadIdx.x; i < NI * G.nr * sr; i += blockDim.x) b[i] = r2[i] = T(0);
  }

  // The filter along the owned axis: RB outputs per work item,
  // op(image, line, first output, outputs).  FP64 where the outputs of a block are few
  // warps: each output's taps in parts on different warps, added in order by a thread per
  // output (the FP64 units of all four schedulers work).
  template <class F>
  __device__ __forceinline__ void filter(const T* src, int stride, int pad, int per, int lines,
                                         int n, int r, int len, const T* s_k, F&& op) {
    const int nseg = (n + RB - 1) / RB, items = NI * lines * nseg;
    const float inv = 1.0f / (float)nseg;
    auto line_of = [&](int ml, int& m, int& l) {
      m = NI == 1 ? 0 : (ml >= lines) + (NI > 2 && ml >= 2 * lines);
      l = NI == 1 ? ml : ml - m * lines;
    };
    if constexpr (RB == 1) {
      const int parts = G.parts;
      for (int f = threadIdx.x; f < parts * items; f += blockDim.x) {
        const int q = parts == 1 ? 0 : f / items, item = f - q * items;
        const int ml = quot(item, inv), i0 = item - ml * nseg;
        int m, l;
        line_of(ml, m, l);
        T acc[1] = {T(0)};
        line_taps_part(acc, src + (m * per + l) * stride, pad, s_k, n, r, i0, q, len);
        if (parts == 1) op(m, l, i0, acc);
        else part[f] = acc[0];
      }
      if (parts == 1) return;
      __syncthreads();
      for (int item = threadIdx.x; item < items; item += blockDim.x) {
        const int ml = quot(item, inv), i0 = item - ml * nseg;
        int m, l;
        line_of(ml, m, l);
        T acc[1] = {part[item]};
        for (int q = 1; q < parts; ++q) acc[0] += part[q * items + item];
        op(m, l, i0, acc);
      }
    } else {
      for (int item = threadIdx.x; item < items; item += blockDim.x) {
        const int ml = quot(item, inv), i0 = (item - ml * nseg) * RB;
        int m, l;
        line_of(ml, m, l);
        T acc[RB];
#pragma unroll
        for (int o = 0; o < RB; ++o) acc[o] = T(0);
        line_taps<RB>(acc, src + (m * per + l) * stride, pad, s_k, n, r, i0);
        op(m, l, i0, acc);
      }
    }
  }
  // f(i, value) for the outputs i0 .. of an item inside the line, one copy of f's code for
  // all of them (the outputs shift through acc[0]): an epilogue runs once a pair, and
  // unrolled it was bound by the instruction fetch.
  template <class F>
  static __device__ __forceinline__ void each(T (&acc)[RB], int i0, int n, F&& f) {
#pragma unroll 1
    for (int i = i0; i < min(i0 + RB, n); ++i) {
      f(i, acc[0]);
#pragma unroll
      for (int o = 0; o + 1 < RB; ++o) acc[o] = acc[o + 1];
    }
  }
  template <class F>
  __device__ __forceinline__ void filter_cols(const T* src, F&& op) {
    filter(src, sc, padc, G.nc, ncg, G.ny, G.ry, G.len_c, ky, op);
  }
  template <class F>
  __device__ __forceinline__ void filter_rows(const T* src, F&& op) {
    filter(src, sr, padr, G.nr, nrg, G.nx, G.rx, G.len_r, kx, op);
  }
  // ... with the outputs into the lines of dst (what lies there has been sent or read)
  __device__ __forceinline__ void filter_cols_to(const T* src, T* dst) {
    filter_cols(src, [&](int m, int l, int i0, T (&acc)[RB]) {
#pragma unroll
      for (int o = 0; o < RB; ++o)
        if (i0 + o < G.ny) dst[at_c(m, l, i0 + o)] = acc[o];
    });
  }
  __device__ __forceinline__ void filter_rows_to(const T* src, T* dst) {
    filter_rows(src, [&](int m, int l, int i0, T (&acc)[RB]) {
#pragma unroll
      for (int o = 0; o < RB; ++o)
        if (i0 + o < G.nx) dst[at_r(m, l, i0 + o)] = acc[o];
    });
  }

  // Sends the lines of src (n elements each, this block's lines [l0, l0 + lines) of
  // `total`): element i goes to block i / d of the other axis.
  __device__ __forceinline__ void send(unsigned long long* X, const T* src, int stride, int pad,
                                       int per, int l0, int lines, int total, int n, int d,
                                       unsigned md, unsigned ep) {
    const size_t region = ((size_t)NI * total * d * KW + 1) & ~(size_t)1;
    for (int k = threadIdx.x; k < NI * n; k += blockDim.x) {
      const int m = NI == 1 ? 0 : (k >= n) + (NI > 2 && k >= 2 * n), i = k - m * n;
      const int g = div_by(i, d, md), il = i - g * d;
      unsigned long long* w = X + g * region + ((size_t)(m * total + l0) * d + il) * KW;
      const T* s = src + m * per * stride + sw<T, RB>(pad + i);
      for (int l = 0; l < lines; ++l) put_elem(w + (size_t)l * d * KW, s[l * stride], ep);
    }
  }
  // Receives this block's lines (d per block, `lines` of them in use, n elements
  // each) into dst: the words [image][element][line].
  __device__ __forceinline__ void receive(const unsigned long long* X, T* dst, int stride, int pad,
                                          int lines, int n, int d, unsigned md, unsigned ep) {
    if (lines == 0) return;
    const size_t region = ((size_t)NI * n * d * KW + 1) & ~(size_t)1;
    const unsigned long long* w0 = X + blockIdx.x * region;
    constexpr int UN = 4;   // pairs of words in flight per thread
    const int npair = (NI * n * d * KW + 1) >> 1;
    // image and element from the running element index
    auto where = [&](int i, int l) {
      const int m = NI == 1 ? 0 : (i >= n) + (NI > 2 && i >= 2 * n);
      return (m * d + l) * stride + sw<T, RB>(pad + i - m * n);
    };
    for (int k0 = threadIdx.x; k0 < npair; k0 += blockDim.x * UN) {
      unsigned long long x[UN], y[UN];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int k = k0 + u * blockDim.x;
        x[u] = y[u] = (unsigned long long)ep << 32;
        if (k < npair) get_words(w0 + 2 * (size_t)k, x[u], y[u]);
      }
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int k = k0 + u * blockDim.x;
        if (k >= npair) continue;
        if (KW == 2) {
          const int i = div_by(k, d, md), l = k - i * d;
          if (l >= lines) continue;
          if (!wait_pair(w0 + 2 * (size_t)k, ep, x[u], y[u], fault)) *fault = 1;
          dst[where(i, l)] = (T)words_double(x[u], y[u]);
        } else {
          // elements 2k and 2k + 1; the last block of a ragged grid has lines
          // that nobody sends, and an odd region ends in an unused word
          const int e0 = 2 * k, e1 = 2 * k + 1;
          const int i0 = div_by(e0, d, md), l0 = e0 - i0 * d;
          const int i1 = div_by(e1, d, md), l1 = e1 - i1 * d;
          const bool u0 = l0 < lines, u1 = i1 < NI * n && l1 < lines;
          for (unsigned t = 0; (u0 && (unsigned)(x[u] >> 32) != ep) ||
                               (u1 && (unsigned)(y[u] >> 32) != ep); ++t) {
            if (t >= kSpin || *(volatile int*)fault) {
              *fault = 1;
              break;
            }
            get_words(w0 + 2 * (size_t)k, x[u], y[u]);
          }
          if (u0) dst[where(i0, l0)] = (T)__uint_as_float((unsigned)x[u]);
          if (u1) dst[where(i1, l1)] = (T)__uint_as_float((unsigned)y[u]);
        }
      }
    }
  }
  // K_y a on its way to the rows, b K_x on its way to the columns, through the lines of c2
  // and r2 (whole segments per store); FP64's parts leave an output per thread, neighbours in
  // order, which go straight out.
  __device__ __forceinline__ void filter_send_cols(unsigned ep) {
    if constexpr (RB == 1) {
      if (G.parts > 1) {
        const size_t region = ((size_t)NI * G.nx * G.nr * KW + 1) & ~(size_t)1;
        filter_cols(a, [&](int m, int l, int i, T (&v)[RB]) {
          const int g = div_by(i, G.nr, G.mr), il = i - g * G.nr;
          put_elem(G.x1 + g * region + ((size_t)(m * G.nx + x0 + l) * G.nr + il) * KW, v[0], ep);
        });
        return;
      }
    }
    filter_cols_to(a, c2);
    __syncthreads();
    send(G.x1, c2, sc, padc, G.nc, x0, ncg, G.nx, G.ny, G.nr, G.mr, ep);
  }
  __device__ __forceinline__ void filter_send_rows(unsigned ep) {
    if constexpr (RB == 1) {
      if (G.parts > 1) {
        const size_t region = ((size_t)NI * G.ny * G.nc * KW + 1) & ~(size_t)1;
        filter_rows(b, [&](int m, int l, int i, T (&v)[RB]) {
          const int g = div_by(i, G.nc, G.mc), il = i - g * G.nc;
          put_elem(G.x2 + g * region + ((size_t)(m * G.ny + y0 + l) * G.nc + il) * KW, v[0], ep);
        });
        return;
      }
    }
    filter_rows_to(b, r2);
    __syncthreads();
    send(G.x2, r2, sr, padr, G.nr, y0, nrg, G.ny, G.nx, G.nc, G.mc, ep);
  }
  // ... into r2 (rows), into c2 (columns)
  __device__ __forceinline__ void receive_rows(unsigned ep) {
    receive(G.x1, r2, sr, padr, nrg, G.nx, G.nr, G.mr, ep);
  }
  __device__ __forceinline__ void receive_cols(unsigned ep) {
    receive(G.x2, c2, sc, padc, ncg, G.ny, G.nc, G.mc, ep);
  }

  // This block's columns of a global [ny][nx] image into dst[l ny + i] (NULL: ones),
  // its rows into dst[l nx + i].
  __device__ __forceinline__ void load_cols(const T* g, T* dst) {
    for (int e = threadIdx.x; e < G.ny * ncg; e += blockDim.x) {
      const int y = e / ncg, xl = e - y * ncg;
      dst[xl * G.ny + y] = g != nullptr ? g[(size_t)y * G.nx + x0 + xl] : T(1);
    }
  }
  __device__ __forceinline__ void load_rows(const T* g, T* dst) {
    for (int e = threadIdx.x; e < G.nx * nrg; e += blockDim.x)
      dst[e] = g != nullptr ? g[(size_t)y0 * G.nx + e] : T(1);
  }
};

// The sum over `blocks` blocks of the doubles they put with epoch ep at xr, in one
// order everywhere (one warp; every lane gets it).
__device__ __forceinline__ double gather_sum(const unsigned long long* xr, int blocks, unsigned ep,
                                             int* fault) {
  constexpr int UN = 5;   // blocks per lane whose words are in flight at once
  const int lane = threadIdx.x & 31;
  double v = 0.0;
  for (int g0 = lane; g0 < blocks; g0 += 32 * UN) {
    unsigned long long lo[UN], hi[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u)
      if (g0 + 32 * u < blocks) get_words(xr + 2 * (g0 + 32 * u), lo[u], hi[u]);
#pragma unroll
    for (int u = 0; u < UN; ++u)
      if (g0 + 32 * u < blocks) {
        if (!wait_pair(xr + 2 * (g0 + 32 * u), ep, lo[u], hi[u], fault)) *fault = 1;
        v += words_double(lo[u], hi[u]);
      }
  }
  return warp_sum(v);
}

}  // namespace strip

// Geometry of a plan's launch, and the cooperative launch of one of these kernels (whose
// max_dynamic_smem the plan has set).
struct StripPlan;
strip::Geo strip_geo(const StripPlan& sp, int nx, int ny, int rx, int ry, const void* taps_x,
                     const void* taps_y, unsigned long long* words);
cudaError_t strip_coop(void* fn, const StripPlan& sp, size_t smem, int threads, void** args,
                       cudaStream_t st);

}  // namespace jko
