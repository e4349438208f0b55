// fft_filter.cu -- the Gibbs-kernel application by FFT convolution (CUDA
// cores, FP32 / FP64): the same pass as filter_pass (simt_filter.cu),
//     out[j][i'] = sum_i k(|i' - i|) in[i][j],   in: [n_i][n_j], out: [n_j][n_i],
// with the same epilogues, but each line is convolved through its discrete
// Fourier transform instead of the 2r+1 taps: O(n log n) per line against
// O(n r), the fast route to the separable Gaussian filtering of Sec. 4.1.
//
// The filter is the exact restriction of the Gaussian to the grid, a Toeplitz
// matrix of band radius r (r: the last offset whose tap is a normal number in
// the working precision, as for the taps).  Embedded in a circulant of length
// L >= n_i + r (a power of two), its product with a line zero-padded to L is
// the linear convolution on the line's n_i outputs: an input index wraps
// around only into the zero padding.  The circulant's first column c is
// symmetric (c[d] = c[L - d] = k(d), d <= r), so its spectrum
// K^[f] = sum_d c[d] e^{-2 pi i f d / L} is real; two real lines x, y packed as
// x + i y give k * x + i (k * y) in one transform.  Per block: FJ = 2 or 4
// columns of the input as one or two complex lines in shared memory.  The
// forward transform is decimation in frequency in place (natural order in,
// bit-reversed out), two radix-2 levels at a time in registers; its innermost
// levels, the product with K^ (which carries 1/L, read at the bit-reversed
// index) and the first levels of the inverse, decimation in time from the
// bit-reversed order, are one pass over the line, so no reordering is ever done.
// The outermost levels read the image directly; where the line fills at most
// half of L the zero half is left out.  Then the epilogue as in filter_pass.
// Spectrum and twiddles are computed in FP64 on the host.
//
// FP64 is bound by its pipe (2 multiply-adds a cycle and SM): 28 instructions for
// four points and two levels, so lines are spread over all SMs (512^2: 128 blocks of
// two lines where 64 blocks of four left 88 SMs idle) and shared memory is
// touched once per two levels.  512^2, L = 1024, FP64: a store pass 108 -> 42 us, with
// the b-update 134 -> 56 us; its multiply-adds alone would take 32 us on all SMs.
//
// Rounding: the transforms are accurate normwise: each output carries an
// error of about eps log2(L) times the largest entry of its input line,
// where the band filter's error is relative to each output's own terms.
#include <cmath>
#include <vector>

#include "jko_internal.cuh"
#include "jko_kernels.h"

namespace jko {

namespace {

constexpr int FNT = 512;   // threads per block at most

// Input columns per block: four (a 32-byte sector of FP64 per row), or two where blocks of
// four would leave more than a third of the SMs without one.  Us a pair with two / four (porous,
// 152 SMs: the line lies at 404): FP64 200^2 96 / 139, 300^2 134 / 234, 400^2 244 / 254, 512^2
// 260 / 270, 600^2 479 / 487, 800^2 755 / 981, 1000^2 1035 / 1043; FP32 300^2 37.6 / 40.5, 400^2
// 51.3 / 53.4, 512^2 52.5 / 53.8, 800^2 123 / 145, 1000^2 162 / 148, 1200^2 170 / 153, 2000^2 557 / 614.
int fft_cols(int n_j) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return n_j > 4 * (2 * sms / 3) ? 4 : 2;
}

template <typename T> struct C2;
template <> struct C2<float> { using t = float2; };
template <> struct C2<double> { using t = double2; };

template <typename V>
__device__ __forceinline__ V cmul(V a, V b) {
  V r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}
template <typename V>
__device__ __forceinline__ V cmul_conj(V a, V b) {   // a * conj(b)
  V r;
  r.x = a.x * b.x + a.y * b.y;
  r.y = a.y * b.x - a.x * b.y;
  return r;
}

// Element i of a line sits at fpad(i): one element skipped per 128 bytes, so that the
// strided accesses of the inner levels spread over the banks.
template <typename T>
__host__ __device__ __forceinline__ int fpad(int i) { return i + (i >> (sizeof(T) == 8 ? 3 : 4)); }

// Two radix-2 levels on (x0, x1, x2, x3) = points k, k + h, k + 2h, k + 3h of a group
// of m = 4h: forward (decimation in frequency) with w_j = e^{-2 pi i j k / m}, and its
// mirror (decimation in time, conjugate twiddles, unnormalised).
template <typename V>
__device__ __forceinline__ void dif4(V& x0, V& x1, V& x2, V& x3, V w1, V w2, V w3) {
  const V s0{x0.x + x2.x, x0.y + x2.y}, s1{x1.x + x3.x, x1.y + x3.y};
  const V d0{x0.x - x2.x, x0.y - x2.y}, d1{x1.y - x3.y, x3.x - x1.x};   // d1 = -i (x1 - x3)
  x0 = V{s0.x + s1.x, s0.y + s1.y};
  x1 = cmul(V{s0.x - s1.x, s0.y - s1.y}, w2);
  x2 = cmul(V{d0.x + d1.x, d0.y + d1.y}, w1);
  x3 = cmul(V{d0.x - d1.x, d0.y - d1.y}, w3);
}
// ... where x2 = x3 = 0
template <typename V>
__device__ __forceinline__ void dif4_half(V& x0, V& x1, V& x2, V& x3, V w1, V w2, V w3) {
  const V d1{x1.y, -x1.x};
  x2 = cmul(V{x0.x + d1.x, x0.y + d1.y}, w1);
  x3 = cmul(V{x0.x - d1.x, x0.y - d1.y}, w3);
  const V s{x0.x - x1.x, x0.y - x1.y};
  x0 = V{x0.x + x1.x, x0.y + x1.y};
  x1 = cmul(s, w2);
}
template <typename V>
__device__ __forceinline__ void dit4(V& y0, V& y1, V& y2, V& y3, V w1, V w2, V w3) {
  const V b1 = cmul_conj(y1, w2), b2 = cmul_conj(y2, w1), b3 = cmul_conj(y3, w3);
  const V s0{y0.x + b1.x, y0.y + b1.y}, s1{y0.x - b1.x, y0.y - b1.y};
  const V d0{b2.x + b3.x, b2.y + b3.y}, d1{b3.y - b2.y, b2.x - b3.x};   // d1 = i (b2 - b3)
  y0 = V{s0.x + d0.x, s0.y + d0.y};
  y1 = V{s1.x + d1.x, s1.y + d1.y};
  y2 = V{s0.x - d0.x, s0.y - d0.y};
  y3 = V{s1.x - d1.x, s1.y - d1.y};
}

template <typename T, int EPI, int EK, int FJ>
__global__ void __launch_bounds__(FNT)
fft_pass_kernel(PassArgs<T> A, ProxArgs<T> P, FftArgs<T> F) {
  using V = typename C2<T>::t;
  constexpr int FNL = FJ / 2;   // complex lines
  Ctrl* ctrl = A.ctrl;
  __shared__ int s_it;
  if (stop_gate(ctrl, A.part, A.nparts, A.decide != 0, &s_it)) return;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int L = F.L, lg = F.log2L, LP = fpad<T>(L) + 1;
  V* s_z = reinterpret_cast<V*>(smem_raw);          // FNL padded lines of L
  V* s_w = s_z + (size_t)FNL * LP;                    // twiddles e^{-2 pi i j / L}, j < 3 L / 4
  __shared__ double s_red[33];
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int j = tid; j < (3 * L) / 4; j += nt) s_w[j] = reinterpret_cast<const V*>(F.tw)[j];
  const int j0 = blockIdx.x * FJ;
  auto at = [&](int line, int i) -> V& { return s_z[line * LP + fpad<T>(i)]; };
  // row i of columns j0 + 2 line, + 1 (zero outside the image)
  auto load = [&](int line, int i) -> V {
    const int jj = j0 + 2 * line;
    V v{T(0), T(0)};
    if (i < A.n_i && jj < A.n_j) {
      const T* g = A.in + (size_t)i * A.n_j + jj;
      v.x = __ldg(g);
      if (jj + 1 < A.n_j) v.y = __ldg(g + 1);
    }
    return v;
  };
  __syncthreads();   // the twiddles
  const int quads = L >> 2;
  const int mid = (lg & 1) ? 2 : 4;   // size of the innermost levels
  // forward, outermost levels: straight from the image
  if (L > mid) {
    const int h = quads;
    for (int b = tid; b < FNL * quads; b += nt) {
      const int line = b % FNL, k = b / FNL;
      V x0 = load(line, k), x1 = load(line, k + h), x2, x3;
      if (2 * A.n_i <= L) {
        dif4_half(x0, x1, x2, x3, s_w[k], s_w[2 * k], s_w[3 * k]);
      } else {
        x2 = load(line, k + 2 * h);
        x3 = load(line, k + 3 * h);
        dif4(x0, x1, x2, x3, s_w[k], s_w[2 * k], s_w[3 * k]);
      }
      at(line, k) = x0;
      at(line, k + h) = x1;
      at(line, k + 2 * h) = x2;
      at(line, k + 3 * h) = x3;
    }
  } else {
    for (int b = tid; b < FNL * L; b += nt) at(b % FNL, b / FNL) = load(b % FNL, b / FNL);
  }
  __syncthreads();
  for (int lm = lg - 2; lm > 2; lm -= 2) {
    const int h = 1 << (lm - 2), ts = lg - lm;
    for (int b = tid; b < FNL * quads; b += nt) {
      const int line = b / quads, bb = b - line * quads;
      const int k = bb & (h - 1), i = ((bb >> (lm - 2)) << lm) + k, w = k << ts;
      V &z0 = at(line, i), &z1 = at(line, i + h), &z2 = at(line, i + 2 * h),
        &z3 = at(line, i + 3 * h);
      V x0 = z0, x1 = z1, x2 = z2, x3 = z3;
      dif4(x0, x1, x2, x3, s_w[w], s_w[2 * w], s_w[3 * w]);
      z0 = x0;
      z1 = x1;
      z2 = x2;
      z3 = x3;
    }
    __syncthreads();
  }
  // innermost levels (their twiddles are 1), the real spectrum (with 1/L), and back:
  // position i holds frequency brev(i)
  for (int b = tid; b < FNL * (L / mid); b += nt) {
    const int line = b / (L / mid), i = (b - line * (L / mid)) * mid;
    auto kh = [&](int e) { return __ldg(F.khat + (__brev((unsigned)(i + e)) >> (32 - lg))); };
    V &z0 = at(line, i), &z1 = at(line, i + 1);
    if (mid == 2) {
      const T k0 = kh(0), k1 = kh(1);
      const V u{(z0.x + z1.x) * k0, (z0.y + z1.y) * k0};
      const V v{(z0.x - z1.x) * k1, (z0.y - z1.y) * k1};
      z0 = V{u.x + v.x, u.y + v.y};
      z1 = V{u.x - v.x, u.y - v.y};
    } else {
      V &z2 = at(line, i + 2), &z3 = at(line, i + 3);
      const T k0 = kh(0), k1 = kh(1), k2 = kh(2), k3 = kh(3);
      const V s0{z0.x + z2.x, z0.y + z2.y}, s1{z1.x + z3.x, z1.y + z3.y};
      const V d0{z0.x - z2.x, z0.y - z2.y}, d1{z1.y - z3.y, z3.x - z1.x};
      const V y0{(s0.x + s1.x) * k0, (s0.y + s1.y) * k0}, y1{(s0.x - s1.x) * k1, (s0.y - s1.y) * k1};
      const V y2{(d0.x + d1.x) * k2, (d0.y + d1.y) * k2}, y3{(d0.x - d1.x) * k3, (d0.y - d1.y) * k3};
      const V t0{y0.x + y1.x, y0.y + y1.y}, t1{y0.x - y1.x, y0.y - y1.y};
      const V e0{y2.x + y3.x, y2.y + y3.y}, e1{y3.y - y2.y, y2.x - y3.x};
      z0 = V{t0.x + e0.x, t0.y + e0.y};
      z1 = V{t1.x + e1.x, t1.y + e1.y};
      z2 = V{t0.x - e0.x, t0.y - e0.y};
      z3 = V{t1.x - e1.x, t1.y - e1.y};
    }
  }
  __syncthreads();
  // inverse: the same levels outwards, natural-order output
  for (int lm = 4 - (lg & 1); lm <= lg; lm += 2) {
    const int h = 1 << (lm - 2), ts = lg - lm;
    const bool half = lm == lg && 2 * A.n_i <= L;   // the upper half is not needed
    for (int b = tid; b < FNL * quads; b += nt) {
      const int line = b / quads, bb = b - line * quads;
      const int k = bb & (h - 1), i = ((bb >> (lm - 2)) << lm) + k, w = k << ts;
      V &z0 = at(line, i), &z1 = at(line, i + h);
      V x0 = z0, x1 = z1, x2 = at(line, i + 2 * h), x3 = at(line, i + 3 * h);
      dit4(x0, x1, x2, x3, s_w[w], s_w[2 * w], s_w[3 * w]);
      z0 = x0;
      z1 = x1;
      if (!half) {
        at(line, i + 2 * h) = x2;
        at(line, i + 3 * h) = x3;
      }
    }
    __syncthreads();
  }

  // ---- epilogue: FJ output rows (columns j0 + c), along each row ----
  const int lane = tid & 31;
  T res_t = T(0);
  int bad = 0;
  const bool have_prev = EPI == EPI_B && s_it > 0;
  const int cols = min(FJ, A.n_j - j0);
  for (int e = tid; e < cols * A.n_i; e += nt) {
    const int c = e / A.n_i, i = e - c * A.n_i;
    const V z = at(c >> 1, i);
    const T acc = (c & 1) ? z.y : z.x;
    const size_t idx = (size_t)(j0 + c) * A.n_i + i;
    if (EPI == EPI_STORE) {
      A.out[idx] = acc;
    } else if (EPI == EPI_B) {
      const T qv = A.q[idx];
      if (have_prev) res_t += abs_residual<T>(A.out[idx], acc, qv);
      const T bn = b_update<T>(qv, acc);
      bad |= !dev_finite(bn);
      A.out[idx] = bn;
    } else {
      // xi b >= 0 for b >= 0: an output below 0 is the transform's rounding
      // (of the line's largest entry) and is taken as 0, so that p >= 0
      const T sv = acc < T(0) ? T(0) : acc;
      const T a = prox_ratio<T, EK>(P, (int)idx, sv);
      bad |= !dev_finite(a);
      A.out[idx] = a;
      A.p[idx] = a * sv;
    }
  }
  if (EPI == EPI_STORE) return;
  bad = warp_or(bad);
  if (EPI == EPI_B) {
    const double res = block_sum((double)res_t, s_red);
    if (tid == 0) A.part[blockIdx.x] = res;
  }
  if (lane == 0 && bad) atomicOr(&ctrl->nonfinite, 1);
  if (EPI == EPI_A && tid == 0 && blockIdx.x == 0) ctrl->it = s_it + 1;
}

template <typename T>
size_t fft_smem(int L, int fj) {
  return sizeof(typename C2<T>::t) * ((size_t)(fj / 2) * (fpad<T>(L) + 1) + (size_t)(3 * L) / 4);
}

template <typename T, int EPI, int EK, int FJ>
cudaError_t launch_fft_fj(const PassArgs<T>& A, const ProxArgs<T>& P, const FftArgs<T>& F,
                          cudaStream_t st) {
  const size_t smem = fft_smem<T>(F.L, FJ);
  auto kern = fft_pass_kernel<T, EPI, EK, FJ>;
  cudaError_t e = max_dynamic_smem((const void*)kern);
  if (e != cudaSuccess) return e;
  // one thread per four points and line, 64 to 512
  int threads = FJ / 2 * F.L / 4;
  threads = threads < 64 ? 64 : threads > FNT ? FNT : threads;
  kern<<<fft_pass_blocks(A.n_j), threads, smem, st>>>(A, P, F);
  return cudaGetLastError();
}
template <typename T, int EPI, int EK>
cudaError_t launch_fft(const PassArgs<T>& A, const ProxArgs<T>& P, const FftArgs<T>& F,
                       cudaStream_t st) {
  return fft_cols(A.n_j) == 4 ? launch_fft_fj<T, EPI, EK, 4>(A, P, F, st)
                              : launch_fft_fj<T, EPI, EK, 2>(A, P, F, st);
}

}  // namespace

int fft_pass_blocks(int n_j) { return (n_j + fft_cols(n_j) - 1) / fft_cols(n_j); }

// Transform length and tables of one axis of n cells with band radius r.
bool fft_axis_tables(int n, int r, double length, double gamma, int max_len, int* L, int* log2L,
                     std::vector<double>* khat, std::vector<double>* tw) {
  int lg = 1;
  while ((1 << lg) < n + r) ++lg;
  const int Ln = 1 << lg;
  if (Ln > max_len) return false;
  *L = Ln;
  *log2L = lg;
  const double h = length / n;
  const double pi = 3.14159265358979323846;
  std::vector<double> c(r + 1);
  for (int d = 0; d <= r; ++d) c[d] = std::exp(-(d * h) * (d * h) / gamma);
  khat->assign(Ln, 0.0);
  for (int f = 0; f < Ln; ++f) {
    // K^[f] = c0 + 2 sum_{d=1}^{r} c_d cos(2 pi f d / L), the angle reduced
    // exactly modulo 2 pi; with the 1/L of the inverse transform
    double s = c[0];
    for (int d = 1; d <= r; ++d) {
      const long long m = ((long long)f * d) % Ln;
      s += 2.0 * c[d] * std::cos(2.0 * pi * (double)m / Ln);
    }
    (*khat)[f] = s / Ln;
  }
  tw->assign(2 * Ln, 0.0);   // interleaved re, im of e^{-2 pi i j / L}, j < L
  for (int j = 0; j < Ln; ++j) {
    (*tw)[2 * j] = std::cos(2.0 * pi * j / Ln);
    (*tw)[2 * j + 1] = -std::sin(2.0 * pi * j / Ln);
  }
  return true;
}

template <typename T>
cudaError_t fft_pass(int epi, int ek, const PassArgs<T>& A, const ProxArgs<T>& P,
                     const FftArgs<T>& F, cudaStream_t st) {
  if (epi == EPI_STORE) return launch_fft<T, EPI_STORE, EK_CROWD>(A, P, F, st);
  if (epi == EPI_B) return launch_fft<T, EPI_B, EK_CROWD>(A, P, F, st);
  switch (ek) {
    case EK_CROWD: return launch_fft<T, EPI_A, EK_CROWD>(A, P, F, st);
    case EK_ENTROPY: return launch_fft<T, EPI_A, EK_ENTROPY>(A, P, F, st);
    default: return launch_fft<T, EPI_A, EK_POWER>(A, P, F, st);
  }
}

template cudaError_t fft_pass<float>(int, int, const PassArgs<float>&, const ProxArgs<float>&,
                                     const FftArgs<float>&, cudaStream_t);
template cudaError_t fft_pass<double>(int, int, const PassArgs<double>&, const ProxArgs<double>&,
                                      const FftArgs<double>&, cudaStream_t);

}  // namespace jko
