// strip_adjoint.cu -- one step of the reverse pass (jko_adjoint.cu) as one
// cooperative launch on the strips of strip.cu: the fixed-point quantities of the
// step recomputed from its tape, the direct terms, the adjoint solve
//     lambda = abar - xi( D (.) xi(R_s (.) lambda) )
// with its stopping test, and the gradients.  Every application of xi is a round
// of two local filters and an exchange, as in the forward pair:
//     columns: T = K_y x               | exchange, columns -> rows
//     rows:    Z = T K_x, y = D Z, U = y K_x
//                                      | exchange, rows -> columns
//     columns: K_y U, the update of lambda, x = R_s lambda
// lambda, abar, R_s and s stay in shared memory by columns, D, 1 / Y and the
// direct term of qbar by rows.  A kernel per filter pass and per pointwise update
// took nine launches an iteration, each a few us of launch and L2 latency, and a host wait
// every eight: the ten-step gradient at 256^2 FP32 took 12.1 ms (106 pairs forward; most of them
// here), with the step and its reverse on strips 3.8.
// Four steps of the reverse pass alone, a kernel per pass / here: 512^2 FP32 3.2 / 1.5 ms,
// 700^2 4.8 / 2.6, 256^2 FP64 8.5 / 6.2.
#include "adjoint_cell.h"
#include "epoch.h"
#include "jko_kernels.h"
#include "strip.cuh"

namespace jko {

namespace {

using namespace strip;

template <typename T>
struct AdjArgs {
  Geo g;
  const T* q;          // tape of this step: its input and final a
  const T* a;
  const T* gin;        // gradient with respect to the step's output
  T* gout;             // ... and to its input (may be gin: read before the first exchange)
  T* wbar;             // accumulates, or NULL
  double mass;         // sum p of the step
  int renorm;
  double tol;
  int budget;
  AdjStatus* out;
  const AdjStatus* after;   // status of the step behind this one (NULL: last of the flow)
};

constexpr int kAdjRows = 3;   // D (first q), 1 / Y, direct term of qbar
constexpr int kAdjCols = 4;   // abar (first g, then its renormalised form), s, lambda, R_s

template <typename T, int EK, int RB, int NT>
__global__ void __launch_bounds__(NT, 1)
strip_adjoint_kernel(const __grid_constant__ AdjArgs<T> A, const __grid_constant__ ProxArgs<T> P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + (-(int)__cvta_generic_to_shared(smem_raw) & 255);
  __shared__ int s_fault;
  __shared__ double s_wres[NT / 32], s_tot;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nthreads = blockDim.x, nwarps = nthreads >> 5;
  const int nx = A.g.nx, ny = A.g.ny;
  if (A.after != nullptr && *(volatile const int*)&A.after->bad) {
    // the solve behind failed: every block returns, the status goes on
    if (tid == 0 && blockIdx.x == 0) A.out->bad = A.after->bad;
    return;
  }
  const Smem S = smem_of<T>(nx, ny, A.g.rx, A.g.ry, A.g.nc, A.g.nr, 1, A.g.parts, kAdjRows, kAdjCols, false);
  Strips<T, 1, RB> X(A.g, S, smem, &s_fault);
  auto row = [&](int k) { return (T*)(smem + S.row + k * S.row_b); };
  auto col = [&](int k) { return (T*)(smem + S.col + k * S.col_b); };
  T *s_D = row(0), *s_iY = row(1), *s_qb = row(2);
  T *s_ab = col(0), *s_s = col(1), *s_lam = col(2), *s_rs = col(3);
  const int ncg = X.ncg, nrg = X.nrg;
  const unsigned ep0 = *(volatile unsigned*)A.g.epoch;
  unsigned ep = ep0;
  if (tid == 0) s_fault = 0;
  X.load_taps();
  X.load_rows(A.q, s_D);
  X.load_cols(A.gin, s_ab);
  __syncthreads();
  for (int e = tid; e < ny * ncg; e += nthreads) {
    const int y = e / ncg, xl = e - y * ncg;
    X.a[X.at_c(0, xl, y)] = A.a[(size_t)y * nx + X.x0 + xl];
  }
  __syncthreads();

  // the two halves of a round: a (columns) -> r2 (rows), b (rows) -> c2 (columns)
  auto to_rows = [&]() {
    ++ep;
    X.filter_send_cols(ep);
    X.receive_rows(ep);
    __syncthreads();
  };
  auto to_cols = [&]() {
    __syncthreads();
    X.filter_send_rows(ep);
    X.receive_cols(ep);
    __syncthreads();
  };
  // op(element of the plain images, element of the lines, value) over a filter's outputs
  auto rows_out = [&](auto&& op) {
    X.filter_rows(X.r2, [&](int, int l, int i0, T (&acc)[RB]) {
      X.each(acc, i0, nx, [&](int i, T v) { op(l * nx + i, X.at_r(0, l, i), v); });
    });
  };
  // the sum of every block's v, the same everywhere; twice buffered as the residuals
  // of the forward step are
  int red = 0;
  auto grid_sum = [&](double v) -> double {
    v = warp_sum(v);
    if (lane == 0) s_wres[wid] = v;
    __syncthreads();
    if (wid == 0) {
      unsigned long long* xr = A.g.xres + (size_t)(red & 1) * A.g.gc * 2;
      const double b = warp_sum(lane < nwarps ? s_wres[lane] : 0.0);
      if (lane == 0 && (int)blockIdx.x < A.g.gc) put_elem(xr + 2 * blockIdx.x, b, ep);
      const double t = gather_sum(xr, A.g.gc, ep, &s_fault);
      if (lane == 0) s_tot = t;
    }
    ++red;
    __syncthreads();
    return s_tot;
  };

  // Y = xi a, b = q / Y and s = xi b of the fixed point; D = b / Y
  to_rows();
  rows_out([&](int e, int i, T Y) {
    const T b = b_update<T>(s_D[e], Y);
    const T iv = Y >= NormalMin<T>::v ? T(1) / Y : T(0);
    X.b[i] = b;
    s_iY[e] = iv;
    s_D[e] = b * iv;
  });
  to_cols();
  // the adjoint of the renormalisation p / sum p: <g, a s>
  double acc_d = 0.0;
  X.filter_cols(X.c2, [&](int, int l, int i0, T (&acc)[RB]) {
    X.each(acc, i0, ny, [&](int i, T s) {
      const int e = l * ny + i;
      s_s[e] = s;
      acc_d += (double)s_ab[e] * (double)X.a[X.at_c(0, l, i)] * (double)s;
    });
  });
  {
    const double dot = grid_sum(acc_d);
    const double c = A.renorm ? dot / A.mass : 0.0, inv = A.renorm ? 1.0 / A.mass : 1.0;
    for (int l = 0; l < ncg; ++l)
      for (int i = tid; i < ny; i += nthreads) {
        const T gt = (T)(((double)s_ab[l * ny + i] - c) * inv);
        s_ab[l * ny + i] = gt;
        X.a[X.at_c(0, l, i)] *= gt;
      }
    __syncthreads();
  }
  // the direct terms: v = xi(a g), qbar_0 = v / Y, abar = s g - xi(D v)
  to_rows();
  rows_out([&](int e, int i, T v) {
    X.b[i] = s_D[e] * v;
    s_qb[e] = v * s_iY[e];
  });
  to_cols();
  acc_d = 0.0;
  X.filter_cols(X.c2, [&](int, int l, int i0, T (&acc)[RB]) {
    X.each(acc, i0, ny, [&](int i, T xv) {
      const int e = l * ny + i;
      const T ab = s_s[e] * s_ab[e] - xv;
      T rs, rw;
      ratio_grad<T, EK>(P, i * nx + X.x0 + l, s_s[e], rs, rw);
      s_ab[e] = ab;
      s_lam[e] = ab;
      s_rs[e] = rs;
      X.a[X.at_c(0, l, i)] = rs * ab;
      acc_d += fabs((double)ab);
    });
  });
  const double norm = grid_sum(acc_d);

  // the solve from lambda = abar; every eight iterations the sum of their changes is
  // tested against eight times tol sum |abar| (the last one dominates a contracting sequence)
  int k = 0, bad = 0;
  acc_d = 0.0;
  while (k < A.budget) {
    to_rows();
    rows_out([&](int e, int i, T z) { X.b[i] = s_D[e] * z; });
    to_cols();
    X.filter_cols(X.c2, [&](int, int l, int i0, T (&acc)[RB]) {
      T u[RB];
#pragma unroll
      for (int o = 0; o < RB; ++o) {   // (all loads before the first store)
        const int e = l * ny + i0 + o;
        u[o] = T(0);
        if (i0 + o >= ny) continue;
        acc[o] = s_ab[e] - acc[o];
        acc_d += lambda_change(acc[o], s_lam[e]);
        u[o] = s_rs[e] * acc[o];
      }
#pragma unroll
      for (int o = 0; o < RB; ++o) {
        if (i0 + o >= ny) continue;
        s_lam[l * ny + i0 + o] = acc[o];
        X.a[X.at_c(0, l, i0 + o)] = u[o];
      }
    });
    ++k;
    if ((k & 7) == 0) {
      const double tot = grid_sum(acc_d);
      acc_d = 0.0;
      bad = !isfinite(tot);
      if (bad || tot <= A.tol * 8.0 * norm) break;
    } else {
      __syncthreads();
    }
    if (s_fault) break;
  }

  // the gradients of this step: g = qbar_0 + xi(R_s lambda) / Y, wbar += R_w lambda
  if (!bad) {
    to_rows();
    rows_out([&](int e, int, T v) {
      A.gout[(size_t)X.y0 * nx + e] = s_qb[e] + v * s_iY[e];
    });
    if (A.wbar != nullptr) {
      for (int e = tid; e < ny * ncg; e += nthreads) {
        const int y = e / ncg, xl = e - y * ncg;
        const size_t at = (size_t)y * nx + X.x0 + xl;
        T rs, rw;
        ratio_grad<T, EK>(P, (int)at, s_s[xl * ny + y], rs, rw);
        A.wbar[at] += rw * s_lam[xl * ny + y];
      }
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (s_fault) atomicOr(&A.out->bad, 2);
    if (blockIdx.x == 0) {
      if (bad) atomicOr(&A.out->bad, 1);
      A.out->iters = k;
      *A.g.epoch = epoch::after(ep0, ep, epoch::of_adjoint(A.budget), s_fault);
    }
  }
}

template <typename T, int RB>
void* adj_fn_ek(int ek) {
  if (ek == EK_CROWD) return (void*)strip_adjoint_kernel<T, EK_CROWD, RB, 512>;
  if (ek == EK_ENTROPY) return (void*)strip_adjoint_kernel<T, EK_ENTROPY, RB, 512>;
  return (void*)strip_adjoint_kernel<T, EK_POWER, RB, 512>;
}
template <typename T>
void* adj_fn(int rb, int ek);
template <>
void* adj_fn<float>(int rb, int ek) { return rb == 8 ? adj_fn_ek<float, 8>(ek) : adj_fn_ek<float, 4>(ek); }
template <>
void* adj_fn<double>(int, int ek) { return adj_fn_ek<double, 1>(ek); }

}  // namespace

// Wherever the step itself runs on strips and the larger set of images still
// fits one block per SM (FP32 up to ~760 cells a side).
template <typename T>
size_t strip_adjoint_smem(const StripPlan& sp, int ek, int nx, int ny, int rx, int ry) {
  int dev = 0, smem_max = 0;
  if (sp.G == 0 || cudaGetDevice(&dev) != cudaSuccess) return 0;
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const Smem S = smem_of<T>(nx, ny, rx, ry, sp.nc, sp.nr, 1, sp.parts, kAdjRows, kAdjCols, false);
  if (S.total + 1024 > (size_t)smem_max) return 0;
  if (max_dynamic_smem(adj_fn<T>(sp.rb, ek)) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return S.total;
}

template <typename T>
cudaError_t strip_adjoint_launch(const StripPlan& sp, size_t smem, int ek, int nx, int ny, int rx,
                                 int ry, const T* taps_x, const T* taps_y, const StripAdjoint<T>& s,
                                 const ProxArgs<T>& P, unsigned long long* words,
                                 cudaStream_t st) {
  AdjArgs<T> A{strip_geo(sp, nx, ny, rx, ry, taps_x, taps_y, words), s.q, s.a, s.gin, s.gout,
               s.wbar, s.mass, s.renorm, s.tol, s.budget, s.out, s.after};
  ProxArgs<T> Pc = P;
  void* args[] = {&A, &Pc};
  return strip_coop(adj_fn<T>(sp.rb, ek), sp, smem, sp.threads, args, st);
}

#define JKO_STRIP_ADJ_INST(T)                                                                     \
  template size_t strip_adjoint_smem<T>(const StripPlan&, int, int, int, int, int);              \
  template cudaError_t strip_adjoint_launch<T>(const StripPlan&, size_t, int, int, int, int, int, \
                                               const T*, const T*, const StripAdjoint<T>&,        \
                                               const ProxArgs<T>&, unsigned long long*,           \
                                               cudaStream_t);
JKO_STRIP_ADJ_INST(float)
JKO_STRIP_ADJ_INST(double)
#undef JKO_STRIP_ADJ_INST

}  // namespace jko
