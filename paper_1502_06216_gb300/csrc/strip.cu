// strip.cu -- persistent CUDA-core form of a JKO step (FP32 / FP64, the separable
// Gaussian by taps): one cooperative launch runs the pairs of the scaling loop
// (Prop. 3.3; with several couplings Prop. prop-implementation-generic) with the
// stopping rule of Sec. 3.4 inside.
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
// images in L2 and four launches.  Steps with several couplings move their two
// or three images together: the same two exchanges a pair, the joint proxes cell
// by cell on the owned strip (attraction and two species: on the columns;
// pairwise attraction: p_1 on the rows, p_2 on the columns).  A
// five-step attraction flow at 256^2 FP32 (band 168, 195 pairs): 6774 us a kernel per pass
// (five launches a pair), 3163 us here.
//
// The exchange is strip.cuh's.  The residual of each block's rows (pairwise:
// columns) travels the same way, twice buffered by pair parity (a block may still
// be reading pair k's when pair k + 1's are written); every block adds all of
// them in one fixed order and takes the same decision.
#include <algorithm>

#include "coupled_prox.cuh"
#include "epoch.h"
#include "jko_kernels.h"
#include "strip.cuh"

namespace jko {

namespace {

using namespace strip;

constexpr int kStripMaxLine = 4096;

// What a step computes between the moves (StripStep::op): images filtered at once.
__host__ __device__ constexpr int op_images(int op) {
  return op == OP_ONE ? 1 : op == OP_PAIR ? 3 : 2;
}

template <typename T>
struct StripArgs {
  Geo g;
  const T* q;                    // the step's input (two densities: 2 N)
  const T* q2;                   // second column marginal: the attraction's target, q + N
  const T* E1;                   // e^{-sigma w} of the two densities (species, pairwise)
  const T* E2;
  T t, kappa;                    // attraction: tau; pairwise: tau alpha; scalar bound (coupled)
  int has_kappa;
  T* a[2];
  Ctrl* ctrl;
  int pairs;
  // the control block starts as `init` (fresh), the input is checked (check), p goes to out,
  // renormalised on request, the control block to record
  T* out;
  Ctrl* record;
  int fresh, check, renorm;
  unsigned long long* xfin;      // at the end: the blocks' max p / kappa and checks, 6 words each
  unsigned long long* xsum;      // and the lines' masses, 2 words each
  Ctrl init;
};

// The plain images of a block: by rows (q and the second marginal; pairwise: q_2,
// e^{-sigma w_1}, p_1) and by columns (p, then the prox fields; species: p_1, p_2, e_1,
// e_2; pairwise: q_1, e^{-sigma w_2}, p_2 and the three blurred images).
template <typename T>
__host__ __device__ inline void strip_images(int op, int ek, const ProxArgs<T>& P, int* rows,
                                             int* cols) {
  const int fields = (ek == EK_CROWD) + (P.sw != nullptr) + (P.c != nullptr) +
                     (P.kappa != nullptr) + (P.m1f != nullptr);
  *rows = op == OP_ONE ? 1 : op == OP_PAIR ? 3 : 2;
  *cols = op == OP_SPECIES ? 4 : op == OP_PAIR ? 6 : 1 + fields;
}

template <typename T, int OP, int EK, int RB, int NT>
__global__ void __launch_bounds__(NT, 1)
strip_kernel(const __grid_constant__ StripArgs<T> A, const __grid_constant__ ProxArgs<T> P) {
  constexpr int NI = op_images(OP);
  // the energy's fields as the prox reads them (one density, attraction)
  constexpr bool FIELDS = OP == OP_ONE || OP == OP_ATTRACT;
  // several couplings with b = q / Y: the step starts from b = 1 with its second half
  constexpr bool FROM_B = OP == OP_ATTRACT || OP == OP_SPECIES;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // 256-byte aligned: window() applies sw() to absolute shared addresses
  unsigned char* smem = smem_raw + (-(int)__cvta_generic_to_shared(smem_raw) & 255);
  __shared__ int s_bad, s_fault, s_dec;
  __shared__ double s_wres[NT / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nthreads = blockDim.x, nwarps = nthreads >> 5;
  const int nx = A.g.nx, ny = A.g.ny;
  int n_row, n_col;
  strip_images<T>(OP, EK, P, &n_row, &n_col);
  const bool has_mask = FIELDS && P.mask != nullptr;
  const Smem S = smem_of<T>(nx, ny, A.g.rx, A.g.ry, A.g.nc, A.g.nr, NI, A.g.parts, n_row, n_col,
                            has_mask);
  Strips<T, NI, RB> X(A.g, S, smem, &s_fault);
  auto row = [&](int k) { return (T*)(smem + S.row + k * S.row_b); };
  auto col = [&](int k) { return (T*)(smem + S.col + k * S.col_b); };
  Ctrl* ctrl = A.ctrl;
  const int ncg = X.ncg, nrg = X.nrg;
  if (A.fresh) {
    if (tid == 0 && blockIdx.x == 0) {
      *ctrl = A.init;
      __threadfence();   // before this block's words, so before any block's counts below
    }
  } else {
    const int done0 = *(volatile int*)&ctrl->done, bad0 = *(volatile int*)&ctrl->nonfinite;
    if (done0 != RUNNING || bad0) {   // the same state for every block: none waits for this one
      if (done0 == RUNNING && tid == 0 && blockIdx.x == 0) ctrl->done = NONFINITE;
      return;
    }
  }
  const int maxit = A.fresh ? A.init.max_iter : ctrl->max_iter;
  const int stall = A.fresh ? A.init.stall : ctrl->stall;
  const double tol = A.fresh ? A.init.tol : ctrl->tol;
  const unsigned ep0 = *(volatile unsigned*)A.g.epoch;
  if (tid == 0) {
    s_bad = 0;
    s_fault = 0;
    s_dec = 0;
  }

  // taps, zeroed lines, the marginals and the prox fields
  X.load_taps();
  ProxArgs<T> L = P;
  if (OP == OP_PAIR) {
    X.load_rows(A.q2, row(0));
    X.load_rows(A.E1, row(1));
    X.load_cols(A.q, col(0));
    X.load_cols(A.E2, col(1));
    for (int e = tid; e < nx * nrg; e += nthreads) row(2)[e] = T(0);
    for (int e = tid; e < ny * ncg; e += nthreads) col(2)[e] = T(0);
  } else {
    X.load_rows(A.q, row(0));
    if (NI == 2) X.load_rows(A.q2, row(1));
    for (int e = tid; e < ny * A.g.nc; e += nthreads) {
      col(0)[e] = T(0);
      if (OP == OP_SPECIES) col(1)[e] = T(0);
    }
  }
  if (OP == OP_SPECIES) {
    X.load_cols(A.E1, col(2));
    X.load_cols(A.E2, col(3));
  }
  if (FIELDS) {
    int k = 1;
    auto field = [&](const T* g) -> const T* {
      T* s = col(k++);
      X.load_cols(g, s);
      return s;
    };
    if (EK == EK_CROWD) L.E = field(P.E);
    if (P.sw != nullptr) L.sw = field(P.sw);
    if (P.c != nullptr) L.c = field(P.c);
    if (P.kappa != nullptr) L.kappa = field(P.kappa);
    if (P.m1f != nullptr) L.m1f = field(P.m1f);
    if (has_mask) {
      uint8_t* s = (uint8_t*)(smem + S.mask);
      for (int e = tid; e < ny * ncg; e += nthreads) {
        const int y = e / ncg, xl = e - y * ncg;
        s[xl * ny + y] = P.mask[(size_t)y * nx + X.x0 + xl];
      }
      L.mask = s;
    }
  }
  __syncthreads();
  // the cold start (Sec. 3.4, Prop. prop-implementation-generic): a = 1, or b = 1
  if (FROM_B) {
    for (int l = 0; l < NI * A.g.nr; ++l)
      for (int i = tid; i < nx; i += nthreads) X.b[X.at_r(0, l, i)] = T(1);
  } else {
    for (int l = 0; l < NI * A.g.nc; ++l)
      for (int i = tid; i < ny; i += nthreads) X.a[X.at_c(0, l, i)] = T(1);
  }
  __syncthreads();

  int it = 0, pair = 0, since = 0;
  double best = INFINITY;
  // warps whose threads have terms of the residual
  const int active =
      OP == OP_PAIR ? nwarps : min(nwarps, (NI * A.g.nr * ((nx + RB - 1) / RB) + 31) >> 5);
  // the block's residual (NaN where it met a non-finite scaling) to every block
  const int n_res = OP == OP_PAIR ? A.g.gc : A.g.gr;
  auto put_residual = [&](unsigned ep) {
    unsigned long long* xr = A.g.xres + (size_t)(pair & 1) * n_res * 2;
    if (wid == nwarps - 1 && (int)blockIdx.x < n_res) {   // the warp with the fewest items
      double v = lane < active ? s_wres[lane] : 0.0;   // at most 16 warps
#pragma unroll
      for (int o = 8; o > 0; o >>= 1)
        if (o < active) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) put_elem(xr + 2 * blockIdx.x, s_bad ? (double)NAN : v, ep);
    }
  };
  // the stop rule (Sec. 3.4) on the sum over the blocks' residuals of pair `of`, put with ep
  auto decide = [&](int of, unsigned ep) {
    const double v = gather_sum(A.g.xres + (size_t)(of & 1) * n_res * 2, n_res, ep, &s_fault);
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
  };
  for (; pair < A.pairs; ++pair) {
    const unsigned ep = ep0 + 1u + (unsigned)pair;
    int bad = 0;
    if (!FROM_B || pair > 0) {
      // columns: T = K_y a
      X.filter_send_cols(ep);
      if (OP == OP_PAIR && pair > 0 && wid == nwarps - 1) decide(pair - 1, ep - 1u);
      X.receive_rows(ep);
      __syncthreads();
      if (OP == OP_PAIR) {
        if (s_dec || s_fault) break;
        // rows: s_m = xi b_m, then the common row marginal p_1 of couplings 1 and 3 and
        // the fixed rows q_2 of coupling 2
        X.filter_rows_to(X.r2, X.b);
        __syncthreads();
        for (int l = 0; l < nrg; ++l)
          for (int i = tid; i < nx; i += nthreads) {
            const int e = l * nx + i;
            T* b1 = X.b + X.at_r(0, l, i);
            T* b2 = X.b + X.at_r(1, l, i);
            T* b3 = X.b + X.at_r(2, l, i);
            const T x1 = *b1, x3 = *b3;
            const T pm = pairwise_marginal<T>(x1, x3, A.t, row(1)[e], A.kappa, A.has_kappa);
            const T r1 = safe_ratio<T>(pm, x1), r3 = safe_ratio<T>(pm, x3);
            const T r2 = b_update<T>(row(0)[e], *b2);
            bad |= !dev_finite(r1) || !dev_finite(r2) || !dev_finite(r3) || !dev_finite(pm);
            *b1 = r1;
            *b2 = r2;
            *b3 = r3;
            row(2)[e] = pm;
          }
        if (bad) s_bad = 1;
      } else {
        // rows: Y = T K_x, the residual |b_old Y - q| and b = q / Y
        const bool have_prev = it > 0;
        // an item's terms in the working precision, as a thread of filter_pass adds its own, and
        // in FP64 from there on
        double sum = 0.0;
        X.filter_rows(X.r2, [&](int m, int l, int i0, T (&acc)[RB]) {
          T res = T(0);
          X.each(acc, i0, nx, [&](int i, T v) {
            const T qv = row(m)[l * nx + i];
            T* bp = X.b + X.at_r(m, l, i);
            if (have_prev) res += abs_residual<T>(*bp, v, qv);
            const T bn = b_update<T>(qv, v);
            bad |= !dev_finite(bn);
            *bp = bn;
          });
          sum += (double)res;
        });
        // warps without items have nothing to add (an FP64 tree takes ~450 cycles)
        if (wid < active) {
          const double wres = warp_sum(sum);
          if (lane == 0) s_wres[wid] = wres;
        }
        if (bad) s_bad = 1;
      }
      __syncthreads();
      if (OP != OP_PAIR) put_residual(ep);
    }
    // U = b K_x, rows -> columns
    X.filter_send_rows(ep);
    if (OP != OP_PAIR && (!FROM_B || pair > 0) && wid == nwarps - 1) decide(pair, ep);
    X.receive_cols(ep);
    __syncthreads();
    if (s_dec || s_fault) break;
    bad = 0;
    if (OP == OP_ONE) {
      // columns: s = K_y U, a = Prox(s) / s, p = a s
      T* s_p = col(0);
      X.filter_cols(X.c2, [&](int, int l, int i0, T (&acc)[RB]) {
        X.each(acc, i0, ny, [&](int i, T v) {
          const int idx = l * ny + i;
          const T a = prox_ratio<T, EK>(L, idx, v);
          bad |= !dev_finite(a);
          X.a[X.at_c(0, l, i)] = a;
          s_p[idx] = a * v;
        });
      });
    } else if (OP == OP_PAIR) {
      // columns: y_m = xi a_m; the residual against the column constraints, p_2 = b_2 y_2,
      // then the common column marginal of couplings 2 and 3 and b_1 = q_1 / y_1
      X.filter_cols(X.c2, [&](int m, int l, int i0, T (&acc)[RB]) {
        T* v = col(3 + m) + l * ny + i0;
#pragma unroll
        for (int o = 0; o < RB; ++o)
          if (i0 + o < ny) v[o] = acc[o];
      });
      __syncthreads();
      double res = 0.0;
      for (int l = 0; l < ncg; ++l)
        for (int i = tid; i < ny; i += nthreads) {
          const int e = l * ny + i;
          const T v1 = col(3)[e], v2 = col(4)[e], v3 = col(5)[e], qq = col(0)[e];
          T* b1 = X.a + X.at_c(0, l, i);
          T* b2 = X.a + X.at_c(1, l, i);
          T* b3 = X.a + X.at_c(2, l, i);
          const T c2 = *b2 * v2;
          res += (double)abs_residual<T>(*b1, v1, qq) + (double)fabs(c2 - *b3 * v3);
          col(2)[e] = c2;
          const T pm = pairwise_marginal<T>(v2, v3, A.t, col(1)[e], A.kappa, A.has_kappa);
          const T r1 = b_update<T>(qq, v1);
          const T r2 = safe_ratio<T>(pm, v2), r3 = safe_ratio<T>(pm, v3);
          bad |= !dev_finite(r1) || !dev_finite(r2) || !dev_finite(r3);
          *b1 = r1;
          *b2 = r2;
          *b3 = r3;
        }
      res = warp_sum(res);
      if (lane == 0) s_wres[wid] = res;
    } else {
      // columns: s_m = K_y U_m, then the joint prox
      X.filter_cols_to(X.c2, X.a);
      __syncthreads();
      const T w1 = T(1) / (T(1) + A.t), w2 = A.t / (T(1) + A.t);
      for (int l = 0; l < ncg; ++l)
        for (int i = tid; i < ny; i += nthreads) {
          const int e = l * ny + i;
          T* a1 = X.a + X.at_c(0, l, i);
          T* a2 = X.a + X.at_c(1, l, i);
          T r1, r2, p1, p2 = T(0);
          if (OP == OP_ATTRACT) {
            attraction_cell<T, EK>(L, e, *a1, *a2, w1, w2, r1, r2, p1);
            bad |= !dev_finite(r1) || !dev_finite(r2) || !dev_finite(p1);
          } else {
            species_cell<T>(*a1, *a2, col(2)[e], col(3)[e], A.kappa, A.has_kappa, r1, r2, p1, p2);
            bad |= !dev_finite(p1) || !dev_finite(p2);
            col(1)[e] = p2;
          }
          *a1 = r1;
          *a2 = r2;
          col(0)[e] = p1;
        }
    }
    if (bad) s_bad = 1;
    ++it;
    __syncthreads();
    if (OP == OP_PAIR) put_residual(ep);
  }

  // the final a, and p of the pair the last residual belongs to: its mass and max p / kappa
  // first (as finalize_reduce_kernel) and the input's checks (as validate_kernel),
  // exchanged like the residuals, then p times 1 / mass (as finalize_write_kernel)
  const size_t N = (size_t)nx * ny;
  double inv = 1.0;
  bool scale = false, keep = true;
  {
    __shared__ double s_fin[3][NT / 32], s_mass;
    const unsigned epf = ep0 + 2u + (unsigned)pair;
    // p line by line in one order (lanes, then their tree), so that the mass has the same
    // bits however the lines are split over blocks
    T mx = T(0);
    auto line_sum = [&](const T* p, int n, const T* kap, int at) {
      double sum = 0.0;
      for (int i = lane; i < n; i += 32) {
        sum += (double)p[i];
        if (P.has_kappa) {
          const T r = p[i] / (kap != nullptr ? kap[i] : P.kappa_s);
          mx = r > mx ? r : mx;
        }
      }
      sum = warp_sum(sum);
      if (lane == 0) put_elem(A.xsum + 2 * (size_t)at, sum, epf);
    };
    for (int l = wid; l < ncg; l += nwarps) {
      const T* kap = FIELDS && P.kappa != nullptr ? L.kappa + l * ny : nullptr;
      line_sum(col(OP == OP_PAIR ? 2 : 0) + l * ny, ny, kap, X.x0 + l);
      if (OP == OP_SPECIES) line_sum(col(1) + l * ny, ny, kap, nx + X.x0 + l);
    }
    if (OP == OP_PAIR)
      for (int l = wid; l < nrg; l += nwarps) line_sum(row(2) + l * nx, nx, nullptr, nx + X.y0 + l);
    double qsum = 0.0;
    unsigned n_neg = 0, n_bad = 0, n_over = 0, n_msk = 0;
    auto check_q = [&](T v, size_t at) {
      if (!isfinite(v)) {
        ++n_bad;
        return;
      }
      qsum += (double)v;
      if (v < T(0)) ++n_neg;
      if (P.has_kappa && (double)v > (double)(P.kappa ? P.kappa[at] : P.kappa_s) * (1.0 + 1e-2))
        ++n_over;
      if (P.mask != nullptr && P.mask[at] && v != T(0)) ++n_msk;
    };
    if (A.check) {
      for (int e = tid; e < nx * nrg; e += nthreads) {
        check_q(row(0)[e], (size_t)X.y0 * nx + e);
        if (OP == OP_SPECIES) check_q(row(1)[e], (size_t)X.y0 * nx + e);
      }
      if (OP == OP_PAIR)   // the first density by columns
        for (int e = tid; e < ny * ncg; e += nthreads)
          check_q(col(0)[e], (size_t)(e % ny) * nx + X.x0 + e / ny);
      if (n_bad) atomicAdd(&ctrl->q_bad, (unsigned long long)n_bad);
      if (n_neg) atomicAdd(&ctrl->q_neg, (unsigned long long)n_neg);
      if (n_over) atomicAdd(&ctrl->q_over, (unsigned long long)n_over);
      if (n_msk) atomicAdd(&ctrl->q_masked, (unsigned long long)n_msk);
      qsum = warp_sum(qsum);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const bool viol = __any_sync(0xffffffffu, (n_neg | n_bad | n_over | n_msk) != 0);
    if (lane == 0) {
      s_fin[0][wid] = (double)mx;
      s_fin[1][wid] = qsum;
      s_fin[2][wid] = viol ? 1.0 : 0.0;
    }
    __syncthreads();
    if (wid == 1) {
      const int n = OP == OP_SPECIES ? 2 * nx : OP == OP_PAIR ? nx + ny : nx;
      const double mass = gather_sum(A.xsum, n, epf, &s_fault);
      if (lane == 0) s_mass = mass;
    }
    if (wid == 0) {
      double v[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] = lane < nwarps ? s_fin[k][lane] : 0.0;
      auto all = [&]() {
        v[1] = warp_sum(v[1]);
        v[2] = warp_sum(v[2]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[0] = fmax(v[0], __shfl_xor_sync(0xffffffffu, v[0], o));
      };
      all();
      // a block that gave up a wait says so by a negative count
      if (s_fault) v[2] = -1e9;
      if (lane < 3)
        put_elem(A.xfin + 6 * (size_t)blockIdx.x + 2 * lane, lane == 0 ? v[0] : lane == 1 ? v[1] : v[2],
                 epf);
      v[0] = v[1] = v[2] = 0.0;
      for (int g = lane; g < (int)gridDim.x; g += 32) {
        const unsigned long long* w = A.xfin + 6 * (size_t)g;
        unsigned long long lo[3], hi[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) get_words(w + 2 * k, lo[k], hi[k]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if (!wait_pair(w + 2 * k, epf, lo[k], hi[k], &s_fault)) s_fault = 1;
          const double d = words_double(lo[k], hi[k]);
          v[k] = k == 0 ? fmax(v[k], d) : v[k] + d;
        }
      }
      all();
      if (lane < 3) s_fin[lane][0] = lane == 0 ? v[0] : lane == 1 ? v[1] : v[2];
    }
    __syncthreads();
    const double mass = s_mass;
    if (s_fin[2][0] < 0.0 && tid == 0) s_fault = 1;
    scale = A.renorm && mass > 0.0 && isfinite(mass);
    inv = scale ? 1.0 / mass : 1.0;
    // a step whose input failed its checks leaves the output untouched
    keep = !A.check || (s_fin[2][0] == 0.0 && fabs(s_fin[1][0] - 1.0) <= 1e-3);
    if (tid == 0 && blockIdx.x == 0) {
      ctrl->mass = mass;
      if (s_fin[0][0] > 0.0) ctrl->maxpk_bits = (unsigned long long)__double_as_longlong(s_fin[0][0]);
      ctrl->q_sum = s_fin[1][0];
      if (!isfinite(mass)) atomicOr(&ctrl->nonfinite, 1);
      ++pair;   // the epoch of this exchange
    }
  }
  auto put_p = [&](size_t at, T v) {
    if (keep) A.out[at] = scale ? (T)((double)v * inv) : v;
  };
  for (int e = tid; e < ny * ncg; e += nthreads) {
    const int y = e / ncg, xl = e - y * ncg;
    const size_t at = (size_t)y * nx + X.x0 + xl;
    if (OP == OP_PAIR) {
      put_p(N + at, col(2)[xl * ny + y]);
    } else {
#pragma unroll
      for (int m = 0; m < (NI < 2 ? NI : 2); ++m) A.a[m][at] = X.a[X.at_c(m, xl, y)];
      put_p(at, col(0)[xl * ny + y]);
      if (OP == OP_SPECIES) put_p(N + at, col(1)[xl * ny + y]);
    }
  }
  if (OP == OP_PAIR)
    for (int e = tid; e < nx * nrg; e += nthreads) put_p((size_t)X.y0 * nx + e, row(2)[e]);
  if (tid == 0) {
    if (s_fault) atomicOr(&ctrl->nonfinite, 2);
    if (blockIdx.x == 0) {
      ctrl->it = it;
      *A.g.epoch = epoch::after(ep0, ep0 + 1u + (unsigned)pair, epoch::of_strip(A.pairs), s_fault);
      if (A.record != nullptr) *A.record = *ctrl;
    }
  }
}

// ---- host ----
template <typename T, int OP, int RB, int NT>
void* strip_fn_ek(int ek) {
  if (OP == OP_SPECIES || OP == OP_PAIR || ek == EK_CROWD)
    return (void*)strip_kernel<T, OP, EK_CROWD, RB, NT>;
  constexpr int O = OP == OP_SPECIES || OP == OP_PAIR ? OP_ONE : OP;
  if (ek == EK_ENTROPY) return (void*)strip_kernel<T, O, EK_ENTROPY, RB, NT>;
  return (void*)strip_kernel<T, O, EK_POWER, RB, NT>;
}
template <typename T, int RB, int NT>
void* strip_fn_op(int op, int ek) {
  switch (op) {
    case OP_ONE: return strip_fn_ek<T, OP_ONE, RB, NT>(ek);
    case OP_ATTRACT: return strip_fn_ek<T, OP_ATTRACT, RB, NT>(ek);
    case OP_SPECIES: return strip_fn_ek<T, OP_SPECIES, RB, NT>(ek);
    default: return strip_fn_ek<T, OP_PAIR, RB, NT>(ek);
  }
}
template <typename T>
void* strip_fn(int rb, int op, int ek);
template <>
void* strip_fn<float>(int rb, int op, int ek) {
  return rb == 8 ? strip_fn_op<float, 8, 512>(op, ek) : strip_fn_op<float, 4, 512>(op, ek);
}
template <>
void* strip_fn<double>(int, int op, int ek) { return strip_fn_op<double, 1, 512>(op, ek); }

}  // namespace

// The rule for the persistent form, on the grid, the band and the precision.
// Both sides measured on a GB300 (us a pair, this form / a kernel per pass, 40 pairs a
// step): crowd FP32 64^2 5.8 / 16.5, 128^2 6.4 / 17.9, 256^2 8.5 / 22.3, 512^2 22.9 / 39.1, 600 x 200
// 15.6 / 29.7, 800 x 64 12.7 / 27.4, 700^2 51 / 80, 1024^2 63 / 79; FP64 64^2 10.2 / 57.4, 128^2
// 23.7 / 96.4, 256^2 140 / 170, 300^2 215 / 376.  Attraction 256^2 FP32 15.5 / 32.4, FP64
// 287 / 343; two species and pairwise alike.  FP64 512^2 (four lines a block) was
// 1253 / 1124: bound by its pipe, whole lines per block (4 against 3.4 on average)
// cost what the launches save, so FP64 takes up to two
// lines a block.  FP32: wherever the strips fit the shared memory of one block
// per SM (about 1060 cells a side).
// Long thin grids, whose short side has too few lines for the blocks (the busiest block has
// more than four times its share of the cells), keep the kernels per pass unless a block's
// lines are little work (in multiply-adds: 5e5, FP64 4e4).  Up to there this form won
// everywhere it was timed (FP32 600 x 8 9.5 / 23.9, 2048 x 32 with a narrow kernel 2.2 / 3.3; FP64
// 152 x 4 19.7 / 62.8).  The line is a cautious one: beyond it the kernels per pass won only where
// lines of 3500 cells and more meet a narrow kernel (FP32 4096 x 16, gamma 1e-4: 47.6 / 38.9;
// 3500 x 24, 5e-5: 33.7 / 31.4) and lost elsewhere (FP32 1000 x 16 14.7 / 29.2, 2000 x 16 36.5 / 178,
// gamma 1e-3; FP64 300 x 8 33.8 / 65.7).
template <typename T>
StripPlan strip_plan(int nx, int ny, int rx, int ry, int op, int ek, const ProxArgs<T>& P,
                     int max_blocks, int parts) {
  StripPlan sp;
  const int ni = op_images(op);
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
  // (256^2: 8.8 us a pair with four, 11.4 with eight; 1024^2 72 and 64, both before the epilogues
  // were rolled); FP64: one
  auto items = [&](int rb) {
    return ni * std::max(sp.nc * ceil_div(ny, rb), sp.nr * ceil_div(nx, rb));
  };
  sp.rb = sizeof(T) == 8 ? 1 : items(8) >= 256 ? 8 : 4;
  // FP64: parts of an output's taps that give every scheduler two warps where the outputs
  // do not (us a pair over whole flows, one part / now: 64^2 19 / 13.3, 128^2 30 / 26)
  if (max_blocks > 0) sp.parts = parts;
  else while (sizeof(T) == 8 && sp.parts < 8 && items(1) * sp.parts < 256) sp.parts *= 2;
  // a warp more than the items fill: it adds and sends the residual while the others filter
  // (not in a batch, whose flows' blocks share the SMs' registers)
  sp.threads = std::min(512, std::max(256, ceil_div(items(sp.rb) * sp.parts, 32) * 32 +
                                               (max_blocks > 0 ? 0 : 32)));
  int rows = 0, cols = 0;
  strip_images<T>(op, ek, P, &rows, &cols);
  const Smem S = smem_of<T>(nx, ny, rx, ry, sp.nc, sp.nr, ni, sp.parts, rows, cols, P.mask != nullptr);
  sp.smem = S.total;
  if (S.total + 1024 > (size_t)smem_max) return StripPlan{};
  void* fn = strip_fn<T>(sp.rb, op, ek);
  int per_sm = 0;
  if (max_dynamic_smem(fn) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, sp.threads, S.total) !=
          cudaSuccess ||
      per_sm * sms < sp.G) {
    cudaGetLastError();
    return StripPlan{};
  }
  const size_t kw = sizeof(T) / 4;
  const size_t r1 = ((size_t)ni * nx * sp.nr * kw + 1) & ~(size_t)1;
  const size_t r2 = ((size_t)ni * ny * sp.nc * kw + 1) & ~(size_t)1;
  sp.x1_words = r1 * ceil_div(ny, sp.nr);
  sp.x2_words = r2 * ceil_div(nx, sp.nc);
  sp.words = sp.x1_words + sp.x2_words + 10 * (size_t)sp.G + 4 * (size_t)std::max(nx, ny) + 2;
  return sp;
}

// Taps of each of an output's parts, which cover the longest range of a line.
static int part_len(int n, int r, int parts) { return ceil_div(std::min(2 * r + 1, n), parts); }

strip::Geo strip_geo(const StripPlan& sp, int nx, int ny, int rx, int ry, const void* taps_x,
                     const void* taps_y, unsigned long long* words) {
  return Geo{nx, ny, rx, ry, sp.nc, sp.nr, ceil_div(ny, sp.nr), ceil_div(nx, sp.nc),
             magic(sp.nc), magic(sp.nr), sp.parts, part_len(ny, ry, sp.parts),
             part_len(nx, rx, sp.parts), taps_x, taps_y, words, words + sp.x1_words,
             words + sp.x1_words + sp.x2_words, (unsigned*)(words + sp.words - 2)};
}

cudaError_t strip_coop(void* fn, const StripPlan& sp, size_t smem, int threads, void** args,
                       cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)sp.G);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

template <typename T>
cudaError_t strip_launch(const StripPlan& sp, int nx, int ny, int rx, int ry, const T* taps_x,
                         const T* taps_y, const StripStep<T>& s, const ProxArgs<T>& P, Ctrl* ctrl,
                         unsigned long long* words, int pairs, cudaStream_t st) {
  StripArgs<T> A{strip_geo(sp, nx, ny, rx, ry, taps_x, taps_y, words), s.q, s.q2, s.E1, s.E2,
                 (T)s.t, P.kappa_s, P.has_kappa, {s.a, s.a2}, ctrl, pairs, s.out, s.record,
                 s.init != nullptr, s.check, s.renorm,
                 words + sp.x1_words + sp.x2_words + 4 * (size_t)sp.G,
                 words + sp.x1_words + sp.x2_words + 10 * (size_t)sp.G,
                 s.init ? *s.init : Ctrl{}};
  ProxArgs<T> Pc = P;
  void* args[] = {&A, &Pc};
  return strip_coop(strip_fn<T>(sp.rb, s.op, s.ek), sp, sp.smem, sp.threads, args, st);
}

#define JKO_STRIP_INST(T)                                                                        \
  template StripPlan strip_plan<T>(int, int, int, int, int, int, const ProxArgs<T>&, int, int); \
  template cudaError_t strip_launch<T>(const StripPlan&, int, int, int, int, const T*, const T*, \
                                       const StripStep<T>&, const ProxArgs<T>&, Ctrl*,           \
                                       unsigned long long*, int, cudaStream_t);
JKO_STRIP_INST(float)
JKO_STRIP_INST(double)
#undef JKO_STRIP_INST

}  // namespace jko
