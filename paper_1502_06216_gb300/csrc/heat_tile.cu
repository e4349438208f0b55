// heat_tile.cu -- the persistent form of a step with the heat kernel (heat.cu) on
// resident tiles: one block per tile of the grid keeps v, the Clenshaw iterates
// b_{k+1}, b_{k+2} and the step's images in shared memory for the whole step, with
// a halo of H cells.  A phase runs up to H Clenshaw steps, each on the tile and a
// halo one cell narrower than the one before (recomputed by the neighbours), then
// the tiles exchange the H cells inside their edges: every value travels as 8-byte
// words {32 bits, epoch} (strip.cuh), polled by their readers, so there is no grid
// barrier, and the interior never leaves the SM.  The words are twice buffered by
// epoch parity: a block writes exchange e + 2 only after it has every
// neighbour's e + 1, which they wrote after reading e.  So every block that reads a block's
// words has to be one it waits for: the blocks with a cell within H cells of its tile,
// whatever the obstacles are (heat_geom.h).  The arithmetic of a cell and the stop rule are
// those of heat.cu's kernels, and the residual is added in their order (in FP64, by groups of
// 16 x 8 cells: the cells' terms travel to the block of their group, its sums to every block),
// so the iterates, the pair counts and the residuals have the same bits.
//
// Bound by the exchange and by the FP64 latency of its steps (five operations a cell, four
// deep, on a pipe of half a lane a cycle and scheduler): 100^2, 150 tiles, degree 54, a
// 33-pair step: 5.69 ms on heat.cu's blocks with a grid barrier a phase, 4.36 on tiles,
// 3.01 with the five-operation step and each thread's cells kept in registers.  H = 4: with
// the longer step 7.0, 5.1, 4.5, 4.4, 4.4 and 4.6 ms for H = 1 to 6 (exchanges against
// halo work).
#include <algorithm>

#include "epoch.h"
#include "heat_cell.cuh"
#include "heat_geom.h"
#include "jko_kernels.h"
#include "strip.cuh"

namespace jko {

namespace {

using namespace strip;

constexpr int HTT = 512;   // threads at most: work warps and one that takes the decision
using heat_geom::FREE;
using heat_geom::H;

template <typename T>
struct HeatTileArgs {
  int nx, ny, tw, th, ntx, D;
  int gx, ng;                // groups along x, and all of them
  double ax, ay;
  const double* coef;
  const uint8_t* mask;
  const T* q;
  T* a;
  T* p;
  Ctrl* ctrl;
  unsigned long long* xb;    // iterates: [2][cells][4]
  unsigned long long* xv;    // v: [2][cells][2]
  unsigned long long* xt;    // terms of the residual, an element a cell
  unsigned long long* xres;  // its sums over groups of HBX x HBY cells: [2][ng][2]
  unsigned* epoch;
  int pairs;
};

// A cell's term of the residual (its word or words), polled until it carries epoch ep.
__device__ __forceinline__ void load_term(const unsigned long long* w, unsigned long long& x,
                                          unsigned long long&, float) {
  x = get_word(w);
}
__device__ __forceinline__ void load_term(const unsigned long long* w, unsigned long long& x,
                                          unsigned long long& y, double) {
  get_words(w, x, y);
}
__device__ __forceinline__ double wait_term(const unsigned long long* w, unsigned ep,
                                            unsigned long long x, unsigned long long, float,
                                            int* fault) {
  for (unsigned i = 0; (unsigned)(x >> 32) != ep; ++i) {
    if (i >= kSpin || *(volatile int*)fault) {
      *fault = 1;
      break;
    }
    x = get_word(w);
  }
  return (double)__uint_as_float((unsigned)x);
}
__device__ __forceinline__ double wait_term(const unsigned long long* w, unsigned ep,
                                            unsigned long long x, unsigned long long y, double,
                                            int* fault) {
  if (!wait_pair(w, ep, x, y, fault)) *fault = 1;
  return words_double(x, y);
}

// The residual's terms over group g of HBX x HBY cells, in FP64 and in the order in which
// heat_bupdate's block of these cells adds them (block_sum: 32 cells a warp, then the warps).
// One warp; every lane gets it.
template <typename T>
__device__ __forceinline__ double group_sum(const HeatTileArgs<T>& A, int g, int lane, unsigned ep,
                                            int* fault) {
  constexpr int W = HBX * HBY / 32;   // warps of that block
  static_assert(W == 4 && 32 % HBX == 0, "the order below");
  const int gy = g / A.gx, xx = (g - gy * A.gx) * HBX + (lane & (HBX - 1));
  unsigned long long x[W], y[W];
  double t[W];
  auto at = [&](int k) -> const unsigned long long* {
    const int yy = gy * HBY + k * (32 / HBX) + lane / HBX;
    return xx < A.nx && yy < A.ny ? A.xt + kWords<T> * ((size_t)yy * A.nx + xx) : nullptr;
  };
#pragma unroll
  for (int k = 0; k < W; ++k)
    if (at(k) != nullptr) load_term(at(k), x[k], y[k], T(0));
#pragma unroll
  for (int k = 0; k < W; ++k)
    t[k] = warp_sum(at(k) != nullptr ? wait_term(at(k), ep, x[k], y[k], T(0), fault) : 0.0);
  return (t[0] + t[2]) + (t[1] + t[3]);
}

template <typename T, int EK>
__global__ void __launch_bounds__(HTT)
heat_tile_kernel(const __grid_constant__ HeatTileArgs<T> A, const __grid_constant__ ProxArgs<T> P) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_bad, s_fault, s_dec;
  const int tid = threadIdx.x, lane = tid & 31;
  const int nwork = blockDim.x - 32;   // the last warp decides
  const bool work = tid < nwork;
  Ctrl* ctrl = A.ctrl;
  const int done0 = *(volatile int*)&ctrl->done, bad0 = *(volatile int*)&ctrl->nonfinite;
  if (done0 != RUNNING || bad0) {   // the same state for every block: none waits for this one
    if (done0 == RUNNING && tid == 0 && blockIdx.x == 0) ctrl->done = NONFINITE;
    return;
  }
  const int maxit = ctrl->max_iter, stall = ctrl->stall;
  const double tol = ctrl->tol;
  const unsigned ep0 = *(volatile unsigned*)A.epoch;
  unsigned ep = ep0;
  const int nx = A.nx, ny = A.ny;
  const size_t N = (size_t)nx * ny;
  const heat_geom::Tile tile = heat_geom::tile_of(blockIdx.x, A.tw, A.th, A.ntx, nx, ny);
  const int x0 = tile.x0, y0 = tile.y0, w = tile.w, h = tile.h;
  const int SX = A.tw + 2 * H, box = SX * (A.th + 2 * H);
  double* sv = (double*)smem;
  double* cur1 = sv + box;
  double* cur2 = cur1 + box;
  T* s_b = (T*)(cur2 + box);
  T* s_q = s_b + A.tw * A.th;
  T* s_p = s_q + A.tw * A.th;
  T* s_a = s_p + A.tw * A.th;
  uint8_t* s_nb = (uint8_t*)(s_a + A.tw * A.th);
  if (tid == 0) {
    s_bad = 0;
    s_fault = 0;
    s_dec = 0;
  }
  // the cells' flags; v = a = 1 (Sec. 3.4)
  for (int c = tid; c < box; c += blockDim.x) {
    const int ey = c / SX, ex = c - ey * SX, x = x0 + ex - H, y = y0 + ey - H;
    const int f = heat_geom::cell_flags(x, y, nx, ny, A.mask);
    s_nb[c] = (uint8_t)f;
    sv[c] = f & FREE ? 1.0 : 0.0;
    cur1[c] = cur2[c] = 0.0;
  }
  for (int c = tid; c < w * h; c += blockDim.x) {
    const int y = c / w, x = c - y * w;
    s_q[c] = A.q[(size_t)(y0 + y) * nx + x0 + x];
    s_a[c] = T(1);
    s_b[c] = s_p[c] = T(0);
  }
  __syncthreads();
  const int ring = heat_geom::ring_cells(tile);
  const float inv_bx = 1.0f / (float)(w + 2 * H);
  // cell i of the halo ring: its place in the box and in the grid, -1 outside the grid
  auto ring_cell = [&](int i, int& c) -> int {
    int ex, ey;
    heat_geom::ring_place(i, tile, inv_bx, ex, ey);
    c = ey * SX + ex;
    return heat_geom::awaited(s_nb[c]) ? (y0 + ey - H) * nx + x0 + ex - H : -1;
  };

  // the cell a work thread takes in a step on the tile and an e-cell halo, where every
  // step has a thread per cell (else the steps loop over cells)
  const bool one = (w + 2 * (H - 1)) * (h + 2 * (H - 1)) <= nwork;
  int c_of[H];
#pragma unroll
  for (int e = 0; e < H; ++e) {
    const int rx = w + 2 * e, yy = quot(tid, 1.0f / (float)rx), xx = tid - yy * rx;
    c_of[e] = work && one && yy < h + 2 * e ? (H - e + yy) * SX + H - e + xx : -1;
  }

  int it = 0, pair = 0, since = 0;
  double best = INFINITY;
  bool run = true;
  for (; pair < A.pairs && run; ++pair) {
    for (int app = 0; app < 2; ++app) {
      // v on the halo; meanwhile the last warp takes the stop decision (Sec. 3.4) on the
      // b-update's residuals
      ++ep;
      if (work) {
        unsigned long long* xv = A.xv + (size_t)(ep & 1) * N * 2;
        const float inv_w = 1.0f / (float)w;
        for (int i = tid; i < w * h; i += nwork) {
          const int y = quot(i, inv_w), x = i - y * w, c = (y + H) * SX + x + H;
          if (heat_geom::sent(x, y, tile))
            put_elem(xv + 2 * ((size_t)(y0 + y) * nx + x0 + x), sv[c], ep);
        }
        for (int i = tid; i < ring; i += nwork) {
          int c;
          const int g = ring_cell(i, c);
          if (g < 0) continue;
          unsigned long long lo, hi;
          get_words(xv + 2 * (size_t)g, lo, hi);
          if (!wait_pair(xv + 2 * (size_t)g, ep, lo, hi, &s_fault)) s_fault = 1;
          sv[c] = words_double(lo, hi);
        }
      } else if (app == 1) {
        unsigned long long* xr = A.xres + (size_t)(pair & 1) * A.ng * 2;
        for (int g = blockIdx.x; g < A.ng; g += gridDim.x) {
          const double mine = group_sum<T>(A, g, lane, ep, &s_fault);
          if (lane == 0) put_elem(xr + 2 * g, mine, ep);
        }
        const double v = gather_sum(xr, A.ng, ep, &s_fault);
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
      __syncthreads();
      if (s_dec || s_fault) {
        run = false;
        break;
      }
      // the first iterates b_D = c_D v, b_{D+1} = 0
      const double cD = __ldg(A.coef + A.D);
      for (int c = tid; c < box; c += blockDim.x) {
        cur1[c] = wscale(cD, sv[c]);
        cur2[c] = 0.0;
      }
      __syncthreads();
      int bad = 0;
      const bool have_prev = app == 0 && it > 0;
      int ns = A.D % H == 0 ? H : A.D % H;
      double v_of[H];
#pragma unroll
      for (int e = 0; e < H; ++e) v_of[e] = c_of[e] >= 0 ? sv[c_of[e]] : 0.0;
      // step kk at cell c
      auto value = [&](int c, int kk, double ck, double v) -> double {
        const double s = kk == 0 ? 0.5 : 1.0;
        const int f = s_nb[c];
        const double bc = cur1[c], b2 = cur2[c];
        const double bl = cur1[c - 1], br = cur1[c + 1], bu = cur1[c - SX], bd = cur1[c + SX];
        const double r = cl_value(ck, v, b2, s * A.ax, s * A.ay, f & heat_geom::LEFT ? bl : bc,
                                  f & heat_geom::RIGHT ? br : bc, f & heat_geom::UP ? bu : bc,
                                  f & heat_geom::DOWN ? bd : bc);
        return f & FREE ? r : 0.0;
      };
      // the last step of a phase at cell i = (x, y) of the tile: to the neighbours, or closed
      // into the b-update or the prox
      auto finish = [&](int i, int x, int y, int c, int kk, double r) {
        const bool f = s_nb[c] & FREE;
        if (kk > 0) {
          const double bc = cur1[c];
          cur2[c] = r;
          if (heat_geom::sent(x, y, tile)) {
            unsigned long long* x4 = A.xb + (size_t)((ep + 1) & 1) * N * 4 +
                                     4 * ((size_t)(y0 + y) * nx + x0 + x);
            put_elem(x4, r, ep + 1);
            put_elem(x4 + 2, bc, ep + 1);
          }
          return;
        }
        const T yv = close_out<T>(r);
        if (app == 0) {
          const T qi = s_q[i];
          const T res = have_prev ? abs_residual<T>(s_b[i], yv, qi) : T(0);
          const T bn = b_update<T>(qi, yv);
          const bool inf = !dev_finite(bn);
          bad |= inf;
          s_b[i] = bn;
          // (NaN where the block has met a non-finite scaling)
          put_elem(A.xt + kWords<T> * ((size_t)(y0 + y) * nx + x0 + x), inf || s_bad ? (T)NAN : res,
                   ep + 1);
          sv[c] = f ? (double)bn : 0.0;
        } else {
          const T ai = prox_ratio<T, EK>(P, (y0 + y) * nx + x0 + x, yv);
          bad |= !dev_finite(ai);
          sv[c] = f ? (double)ai : 0.0;
          s_a[i] = ai;
          s_p[i] = ai * yv;
        }
      };
      auto swap = [&]() {
        double* t = cur2;
        cur2 = cur1;
        cur1 = t;
      };
      const float inv_w = 1.0f / (float)w;
      for (int k = A.D - 1; k >= 0;) {
        if (one) {
          double ck[H];
#pragma unroll
          for (int e = 0; e < H; ++e) ck[e] = e < ns ? __ldg(A.coef + (k - (ns - 1 - e))) : 0.0;
#pragma unroll
          for (int e = H - 1; e >= 0; --e) {
            if (e >= ns) continue;
            const int kk = k - (ns - 1 - e), c = c_of[e];
            if (c >= 0) {
              const double r = value(c, kk, ck[e], v_of[e]);
              if (e > 0) {
                cur2[c] = r;
              } else {
                const int y = quot(tid, inv_w);
                finish(tid, tid - y * w, y, c, kk, r);
              }
            }
            swap();
            if (e > 0) __syncthreads();
          }
        } else {
          for (int e = ns - 1; e >= 0; --e) {
            const int kk = k - (ns - 1 - e);
            const double ck = __ldg(A.coef + kk);
            const int rx = w + 2 * e, cells = rx * (h + 2 * e);
            const float inv = 1.0f / (float)rx;
            for (int i = work ? tid : cells; i < cells; i += nwork) {
              const int yy = quot(i, inv), xx = i - yy * rx;
              const int c = (H - e + yy) * SX + H - e + xx;
              const double r = value(c, kk, ck, sv[c]);
              if (e > 0) cur2[c] = r;
              else finish(i, xx, yy, c, kk, r);
            }
            swap();
            if (e > 0) __syncthreads();
          }
        }
        k -= ns;
        ns = H;
        if (k < 0) break;
        // the neighbours' newest iterate and the one before, on the halo (the loads in
        // flight while the block finishes its step)
        ++ep;
        unsigned long long* xb = A.xb + (size_t)(ep & 1) * N * 4;
        constexpr int UN = 2;
        unsigned long long q0[UN], q1[UN], q2[UN], q3[UN];
        int cc[UN], gg[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          const int i = tid + u * nwork;
          gg[u] = work && i < ring ? ring_cell(i, cc[u]) : -1;
          if (gg[u] >= 0) {
            get_words(xb + 4 * (size_t)gg[u], q0[u], q1[u]);
            get_words(xb + 4 * (size_t)gg[u] + 2, q2[u], q3[u]);
          }
        }
        __syncthreads();
        auto take = [&](int g, int c, unsigned long long a, unsigned long long b,
                        unsigned long long d, unsigned long long e) {
          if (!wait_pair(xb + 4 * (size_t)g, ep, a, b, &s_fault) ||
              !wait_pair(xb + 4 * (size_t)g + 2, ep, d, e, &s_fault))
            s_fault = 1;
          cur1[c] = words_double(a, b);
          cur2[c] = words_double(d, e);
        };
#pragma unroll
        for (int u = 0; u < UN; ++u)
          if (gg[u] >= 0) take(gg[u], cc[u], q0[u], q1[u], q2[u], q3[u]);
        for (int i = tid + UN * nwork; work && i < ring; i += nwork) {
          int c;
          const int g = ring_cell(i, c);
          if (g < 0) continue;
          unsigned long long a, b, d, e;
          get_words(xb + 4 * (size_t)g, a, b);
          get_words(xb + 4 * (size_t)g + 2, d, e);
          take(g, c, a, b, d, e);
        }
        __syncthreads();
        if (s_fault) break;
      }
      if (app == 1) ++it;
      if (bad) s_bad = 1;
      __syncthreads();
    }
  }

  // the final a and p (p of the pair the last residual belongs to)
  for (int i = tid; i < w * h; i += blockDim.x) {
    const int y = i / w, x = i - y * w;
    const size_t at = (size_t)(y0 + y) * nx + x0 + x;
    A.a[at] = s_a[i];
    A.p[at] = s_p[i];
  }
  if (tid == 0) {
    if (s_fault) atomicOr(&ctrl->nonfinite, 2);
    if (blockIdx.x == 0) {
      ctrl->it = it;
      *A.epoch = epoch::after(ep0, ep, epoch::of_heat(A.pairs, A.D, H), s_fault);
    }
  }
}

template <typename T>
void* heat_tile_fn(int ek) {
  if (ek == EK_CROWD) return (void*)heat_tile_kernel<T, EK_CROWD>;
  if (ek == EK_ENTROPY) return (void*)heat_tile_kernel<T, EK_ENTROPY>;
  return (void*)heat_tile_kernel<T, EK_POWER>;
}

}  // namespace

// One tile per block and at most one block per SM: the tile shape with the least work per
// phase.  Where a tile with its halo does not fit the shared memory (on 152 SMs beyond about 850
// cells a side in FP32, 730 in FP64) heat.cu's form stays, whose blocks walk over several tiles.
template <typename T>
HeatTilePlan heat_tile_plan(int nx, int ny, int ek) {
  HeatTilePlan tp;
  int dev = 0, coop = 0, sms = 0, smem_max = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return tp;
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (!coop || sms < 1) return tp;
  heat_geom::tile_shape(nx, ny, sms, &tp.tw, &tp.th);
  tp.ntx = ceil_div(nx, tp.tw);
  const int nb = tp.ntx * ceil_div(ny, tp.th);
  tp.smem = heat_geom::tile_bytes(tp.tw, tp.th, sizeof(T));
  const int area = (tp.tw + 2 * H - 2) * (tp.th + 2 * H - 2);
  tp.threads = 32 + std::min(HTT - 32, (area + 31) / 32 * 32);
  if (tp.smem + 1024 > (size_t)smem_max) return tp;
  void* fn = heat_tile_fn<T>(ek);
  int per_sm = 0;
  if (max_dynamic_smem(fn) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, tp.threads, tp.smem) !=
          cudaSuccess ||
      per_sm * sms < nb) {
    cudaGetLastError();
    return tp;
  }
  tp.G = nb;
  const size_t N = (size_t)nx * ny;
  tp.words = N * 12 + ((N * kWords<T> + 1) & ~(size_t)1) +
             4 * (size_t)(ceil_div(nx, HBX) * ceil_div(ny, HBY)) + 2;
  return tp;
}

template <typename T>
cudaError_t heat_tile_launch(const HeatTilePlan& tp, const HeatPlan& hp, const HeatBuffers& B,
                             int ek, const T* q, T* a, T* p, int nx, int ny, const uint8_t* mask,
                             const ProxArgs<T>& P, Ctrl* ctrl, unsigned long long* words,
                             int pairs, cudaStream_t st) {
  const size_t N = (size_t)nx * ny;
  const double inv_delta = hp.delta > 0 ? 1.0 / hp.delta : 0.0;
  const int gx = ceil_div(nx, HBX), ng = gx * ceil_div(ny, HBY);
  HeatTileArgs<T> A{nx, ny, tp.tw, tp.th, tp.ntx, hp.D, gx, ng, 2.0 * inv_delta * hp.cx,
                    2.0 * inv_delta * hp.cy, (const double*)B.coef, mask, q, a, p, ctrl, words,
                    words + 8 * N, words + 12 * N, words + tp.words - 2 - 4 * (size_t)ng,
                    (unsigned*)(words + tp.words - 2), pairs};
  ProxArgs<T> Pc = P;
  void* args[] = {&A, &Pc};
  StripPlan sp;
  sp.G = tp.G;
  return strip_coop(heat_tile_fn<T>(ek), sp, tp.smem, tp.threads, args, st);
}

#define JKO_HEAT_TILE_INST(T)                                                                    \
  template HeatTilePlan heat_tile_plan<T>(int, int, int);                                        \
  template cudaError_t heat_tile_launch<T>(const HeatTilePlan&, const HeatPlan&,                 \
                                           const HeatBuffers&, int, const T*, T*, T*, int, int,  \
                                           const uint8_t*, const ProxArgs<T>&, Ctrl*,            \
                                           unsigned long long*, int, cudaStream_t);
JKO_HEAT_TILE_INST(float)
JKO_HEAT_TILE_INST(double)
#undef JKO_HEAT_TILE_INST

}  // namespace jko
