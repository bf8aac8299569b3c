// One-block step kernel with the whole iteration problem in shared memory (rows A4-A7
// of the hot path for small LPs, pdlp_params.persistent = 2).
//
// The 200 x 400 MIP relaxations (1,600 nonzeros) leave a GPU-wide kernel nothing to
// spread: every step is a chain of dependent global loads (row pointer, column index,
// gathered entry) that a handful of warps cannot hide, and a launch per kernel costs as
// much as the work.  Here one block copies A and A^T (row pointers, column indices and
// values in the iterate type; none for a 0/1 pattern), the problem vectors and both
// iterate buffers into shared memory once per launch, then runs step attempts back to
// back until a KKT check falls due, the state stops the solve or `max_attempts` ran:
//   primal: x' = proj_[l,u](x - tau (c - K^T y)), the columns of A^T; ||x' - x||^2;
//   dual:   y' = proj_Y(y + sigma (q - K(2x' - x))) from the (x', x' - x) pairs, the rows
//           of A; ||y' - y||^2 and (y' - y)^T K (x' - x);
//   decision (A6) by thread 0 on the block's copy of the state, its factors fetched while
//           the steps run and its records written by another warp during the next one,
// with a block barrier between the phases.  The block has threads for one round of rows
// where it can (SmemThreads), and up to eight lanes share a row where that leaves some
// over: an attempt is a chain of latencies.  The rows go longest first (a stable order by
// length, built once per solve at setup), so those of a warp have nearly equal lengths: a
// float64 warp instruction holds the SM's float64 pipe ~16 cycles whatever its active
// lanes, and a warp's sum loop runs as long as its longest row.  At exit the iterate
// buffers and running sums go back to global memory (where the KKT block reads them) with
// the state.  The same iteration as the two-launch kernels; the sums are added in another
// order, so float64 iterates agree with theirs to rounding.
#pragma once

#include "internal.h"
#include "iter_kernels.cuh"
#include "resident_kernels.cuh"  // the decision in two halves, div_pos

namespace pdlp {

// threads of the block at most; the rows a side has decide how many there are
// (float64: 256, whose sums fit the static shared memory)
template <typename T> struct SmemThreads { static constexpr int value = sizeof(T) == 8 ? 256 : 512; };

__device__ __forceinline__ float smem_div(float n, float d) { return div_pos(n, d); }
__device__ __forceinline__ double smem_div(double n, double d) { return n / d; }

// acc += value times gathered entry
template <typename T>
__device__ __forceinline__ void smem_add(T& acc, T v, T x) { acc = fma(v, x, acc); }
template <typename T>
__device__ __forceinline__ void smem_add(P2<T>& acc, T v, const vec2_t<T>& x) {
  acc.a = fma(v, x.x, acc.a);
  acc.b = fma(v, x.y, acc.b);
}
// Sums of the rows' entries, LANES lanes per row, the rows in the order `ord`.  Four entries of a
// lane at a time, those past the end of the row read as zeros: a row waits for one chain of loads
// per four entries, with no tail of single ones.
template <int LANES, typename T, typename Acc, typename G, typename Val, typename At, typename Fin>
__device__ __forceinline__ void smem_rows(int rows, const int* ord, const int* ptr, Val val, At at,
                                          Fin fin) {
  const int lane = threadIdx.x & (LANES - 1);
  for (int t = threadIdx.x / LANES; t < rows; t += blockDim.x / LANES) {
    const int r = ord[t], e = ptr[r + 1];
    Acc acc{};
    for (int p = ptr[r] + lane; p < e; p += 4 * LANES) {
      T v[4];
      G x[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int pk = p + k * LANES;
        v[k] = (T)0;
        x[k] = G{};
        if (pk < e) {
          v[k] = val(pk);
          x[k] = at(pk);
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) smem_add(acc, v[k], x[k]);
    }
    acc = group_sum<LANES>(acc);
    if (lane == 0) fin(r, acc);
  }
}
template <typename T, typename Acc, typename G, typename Val, typename At, typename Fin>
__device__ __forceinline__ void smem_rows_lanes(int lanes, int rows, const int* ord, const int* ptr,
                                                Val val, At at, Fin fin) {
  switch (lanes) {
    case 1: return smem_rows<1, T, Acc, G>(rows, ord, ptr, val, at, fin);
    case 2: return smem_rows<2, T, Acc, G>(rows, ord, ptr, val, at, fin);
    case 4: return smem_rows<4, T, Acc, G>(rows, ord, ptr, val, at, fin);
    default: return smem_rows<8, T, Acc, G>(rows, ord, ptr, val, at, fin);
  }
}

template <typename T, typename V, bool IMPLICIT>
__global__ void __launch_bounds__(SmemThreads<T>::value) k_smem(IterData<T, V> d, SmemLayout L, int lanes_t,
                                                               int lanes_a, int max_attempts) {
  constexpr bool VALS = !std::is_same<V, Pattern>::value;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ DevState ls;
  __shared__ int stop;
  // the threads' sums (float64: one warp adds them) or the warps'
  __shared__ T red[3][std::is_same<T, double>::value ? SmemThreads<T>::value : 32];
  DevState* gst = d.st;
  if (threadIdx.x == 0) {
    ls = *gst;
    stop = (ls.status != 0 || ls.check_due) ? 1 : 0;
  }
  __syncthreads();
  if (stop) return;
  const int m = d.m, n = d.n, tid = threadIdx.x, NT = blockDim.x;
  int* tp = (int*)(sm + L.t_ptr);
  int* tc = (int*)(sm + L.t_col);
  T* tv = VALS ? (T*)(sm + L.t_val) : nullptr;
  int* ap = (int*)(sm + L.a_ptr);
  int* ac = (int*)(sm + L.a_col);
  T* av = VALS ? (T*)(sm + L.a_val) : nullptr;
  T* c = (T*)(sm + L.c);
  T* l = (T*)(sm + L.l);
  T* u = (T*)(sm + L.u);
  T* tw = IMPLICIT ? (T*)(sm + L.tw) : nullptr;
  T* q = (T*)(sm + L.q);
  T* sw = IMPLICIT ? (T*)(sm + L.sw) : nullptr;
  unsigned char* kind = sm + L.kind;
  vec2_t<T>* xs[2] = {(vec2_t<T>*)(sm + L.x0), (vec2_t<T>*)(sm + L.x1)};
  T* ys[2] = {(T*)(sm + L.y0), (T*)(sm + L.y1)};
  T* sx = (T*)(sm + L.sx);
  T* sy = (T*)(sm + L.sy);
  int* ot = (int*)(sm + L.ot);
  int* oa = (int*)(sm + L.oa);
  // ---- copy in (iterates with ordinary loads: the KKT block of the same graph wrote them)
  const int nnz = __ldg(d.t_ptr + n);
  for (int i = tid; i <= n; i += NT) tp[i] = __ldg(d.t_ptr + i);
  for (int i = tid; i <= m; i += NT) ap[i] = __ldg(d.a_ptr + i);
  // the order the threads take the columns and rows in (longest first, built at setup)
  for (int i = tid; i < n; i += NT) ot[i] = __ldg(d.ord_t + i);
  for (int i = tid; i < m; i += NT) oa[i] = __ldg(d.ord_a + i);
  for (int p = tid; p < nnz; p += NT) {
    tc[p] = __ldg(d.t_col + p);
    ac[p] = __ldg(d.a_col + p);
    if constexpr (VALS) {
      tv[p] = Ld<T, V>::get(d.t_val, p);
      av[p] = Ld<T, V>::get(d.a_val, p);
    }
  }
  for (int j = tid; j < n; j += NT) {
    c[j] = __ldg(d.c + j);
    l[j] = __ldg(d.l + j);
    u[j] = __ldg(d.u + j);
    if constexpr (IMPLICIT) tw[j] = __ldg(d.tw + j);
    xs[0][j] = d.x[0][j];
    xs[1][j] = d.x[1][j];
    sx[j] = d.sum_x[j];
  }
  for (int i = tid; i < m; i += NT) {
    q[i] = __ldg(d.q + i);
    if constexpr (IMPLICIT) sw[i] = __ldg(d.sw + i);
    kind[i] = __ldg(d.row_kind + i);
    ys[0][i] = d.y[0][i];
    ys[1][i] = d.y[1][i];
    sy[i] = d.sum_y[i];
  }
  // accepted steps to the next check (thread 0)
  int left = 0;
  if (tid == 0) {
    const long long p = ls.period - ls.iters % ls.period, q = ls.iter_limit - ls.iters;
    left = (int)(p < q ? p : q > 1 ? q : 1);
  }
  for (int i = tid; i < (int)(sizeof(red[0]) / sizeof(T)); i += NT) red[0][i] = red[1][i] = red[2][i] = (T)0;
  __shared__ ResDecision<T> dec[2];  // of this attempt and of the one before
  const long long first_attempt = ls.attempts;
  __syncthreads();
  int att = 0;
  for (; att < max_attempts; ++att) {
    const int cur = ls.cur;
    const T pw = StepT<T>::pw(&ls), tau = StepT<T>::tau(&ls), sigma = StepT<T>::sigma(&ls);
    const vec2_t<T>* x = xs[cur];
    vec2_t<T>* xn = xs[cur ^ 1];
    const T* y = ys[cur];
    T* yn = ys[cur ^ 1];
    T fd = 0, fi = 0;
    if (tid == 0) step_factors(&ls, first_attempt + att + 1, &fd, &fi);
    // the attempt before, recorded by the warp with the shortest columns or none
    if (tid == NT - 32 && att > 0) res_record<T>(&ls, dec[(att & 1) ^ 1]);
    // ---- A4: primal step
    T dx2 = 0;
    smem_rows_lanes<T, T, T>(
        lanes_t, n, ot, tp, [&](int p) -> T { return VALS ? tv[p] : (T)1; },
        [&](int p) -> T { return y[tc[p]]; },
        [&](int j, T aty) {
          const T xo = x[j].x;
          const T step = IMPLICIT ? tau * tw[j] : tau;
          const T xv = clampv(xo - step * (c[j] - aty), l[j], u[j]);
          const T dd = xv - xo;
          vec2_t<T> o;
          o.x = xv;
          o.y = dd;
          xn[j] = o;
          if (pw != (T)0) sx[j] += pw * xo;  // A7: add the iterate whose weight is pending
          if constexpr (IMPLICIT) dx2 += smem_div(dd * dd, tw[j]);
          else dx2 += dd * dd;
        });
    __syncthreads();  // xn complete before the dual phase gathers it
    // ---- A5: dual step; the sums are (K x')_i, (K dx)_i
    T dy2 = 0, dkd = 0;
    smem_rows_lanes<T, P2<T>, vec2_t<T>>(
        lanes_a, m, oa, ap, [&](int p) -> T { return VALS ? av[p] : (T)1; },
        [&](int p) -> vec2_t<T> { return xn[ac[p]]; },
        [&](int i, P2<T> k) {
          const T yo = y[i];
          const T step = IMPLICIT ? sigma * sw[i] : sigma;
          T yv = yo + step * (q[i] - (k.a + k.b));
          if (kind[i] != 1) yv = maxv(yv, (T)0);
          yn[i] = yv;
          if (pw != (T)0) sy[i] += pw * yo;
          const T dd = yv - yo;
          if constexpr (IMPLICIT) dy2 += smem_div(dd * dd, sw[i]);
          else dy2 += dd * dd;
          dkd += dd * k.b;
        });
    // the three sums: in float32 every warp adds its own and one warp the warps'; in float64
    // one warp adds all the threads' through shared memory (a float64 warp instruction holds
    // the pipe as long with one active lane as with 32)
    T s[3] = {dx2, dy2, dkd};
    if constexpr (std::is_same<T, float>::value) {
      res_warp_sums(s, 1, 32);
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if ((tid & 31) == 0) red[k][tid >> 5] = s[k];
    } else {
#pragma unroll
      for (int k = 0; k < 3; ++k) red[k][tid] = s[k];
    }
    __syncthreads();
    if (tid < 32) {
      if constexpr (std::is_same<T, float>::value) {
#pragma unroll
        for (int k = 0; k < 3; ++k) s[k] = red[k][tid];
      } else {
        constexpr int W = SmemThreads<T>::value / 32;  // (threads beyond the block's left zeros)
        T w[3][W];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
          for (int i = 0; i < W; ++i) w[k][i] = red[k][tid + 32 * i];
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1)
#pragma unroll
          for (int i = 0; i < o; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) w[k][i] += w[k][i + o];
#pragma unroll
        for (int k = 0; k < 3; ++k) s[k] = w[k][0];
      }
      res_warp_sums(s, 1, 32);
      // ---- A6: the decision
      if (tid == 0) dec[att & 1] = res_decide<T>(&ls, s[0], s[1], s[2], fd, fi, left);
    }
    __syncthreads();
    if (ls.status != 0 || ls.check_due) {
      ++att;
      break;
    }
  }
  if (tid == 0 && att > 0) res_record<T>(&ls, dec[(att - 1) & 1]);  // of the last attempt
  // ---- copy out
  for (int j = tid; j < n; j += NT) {
    d.x[0][j] = xs[0][j];
    d.x[1][j] = xs[1][j];
    d.sum_x[j] = sx[j];
  }
  for (int i = tid; i < m; i += NT) {
    d.y[0][i] = ys[0][i];
    d.y[1][i] = ys[1][i];
    d.sum_y[i] = sy[i];
  }
  if (tid == 0) store_step_state(gst, ls);
}

}  // namespace pdlp
