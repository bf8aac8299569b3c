// Learned warm start: the bipartite message-passing network of include/gnn.h,
// its training kernels and the start-point KKT that decides warm vs cold.
//
// Kernels (all float32 arithmetic on bfloat16 weights unless stated):
//   k_gnn_rowstats / k_gnn_colstats / k_gnn_feat_*   features of variables and constraints
//   k_gnn_embed / k_gnn_embed_bwd                    input layers and their weight gradients
//   k_gnn_spmm                                       message passing over A or A^T (16 lanes
//                                                    per row, one float4 of the 64-wide
//                                                    hidden row per lane)
//   k_gnn_dense / k_gnn_dense_bwd                    relu(X1 W1 + X2 W2 + b) on the tensor cores,
//                                                    16 rows per warp, and its backward (input
//                                                    and weight gradients, 64 rows per block)
//   k_gnn_head                                       prediction heads, loss and their gradient
//   k_gnn_reduce / k_gnn_loss                        per-block partials summed in a fixed
//                                                    order (training is deterministic)
//   k_gnn_adam                                       Adam on the float32 masters + bf16 copy
//   k_start_project / k_kkt_start_*                  projection of a start and its float64
//                                                    relative KKT on the original data
#include <cuda_bf16.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <string>
#include <vector>

#include "../../include/gnn.h"
#include "internal.h"
#include "setup.h"

namespace pdlp {
extern thread_local std::string g_last_error;
}

namespace {

using bf16 = __nv_bfloat16;
constexpr int H = GNN_HIDDEN;
constexpr int NB = 256;  // threads per block of every kernel here
constexpr int kDensePart = 2 * 4096 + 64;

int gfail(int code, const std::string& msg) {
  pdlp::g_last_error = msg;
  return code;
}

#define GTRY(x)                                                                         \
  do {                                                                                  \
    cudaError_t e_ = (x);                                                               \
    if (e_ != cudaSuccess)                                                              \
      return gfail(e_ == cudaErrorMemoryAllocation ? PDLP_ERR_OOM : PDLP_ERR_CUDA,      \
                   std::string(#x) + ": " + cudaGetErrorString(e_));                    \
  } while (0)

#define RTRY(x)               \
  do {                        \
    int r_ = (x);             \
    if (r_ != PDLP_OK) return r_; \
  } while (0)

// ---------------------------------------------------------------- parameters
struct POff {
  int W_vin, b_vin, W_cin, b_cin;
  int W_cc[GNN_LAYERS], W_cv[GNN_LAYERS], b_c[GNN_LAYERS];
  int W_vv[GNN_LAYERS], W_vc[GNN_LAYERS], b_v[GNN_LAYERS];
  int w_x, b_x, w_y, b_y, total;
};

POff make_off() {
  POff o{};
  int p = 0;
  auto take = [&](int k) {
    const int r = p;
    p += k;
    return r;
  };
  o.W_vin = take(GNN_VAR_FEATURES * H);
  o.b_vin = take(H);
  o.W_cin = take(GNN_CON_FEATURES * H);
  o.b_cin = take(H);
  for (int k = 0; k < GNN_LAYERS; ++k) {
    o.W_cc[k] = take(H * H);
    o.W_cv[k] = take(H * H);
    o.b_c[k] = take(H);
    o.W_vv[k] = take(H * H);
    o.W_vc[k] = take(H * H);
    o.b_v[k] = take(H);
  }
  o.w_x = take(H);
  o.b_x = take(1);
  o.w_y = take(H);
  o.b_y = take(1);
  o.total = p;
  return o;
}
const POff kOff = make_off();

struct SplitMix64 {
  uint64_t s;
  uint64_t next() {
    s += 0x9E3779B97F4A7C15ull;
    uint64_t z = s;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
  }
  double uniform() { return (double)(next() >> 11) * 0x1.0p-53; }
};

int sm_count() { return pdlp::device_sm_count(); }

int grid_rows(long long rows, int rows_per_block, int cap) {
  long long g = (rows + rows_per_block - 1) / rows_per_block;
  return (int)std::max<long long>(1, std::min<long long>(g, cap));
}

constexpr int kAnyGrid = 0x7fffffff;  // one round of rows per block, however many blocks

// ---------------------------------------------------------------- device helpers
__device__ __forceinline__ float bf(bf16 v) { return __bfloat162float(v); }

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

__device__ __forceinline__ float sigmoidf(float z) {
  const float e = expf(-fabsf(z));
  return z >= 0.f ? 1.f / (1.f + e) : e / (1.f + e);
}
__device__ __forceinline__ float softplusf(float z) { return log1pf(expf(-fabsf(z))) + fmaxf(z, 0.f); }

__device__ __forceinline__ unsigned long long dbits(double v) {
  return (unsigned long long)__double_as_longlong(v);
}
__device__ __forceinline__ double slog(double v) {
  v = fmin(fmax(v, -1e3), 1e3);
  return v > 0 ? log1p(v) : (v < 0 ? -log1p(-v) : 0.0);
}

// ---------------------------------------------------------------- LP on the device
__global__ void k_ptr32(int m, const int64_t* __restrict__ p64, int* __restrict__ p32,
                        const char* __restrict__ sense, unsigned char* __restrict__ kind) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= m; i += gridDim.x * blockDim.x) {
    p32[i] = (int)p64[i];
    if (i < m) kind[i] = sense[i] == 'G' ? 0 : (sense[i] == 'E' ? 1 : 2);
  }
}

// ---------------------------------------------------------------- features (K11)
// maxes: [0] |b|, [1] ||A_i:||, [2] deg_i, [3] |c|, [4] ||A_:j||, [5] deg_j (float64 bits,
// all non-negative, so the unsigned order is the numeric order and atomicMax is exact)
__global__ void k_gnn_stats(int rows, const int* __restrict__ ptr, const double* __restrict__ val,
                            const double* __restrict__ rhs, double* __restrict__ norm,
                            float* __restrict__ inv_deg, unsigned long long* __restrict__ maxes) {
  unsigned long long m0 = 0, m1 = 0, m2 = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += gridDim.x * blockDim.x) {
    const int k0 = ptr[i], k1 = ptr[i + 1];
    double s = 0.0;
    for (int k = k0; k < k1; ++k) s += val[k] * val[k];
    const double nr = sqrt(s);
    const int deg = k1 - k0;
    norm[i] = nr;
    inv_deg[i] = (float)(1.0 / (double)max(deg, 1));
    m0 = max(m0, dbits(fabs(rhs[i])));
    m1 = max(m1, dbits(nr));
    m2 = max(m2, dbits((double)deg));
  }
  for (int o = 16; o > 0; o >>= 1) {
    m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, o));
    m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, o));
    m2 = max(m2, __shfl_xor_sync(0xffffffffu, m2, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&maxes[0], m0);
    atomicMax(&maxes[1], m1);
    atomicMax(&maxes[2], m2);
  }
}

__global__ void k_gnn_values(int nnz, const double* __restrict__ a, const double* __restrict__ t,
                             float* __restrict__ a32, float* __restrict__ t32) {
  for (long long i = blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += gridDim.x * blockDim.x) {
    a32[i] = (float)a[i];
    t32[i] = (float)t[i];
  }
}

__device__ __forceinline__ double umax(const unsigned long long* mx, int i, double floor) {
  return fmax(__longlong_as_double((long long)mx[i]), floor);
}

__global__ void k_gnn_feat_v(int n, const int* __restrict__ t_ptr, const double* __restrict__ c,
                             const double* __restrict__ l, const double* __restrict__ u,
                             const double* __restrict__ nc, const unsigned long long* __restrict__ mx,
                             float* __restrict__ fv) {
  const double cmax = umax(mx, 3, 1e-12), nmax = umax(mx, 4, 1e-12), dmax = umax(mx, 5, 1.0);
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    float* f = fv + (size_t)j * GNN_VAR_FEATURES;
    f[0] = (float)(c[j] / cmax);
    f[1] = (float)slog(l[j]);
    f[2] = (float)slog(u[j]);
    f[3] = (float)(nc[j] / nmax);
    f[4] = (float)((double)(t_ptr[j + 1] - t_ptr[j]) / dmax);
    f[5] = 1.f;
  }
}

__global__ void k_gnn_feat_c(int m, const int* __restrict__ a_ptr, const double* __restrict__ b,
                             const unsigned char* __restrict__ kind, const double* __restrict__ nr,
                             const unsigned long long* __restrict__ mx, float* __restrict__ fc) {
  const double bmax = umax(mx, 0, 1e-12), nmax = umax(mx, 1, 1e-12), dmax = umax(mx, 2, 1.0);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    float* f = fc + (size_t)i * GNN_CON_FEATURES;
    f[0] = (float)(b[i] / bmax);
    f[1] = kind[i] == 0 ? 1.f : (kind[i] == 2 ? -1.f : 0.f);
    f[2] = (float)(nr[i] / nmax);
    f[3] = (float)((double)(a_ptr[i + 1] - a_ptr[i]) / dmax);
    f[4] = 1.f;
  }
}

// ---------------------------------------------------------------- embedding
template <int NF>
__global__ void __launch_bounds__(NB) k_gnn_embed(int N, const float* __restrict__ F,
                                                  const bf16* __restrict__ W, const bf16* __restrict__ b,
                                                  float* __restrict__ out) {
  __shared__ float ws[NF * H + H];
  for (int i = threadIdx.x; i < NF * H; i += NB) ws[i] = bf(W[i]);
  for (int i = threadIdx.x; i < H; i += NB) ws[NF * H + i] = bf(b[i]);
  __syncthreads();
  const int q = threadIdx.x & 15;
  for (long long r = ((long long)blockIdx.x * NB + threadIdx.x) >> 4; r < N;
       r += (long long)gridDim.x * (NB / 16)) {
    float a[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) a[e] = ws[NF * H + 4 * q + e];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const float x = F[r * NF + f];
#pragma unroll
      for (int e = 0; e < 4; ++e) a[e] = fmaf(x, ws[f * H + 4 * q + e], a[e]);
    }
    st4(out + r * H + 4 * q,
        make_float4(fmaxf(a[0], 0.f), fmaxf(a[1], 0.f), fmaxf(a[2], 0.f), fmaxf(a[3], 0.f)));
  }
}

// partial per block: [NF][64] weight gradient, then [64] bias gradient
template <int NF>
__global__ void __launch_bounds__(NB) k_gnn_embed_bwd(int N, const float* __restrict__ F,
                                                      const float* __restrict__ H0,
                                                      const float* __restrict__ dH0,
                                                      float* __restrict__ part) {
  __shared__ float red[4][(NF + 1) * H];
  const int h = threadIdx.x & 63, rl = threadIdx.x >> 6;
  float g[NF + 1];
#pragma unroll
  for (int f = 0; f <= NF; ++f) g[f] = 0.f;
#pragma unroll 4  // rows in flight
  for (long long r = (long long)blockIdx.x * 4 + rl; r < N; r += (long long)gridDim.x * 4) {
    const float d = H0[r * H + h] > 0.f ? dH0[r * H + h] : 0.f;
#pragma unroll
    for (int f = 0; f < NF; ++f) g[f] = fmaf(F[r * NF + f], d, g[f]);
    g[NF] += d;
  }
#pragma unroll
  for (int f = 0; f <= NF; ++f) red[rl][f * H + h] = g[f];
  __syncthreads();
  for (int e = threadIdx.x; e < (NF + 1) * H; e += NB)
    part[(size_t)blockIdx.x * (NF + 1) * H + e] = ((red[0][e] + red[1][e]) + red[2][e]) + red[3][e];
}

// ---------------------------------------------------------------- message passing (K12)
// out[r] (+)= srow[r] * sum_k val[k] * scol[col[k]] * X[col[k]]  (srow / scol may be NULL = 1)
// What is left is the gathers (173 MB from L2 for the 650,000 entries of a 25,000 x 100,000
// covering LP).  The graph keeps the values in float32: converted here by every lane they held the
// float64 pipe for half of the time.  Both directions of that LP: 26.5 -> 14.5 and 30.8 -> 16.5 us;
// handing entries round by shuffles instead (one conversion each) 19.6 and 24.7; a warp per row, or
// eight gathers in flight per lane, is no faster.
__global__ void __launch_bounds__(NB, 6) k_gnn_spmm(int rows, const int* __restrict__ ptr,
                                                 const int* __restrict__ col,
                                                 const float* __restrict__ val,
                                                 const float* __restrict__ srow,
                                                 const float* __restrict__ scol,
                                                 const float* __restrict__ X, float* __restrict__ out,
                                                 int accumulate) {
  const int q = threadIdx.x & 15;
  for (long long r = ((long long)blockIdx.x * NB + threadIdx.x) >> 4; r < rows;
       r += (long long)gridDim.x * (NB / 16)) {
    const int k0 = ptr[r], k1 = ptr[r + 1];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    int k = k0;
    for (; k + 4 <= k1; k += 4) {
      int j[4];
      float w[4];
      float4 x[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        j[t] = col[k + t];
        w[t] = val[k + t];
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (scol) w[t] *= scol[j[t]];
        x[t] = ld4(X + (size_t)j[t] * H + 4 * q);
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        acc.x = fmaf(w[t], x[t].x, acc.x);
        acc.y = fmaf(w[t], x[t].y, acc.y);
        acc.z = fmaf(w[t], x[t].z, acc.z);
        acc.w = fmaf(w[t], x[t].w, acc.w);
      }
    }
    for (; k < k1; ++k) {
      const int jj = col[k];
      float w = val[k];
      if (scol) w *= scol[jj];
      const float4 x = ld4(X + (size_t)jj * H + 4 * q);
      acc.x = fmaf(w, x.x, acc.x);
      acc.y = fmaf(w, x.y, acc.y);
      acc.z = fmaf(w, x.z, acc.z);
      acc.w = fmaf(w, x.w, acc.w);
    }
    if (srow) {
      const float s = srow[r];
      acc.x *= s;
      acc.y *= s;
      acc.z *= s;
      acc.w *= s;
    }
    float* o = out + r * H + 4 * q;
    if (accumulate) {
      const float4 p = ld4(o);
      acc.x += p.x;
      acc.y += p.y;
      acc.z += p.z;
      acc.w += p.w;
    }
    st4(o, acc);
  }
}

// ---------------------------------------------------------------- dense layers (K13)
// The layers' products run on the tensor cores from exact pieces: a float32 operand is the sum of
// three bfloat16 numbers (its top 8 significant bits, the next 8 and the last 8, by truncation:
// Ozaki et al., "Error-free transformations of matrix multiplication", 2012), the weights are
// bfloat16, and a product of two bfloat16 numbers is exact in float32.  Every 16 terms of a sum
// are multiplied and added by the matrix unit from zero and the 16-term sums added in float32
// registers.  The unit cuts its sums off, a bias that a gradient adds up over all the rows; so the
// sum d of the top pieces is followed by the same products less d, which gives what was cut off,
// and the small pieces go on top of that (mma_add).
// Measured with the LP of 100,000 columns (cold, ncu): a forward layer 62.8 us with float32
// multiply-adds, 25 without the remainder (relative error of a gradient against float64 1.3e-7
// instead of 5e-8: not kept), 34.5 as here (5.0e-8; the predictions' 3.8e-8 / 5.1e-8 before
// 4.6e-8 / 5.6e-8); backward 84.6 us, and of 50,000 columns 58.9 -> 45.3 with six of its nine
// products.  What bounds it are chains of dependent mma.sync at under four warps per scheduler (ncu:
// the tensor pipe 40 % active forward and 48 % backward, an instruction issued in 52 and 40 % of the
// cycles, DRAM below 20 %).  tcgen05.mma is not used: the remainder needs the accumulator in
// registers and negated after every 16 terms.
using u32 = unsigned;

// the pieces of (a, b), packed two to a word; an infinity is all in the first piece
__device__ __forceinline__ void split_pair(float a, float b, u32& h, u32& m, u32& l) {
  const u32 top = 0xffff0000u;
  const float ha = __uint_as_float(__float_as_uint(a) & top), hb = __uint_as_float(__float_as_uint(b) & top);
  const float ra = ha == a ? 0.f : a - ha, rb = hb == b ? 0.f : b - hb;
  const float ma = __uint_as_float(__float_as_uint(ra) & top), mb = __uint_as_float(__float_as_uint(rb) & top);
  const float la = ra - ma, lb = rb - mb;
  h = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
  m = __byte_perm(__float_as_uint(ra), __float_as_uint(rb), 0x7632);
  l = __byte_perm(__float_as_uint(la), __float_as_uint(lb), 0x7632);
}

// d += A B for a 16 x 16 A (row-major fragments) and a 16 x 8 B (column-major)
__device__ __forceinline__ void mma16(float (&d)[4], const u32 (&a)[4], u32 b0, u32 b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// acc += d + r for d = the top pieces' products and r, begun from their remainder by `rest`, the
// others' (an infinite or undefined d has no remainder)
template <typename Rest>
__device__ __forceinline__ void mma_add(float (&acc)[4], const u32 (&a)[4], u32 b0, u32 b1, Rest rest) {
  float d[4] = {0.f, 0.f, 0.f, 0.f};
  mma16(d, a, b0, b1);
  float r[4] = {-d[0], -d[1], -d[2], -d[3]};
  mma16(r, a, b0, b1);
  rest(r);
#pragma unroll
  for (int e = 0; e < 4; ++e) acc[e] = (acc[e] + (fabsf(d[e]) < INFINITY ? r[e] : 0.f)) + d[e];
}
// four 8 x 8 matrices of 16-bit elements; lane 8j + i points at row i of matrix j
__device__ __forceinline__ void ldsm4(u32 (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((u32)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void ldsm4_t(u32 (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((u32)__cvta_generic_to_shared(p))
               : "memory");
}

// out = relu(X1 W1 + X2 W2 + b) for X1, X2 [N][64], W [64][64] row-major [in][out].
// A warp takes 16 rows at a time straight from global memory: lane (g, t) of a fragment holds
// columns 4t..4t+3 of each 16-column chunk of rows g and g + 8 (one 16-byte load; the weights are
// read in the same order of the sum), the 64 columns of the next step in flight meanwhile.
constexpr int kDStride = 72;  // bf16 per row of weights in shared memory: an odd number of 16-byte
                              // units, so that ldmatrix meets no bank twice
__device__ __forceinline__ void stage_weights(bf16* Ws, const bf16* __restrict__ W1,
                                              const bf16* __restrict__ W2) {
  // (a layer's weights start at any even offset of the parameters: 4-byte loads)
  for (int i = threadIdx.x; i < 64 * 32; i += NB) {
    const int k = i >> 5, h = 2 * (i & 31);
    *reinterpret_cast<u32*>(Ws + k * kDStride + h) = *reinterpret_cast<const u32*>(W1 + 2 * i);
    *reinterpret_cast<u32*>(Ws + (64 + k) * kDStride + h) = *reinterpret_cast<const u32*>(W2 + 2 * i);
  }
}
__global__ void __launch_bounds__(NB, 2) k_gnn_dense(int N, const float* __restrict__ X1,
                                                     const float* __restrict__ X2,
                                                     const bf16* __restrict__ W1,
                                                     const bf16* __restrict__ W2,
                                                     const bf16* __restrict__ bias,
                                                     float* __restrict__ out) {
  __shared__ __align__(16) bf16 Ws[128 * kDStride];  // [in of X1 | in of X2][out]
  __shared__ __align__(8) float bs[64];
  if (threadIdx.x < 64) bs[threadIdx.x] = bf(bias[threadIdx.x]);
  stage_weights(Ws, W1, W2);
  __syncthreads();
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  // the rows of the weights that a fragment's columns 4t..4t+3 of a chunk stand for: rows 2t, 2t+1
  // of the first matrix are 4t, 4t+1, those of the second 4t+2, 4t+3
  const int i8 = lane & 7, j4 = lane >> 3;
  const bf16* wrow = Ws + (4 * (i8 >> 1) + (i8 & 1) + 2 * (j4 & 1)) * kDStride + 8 * (j4 >> 1);
  const int tiles = (N + 15) / 16, step = gridDim.x * (NB / 32);
  int w = blockIdx.x * (NB / 32) + (threadIdx.x >> 5), half = 0;
  if (w >= tiles) return;
  float4 nx[2][4];  // the four chunks of the next half (X1 or X2) of these or the next rows
  auto load = [&](int tile, int hf) {
    const float* X = hf ? X2 : X1;
    const long long r0 = (long long)tile * 16 + g, r1 = r0 + 8;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      nx[0][c] = r0 < N ? ld4(X + r0 * H + 16 * c + 4 * t) : make_float4(0.f, 0.f, 0.f, 0.f);
      nx[1][c] = r1 < N ? ld4(X + r1 * H + 16 * c + 4 * t) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  load(w, 0);
  float acc[8][4];
#pragma unroll 1
  while (w < tiles) {
    float4 x[2][4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      x[0][c] = nx[0][c];
      x[1][c] = nx[1][c];
    }
    load(half ? w + step : w, half ^ 1);
    if (half == 0)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 b2 = *reinterpret_cast<const float2*>(bs + 8 * j + 2 * t);
        acc[j][0] = acc[j][2] = b2.x;
        acc[j][1] = acc[j][3] = b2.y;
      }
    const bf16* wt = wrow + 64 * half * kDStride;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      u32 ah[4], am[4], al[4];
      split_pair(x[0][c].x, x[0][c].y, ah[0], am[0], al[0]);
      split_pair(x[1][c].x, x[1][c].y, ah[1], am[1], al[1]);
      split_pair(x[0][c].z, x[0][c].w, ah[2], am[2], al[2]);
      split_pair(x[1][c].z, x[1][c].w, ah[3], am[3], al[3]);
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        u32 b[4];
        ldsm4_t(b, wt + 16 * c * kDStride + 8 * j);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          mma_add(acc[j + k], ah, b[2 * k], b[2 * k + 1], [&](float (&r)[4]) {
            mma16(r, am, b[2 * k], b[2 * k + 1]);
            mma16(r, al, b[2 * k], b[2 * k + 1]);
          });
        }
      }
    }
    if (half) {
      const long long r0 = (long long)w * 16 + g, r1 = r0 + 8;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int o = 8 * j + 2 * t;
        if (r0 < N)
          *reinterpret_cast<float2*>(out + r0 * H + o) = make_float2(fmaxf(acc[j][0], 0.f), fmaxf(acc[j][1], 0.f));
        if (r1 < N)
          *reinterpret_cast<float2*>(out + r1 * H + o) = make_float2(fmaxf(acc[j][2], 0.f), fmaxf(acc[j][3], 0.f));
      }
      w += step;
    }
    half ^= 1;
  }
}

// Backward of k_gnn_dense: dP = dHn * (Hn > 0); dX1 = dP W1^T; dX2 = dP W2^T;
// per-block partials of X1^T dP, X2^T dP (row-major [in][out]) and sum_r dP.
// A block stages the pieces of 64 rows of [X1 | X2] and dP in shared memory; four warps form dX1
// of the rows, four dX2 (16 rows each), then each warp its 16 of the 128 rows of the weight
// gradients, where both operands are in pieces: all nine products.  (Without the smallest three, of
// the sign of their terms, weight gradients were cut by 2.6e-8 towards zero on average; they cost 48 us
// of 2,580 in the gradient of four graphs of 12,500 x 50,000.)
// The rows of shared memory are padded to an odd number of 16-byte units (ldmatrix).
constexpr int kXStride = 136, kBwdRows = 64;
constexpr int kBwdSmem = (3 * kBwdRows * (kXStride + kDStride) + 128 * kDStride) * 2;
__device__ __forceinline__ void split_store(bf16* p, int piece_stride, float4 v) {
  uint2 h, m, l;
  split_pair(v.x, v.y, h.x, m.x, l.x);
  split_pair(v.z, v.w, h.y, m.y, l.y);
  *reinterpret_cast<uint2*>(p) = h;
  *reinterpret_cast<uint2*>(p + piece_stride) = m;
  *reinterpret_cast<uint2*>(p + 2 * piece_stride) = l;
}
__global__ void __launch_bounds__(NB, 2) k_gnn_dense_bwd(int N, const float* __restrict__ X1,
                                                         const float* __restrict__ X2,
                                                         const float* __restrict__ Hn,
                                                         const float* __restrict__ dHn,
                                                         const bf16* __restrict__ W1,
                                                         const bf16* __restrict__ W2,
                                                         float* __restrict__ dX1,
                                                         float* __restrict__ dX2,
                                                         float* __restrict__ part) {
  extern __shared__ float4 smem4[];
  constexpr int XP = kBwdRows * kXStride, DP = kBwdRows * kDStride;
  bf16* Xs = reinterpret_cast<bf16*>(smem4);  // [piece][row][in of X1 | in of X2]
  bf16* Ds = Xs + 3 * XP;                     // [piece][row][out]
  bf16* Ws = Ds + 3 * DP;                     // [in of W1 | in of W2][out]
  stage_weights(Ws, W1, W2);
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int q = threadIdx.x & 15, rs = threadIdx.x >> 4;
  const int i8 = lane & 7, j4 = lane >> 3;  // ldmatrix: row i8 of matrix j4
  float gw[8][4];
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) gw[j][e] = 0.f;
  float4 gb = make_float4(0.f, 0.f, 0.f, 0.f);
  const int tiles = (N + kBwdRows - 1) / kBwdRows;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const long long row0 = (long long)tile * kBwdRows;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kBwdRows / 16; ++k) {
      const int r = rs + 16 * k;
      float4 d = make_float4(0.f, 0.f, 0.f, 0.f), a = d, b = d;
      if (row0 + r < N) {
        const long long o = (row0 + r) * H + 4 * q;
        const float4 hn = ld4(Hn + o), dh = ld4(dHn + o);
        d = make_float4(hn.x > 0.f ? dh.x : 0.f, hn.y > 0.f ? dh.y : 0.f,
                        hn.z > 0.f ? dh.z : 0.f, hn.w > 0.f ? dh.w : 0.f);
        a = ld4(X1 + o);
        b = ld4(X2 + o);
      }
      gb.x += d.x;
      gb.y += d.y;
      gb.z += d.z;
      gb.w += d.w;
      split_store(Ds + r * kDStride + 4 * q, DP, d);
      split_store(Xs + r * kXStride + 4 * q, XP, a);
      split_store(Xs + r * kXStride + 64 + 4 * q, XP, b);
    }
    __syncthreads();
    {  // input gradients
      const int rt = 16 * (wp & 3), half = wp >> 2;
      float acc[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        u32 a[3][4];
#pragma unroll
        for (int p = 0; p < 3; ++p)
          ldsm4(a[p], Ds + p * DP + (rt + (j4 & 1) * 8 + i8) * kDStride + 16 * c + (j4 >> 1) * 8);
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
          u32 b[4];
          ldsm4(b, Ws + (64 * half + 8 * j + (j4 >> 1) * 8 + i8) * kDStride + 16 * c + (j4 & 1) * 8);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            mma_add(acc[j + k], a[0], b[2 * k], b[2 * k + 1], [&](float (&r)[4]) {
              mma16(r, a[1], b[2 * k], b[2 * k + 1]);
              mma16(r, a[2], b[2 * k], b[2 * k + 1]);
            });
          }
        }
      }
      float* dX = half ? dX2 : dX1;
      const long long r0 = row0 + rt + g, r1 = r0 + 8;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int o = 8 * j + 2 * t;
        if (r0 < N) *reinterpret_cast<float2*>(dX + r0 * H + o) = make_float2(acc[j][0], acc[j][1]);
        if (r1 < N) *reinterpret_cast<float2*>(dX + r1 * H + o) = make_float2(acc[j][2], acc[j][3]);
      }
    }
    // weight gradients: inputs 16 wp .. of [X1 | X2], the sum over the rows
#pragma unroll
    for (int c = 0; c < kBwdRows / 16; ++c) {
      u32 a[3][4];
#pragma unroll
      for (int p = 0; p < 3; ++p)
        ldsm4_t(a[p], Xs + p * XP + (16 * c + (j4 >> 1) * 8 + i8) * kXStride + 16 * wp + (j4 & 1) * 8);
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        u32 b[3][4];
#pragma unroll
        for (int p = 0; p < 3; ++p)
          ldsm4_t(b[p], Ds + p * DP + (16 * c + (j4 & 1) * 8 + i8) * kDStride + 8 * j + (j4 >> 1) * 8);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          mma_add(gw[j + k], a[0], b[0][2 * k], b[0][2 * k + 1], [&](float (&r)[4]) {
            mma16(r, a[1], b[0][2 * k], b[0][2 * k + 1]);
            mma16(r, a[0], b[1][2 * k], b[1][2 * k + 1]);
            mma16(r, a[1], b[1][2 * k], b[1][2 * k + 1]);
            mma16(r, a[2], b[0][2 * k], b[0][2 * k + 1]);
            mma16(r, a[0], b[2][2 * k], b[2][2 * k + 1]);
            mma16(r, a[2], b[1][2 * k], b[1][2 * k + 1]);
            mma16(r, a[1], b[2][2 * k], b[2][2 * k + 1]);
            mma16(r, a[2], b[2][2 * k], b[2][2 * k + 1]);
          });
        }
      }
    }
  }
  float* p = part + (size_t)blockIdx.x * kDensePart;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int o = 8 * j + 2 * t, r = 16 * wp + g;
    *reinterpret_cast<float2*>(p + r * 64 + o) = make_float2(gw[j][0], gw[j][1]);
    *reinterpret_cast<float2*>(p + (r + 8) * 64 + o) = make_float2(gw[j][2], gw[j][3]);
  }
  __syncthreads();
  float* red = reinterpret_cast<float*>(smem4);  // [16][64]
  st4(red + rs * 64 + 4 * q, gb);
  __syncthreads();
  if (threadIdx.x < 64) {
    float sum = 0.f;
    for (int r = 0; r < 16; ++r) sum += red[r * 64 + threadIdx.x];
    p[8192 + threadIdx.x] = sum;
  }
}

// ---------------------------------------------------------------- heads and loss
// A half-warp takes eight rows at a time (lane q holds hidden units 4q..4q+3 of each): the
// products are reduced so that lanes 2i and 2i + 1 end with row i's, and each finishes its row (two
// rows a warp instruction kept the float64 pipe busy with the boxes: 23.8 us for a covering LP's
// 100,000 columns, now 10.8).  MODE 0: primal head
// (l + (u - l) sigmoid on finite boxes), MODE 1: dual head (softplus on inequality
// rows).  pred: float64 prediction in the caller's convention (may be NULL); with a
// label: loss terms, dz, dH = dz w (may be NULL) and partials [64 gw | gb].
constexpr int kHeadRows = 8 * 16;  // rows of a block at a time
template <int MODE>
__global__ void __launch_bounds__(NB) k_gnn_head(int N, const float* __restrict__ Hn,
                                                 const bf16* __restrict__ w,
                                                 const bf16* __restrict__ bconst,
                                                 const double* __restrict__ l,
                                                 const double* __restrict__ u,
                                                 const unsigned char* __restrict__ kind, double cmax,
                                                 const float* __restrict__ label, float two_over_n,
                                                 double* __restrict__ pred, float* __restrict__ dH,
                                                 float* __restrict__ part,
                                                 double* __restrict__ loss_part) {
  __shared__ float4 red[16][16];
  __shared__ float redb[16];
  __shared__ double redl[16];
  const int q = threadIdx.x & 15, hw = threadIdx.x >> 4;
  const unsigned mask = 0xffffu << (threadIdx.x & 16);
  const float4 wv = make_float4(bf(w[4 * q]), bf(w[4 * q + 1]), bf(w[4 * q + 2]), bf(w[4 * q + 3]));
  const float b0 = bf(bconst[0]);
  float4 gw = make_float4(0.f, 0.f, 0.f, 0.f);
  float gb = 0.f;
  double ls = 0.0;
  for (long long r0 = ((long long)blockIdx.x * 16 + hw) * 8; r0 < N; r0 += (long long)gridDim.x * kHeadRows) {
    float4 h[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      h[i] = r0 + i < N ? ld4(Hn + (r0 + i) * H + 4 * q) : make_float4(0.f, 0.f, 0.f, 0.f);
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = h[i].x * wv.x + h[i].y * wv.y + h[i].z * wv.z + h[i].w * wv.w;
#pragma unroll
    for (int o = 8, keep = 4; o > 1; o >>= 1, keep >>= 1)
#pragma unroll
      for (int i = 0; i < keep; ++i) {
        const bool up = (q & o) != 0;
        const float send = up ? v[i] : v[i + keep];
        v[i] = (up ? v[i + keep] : v[i]) + __shfl_xor_sync(mask, send, o, 16);
      }
    const float z = v[0] + __shfl_xor_sync(mask, v[0], 1, 16) + b0;
    const long long r = r0 + (q >> 1);
    const bool live = r < N, lead = live && (q & 1) == 0;
    float p = 0.f, dpdz = 0.f, rng = 1.f;
    unsigned char kd = 0;
    if (live && MODE == 0) {
      const double lj = l[r], uj = u[r];
      if (isfinite(lj) && isfinite(uj)) {
        const float s = sigmoidf(z), width = (float)(uj - lj);
        p = (float)lj + width * s;
        dpdz = width * s * (1.f - s);
        rng = width > 0.f ? width : 1.f;
      } else {
        p = z;
        dpdz = 1.f;
      }
    } else if (live) {
      kd = kind[r];
      if (kd == 1) {
        p = z;
        dpdz = 1.f;
      } else {
        p = softplusf(z);
        dpdz = sigmoidf(z);
      }
    }
    if (pred && lead)
      pred[r] = MODE == 0 ? (double)p : (kd == 2 ? -cmax * (double)p : cmax * (double)p);
    if (label) {
      const float e = live ? (p - label[r]) / rng : 0.f;
      const float dz = live ? two_over_n * e / rng * dpdz : 0.f;
      if (lead) {
        ls += (double)e * (double)e;
        gb += dz;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float di = __shfl_sync(mask, dz, 2 * i, 16);
        if (r0 + i >= N) continue;
        gw.x = fmaf(di, h[i].x, gw.x);
        gw.y = fmaf(di, h[i].y, gw.y);
        gw.z = fmaf(di, h[i].z, gw.z);
        gw.w = fmaf(di, h[i].w, gw.w);
        if (dH)
          st4(dH + (r0 + i) * H + 4 * q, make_float4(di * wv.x, di * wv.y, di * wv.z, di * wv.w));
      }
    }
  }
  if (!part) return;
#pragma unroll
  for (int o = 8; o > 1; o >>= 1) {  // (the odd lanes hold none)
    gb += __shfl_xor_sync(mask, gb, o, 16);
    ls += __shfl_xor_sync(mask, ls, o, 16);
  }
  red[hw][q] = gw;
  if (q == 0) {
    redb[hw] = gb;
    redl[hw] = ls;
  }
  __syncthreads();
  if (threadIdx.x < 64) {
    const int qq = threadIdx.x >> 2, c = threadIdx.x & 3;
    float s = 0.f;
    for (int i = 0; i < 16; ++i) {
      const float4 v = red[i][qq];
      s += c == 0 ? v.x : (c == 1 ? v.y : (c == 2 ? v.z : v.w));
    }
    part[(size_t)blockIdx.x * 65 + threadIdx.x] = s;
  } else if (threadIdx.x == 64) {
    float s = 0.f;
    double sl = 0.0;
    for (int i = 0; i < 16; ++i) {
      s += redb[i];
      sl += redl[i];
    }
    part[(size_t)blockIdx.x * 65 + 64] = s;
    loss_part[blockIdx.x] = sl;
  }
}

// ---------------------------------------------------------------- reductions
struct Seg {
  int src, len, dst;
};
// a += x; what the rounding cut off (Knuth's two-sum)
__device__ __forceinline__ float two_sum(float& a, float x) {
  const float s = a + x, b = s - a, cut = (a - (s - b)) + (x - b);
  a = s;
  return cut;
}
// a sum as three float32 numbers: what is cut off from the first goes to the second, from that to
// the third, so that its error is below that of a float64 sum
struct Sum3 {
  float a, b, c;
  __device__ __forceinline__ void add(float x) { c += two_sum(b, two_sum(a, x)); }
};
// grad[dst + e] += scale * sum_b part[b * stride + src + e].  A block takes 32 elements: 32 warps
// each add every 32nd partial of them (one 128-byte line per warp and partial), then one warp adds
// the 32 sums in order.  In float64 the conversions and additions held that pipe (2.5 million of
// each for the 304 partials of a dense layer); the float32 triples cost thirteen additions of the
// other pipe and are no less accurate (a dense layer's partials: 10.5 us cold).  A sum that leaves their range (or is undefined) is added up
// again in float64.
constexpr int kReduceNB = 1024;
__global__ void __launch_bounds__(kReduceNB) k_gnn_reduce(const float* __restrict__ part, int nblk,
                                                          int stride, Seg s0, Seg s1, Seg s2,
                                                          float* __restrict__ grad, float scale) {
  __shared__ Sum3 sh[kReduceNB / 32][32];
  const int total = s0.len + s1.len + s2.len, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  Seg s = s0;
  int i = e;
  if (i >= s0.len) {
    i -= s0.len;
    s = s1;
    if (i >= s1.len) {
      i -= s1.len;
      s = s2;
    }
  }
  const float* p = part + s.src + i;
  Sum3 sum{0.f, 0.f, 0.f};
  if (e < total) {
#pragma unroll 10
    for (int b = w; b < nblk; b += kReduceNB / 32) sum.add(p[(size_t)b * stride]);
  }
  sh[w][lane] = sum;
  __syncthreads();
  if (w == 0 && e < total) {
    for (int k = 1; k < kReduceNB / 32; ++k) {
      const Sum3 v = sh[k][lane];
      sum.add(v.a);
      sum.add(v.b);
      sum.c += v.c;
    }
    double all = (double)sum.a + ((double)sum.b + (double)sum.c);
    if (!isfinite(all)) {
      all = 0.0;
      for (int b = 0; b < nblk; ++b) all += (double)p[(size_t)b * stride];
    }
    grad[s.dst + i] += scale * (float)all;
  }
}

// Sums of NV columns of v[rows][NV] by one block, each thread a strided share and then a
// fixed tree; thread 0 gets them.
template <int NV>
__device__ __forceinline__ void block_columns(const double* __restrict__ v, int rows,
                                              double (&out)[NV]) {
  __shared__ double sh[NB / 32][NV];
  double a[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) a[k] = 0.0;
  for (int b = threadIdx.x; b < rows; b += NB)
#pragma unroll
    for (int k = 0; k < NV; ++k) a[k] += v[(size_t)NV * b + k];
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    for (int o = 16; o > 0; o >>= 1) a[k] += __shfl_xor_sync(0xffffffffu, a[k], o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5][k] = a[k];
  }
  __syncthreads();
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      out[k] = 0.0;
      for (int w = 0; w < NB / 32; ++w) out[k] += sh[w][k];
    }
  __syncthreads();
}

// One block: a single thread adding up to 2,432 partials took 96 us, the block 5 us.
__global__ void __launch_bounds__(NB) k_gnn_loss(const double* __restrict__ lx, int nbx,
                                                 double inv_n, const double* __restrict__ ly,
                                                 int nby, double inv_m, double* __restrict__ out) {
  double sx[1], sy[1];
  block_columns<1>(lx, nbx, sx);
  block_columns<1>(ly, nby, sy);
  if (threadIdx.x == 0) *out = sx[0] * inv_n + sy[0] * inv_m;
}

// ---------------------------------------------------------------- Adam (K14)
__global__ void k_gnn_adam(int P, float* __restrict__ theta, const float* __restrict__ grad,
                           float* __restrict__ m1, float* __restrict__ m2, bf16* __restrict__ w16,
                           float lr, float b1, float b2, float eps, float bc1, float bc2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x) {
    const float g = grad[i];
    const float m = b1 * m1[i] + (1.f - b1) * g;
    const float v = b2 * m2[i] + (1.f - b2) * g * g;
    m1[i] = m;
    m2[i] = v;
    const float th = theta[i] - lr * (m / bc1) / (sqrtf(v / bc2) + eps);
    theta[i] = th;
    w16[i] = __float2bfloat16_rn(th);
  }
}

__global__ void k_gnn_to_bf16(int P, const float* __restrict__ theta, bf16* __restrict__ w16) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x)
    w16[i] = __float2bfloat16_rn(theta[i]);
}

// ---------------------------------------------------------------- start projection + KKT (K15)
// x onto [l, u]; y onto the caller's cone (<= 0 on 'L', >= 0 on 'G', free on 'E').
// A NaN component is replaced by the cold start's (proj(0) and 0).
__global__ void k_start_project(int n, int m, double* __restrict__ x, double* __restrict__ y,
                                const double* __restrict__ l, const double* __restrict__ u,
                                const unsigned char* __restrict__ kind, int cold) {
  const int tot = n + m;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += gridDim.x * blockDim.x) {
    if (i < n) {
      double v = cold ? 0.0 : x[i];
      if (v != v) v = 0.0;
      x[i] = fmin(fmax(v, l[i]), u[i]);
    } else {
      const int r = i - n;
      double v = cold ? 0.0 : y[r];
      if (v != v) v = 0.0;
      y[r] = kind[r] == 2 ? fmin(v, 0.0) : (kind[r] == 0 ? fmax(v, 0.0) : v);
    }
  }
}

__device__ __forceinline__ double warp_sum_d(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// one warp per row; partial per block: [sum r_p^2, sum q y (>=-form), sum q^2]
__global__ void __launch_bounds__(NB) k_kkt_start_rows(int m, const int* __restrict__ ptr,
                                                       const int* __restrict__ col,
                                                       const double* __restrict__ val,
                                                       const double* __restrict__ x,
                                                       const double* __restrict__ y,
                                                       const double* __restrict__ b,
                                                       const unsigned char* __restrict__ kind,
                                                       double* __restrict__ part) {
  __shared__ double red[NB / 32][3];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double s0 = 0.0, s1 = 0.0, s2 = 0.0;
  for (long long i = ((long long)blockIdx.x * NB + threadIdx.x) >> 5; i < m;
       i += (long long)gridDim.x * (NB / 32)) {
    double ax = 0.0;
    for (int k = ptr[i] + lane; k < ptr[i + 1]; k += 32) ax += val[k] * x[col[k]];
    ax = warp_sum_d(ax);
    if (lane == 0) {
      const double s = kind[i] == 2 ? -1.0 : 1.0;
      const double q = s * b[i];
      double rp = q - s * ax;
      if (kind[i] != 1) rp = fmax(rp, 0.0);
      s0 += rp * rp;
      s1 += q * (s * y[i]);
      s2 += q * q;
    }
  }
  if (lane == 0) {
    red[wid][0] = s0;
    red[wid][1] = s1;
    red[wid][2] = s2;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double s = 0.0;
    for (int w = 0; w < NB / 32; ++w) s += red[w][threadIdx.x];
    part[(size_t)blockIdx.x * 3 + threadIdx.x] = s;
  }
}

// one warp per column; partial per block: [sum r_d^2, c^T x, sum c^2, bound terms of the dual]
__global__ void __launch_bounds__(NB) k_kkt_start_cols(int n, const int* __restrict__ ptr,
                                                       const int* __restrict__ row,
                                                       const double* __restrict__ val,
                                                       const double* __restrict__ x,
                                                       const double* __restrict__ y,
                                                       const double* __restrict__ c,
                                                       const double* __restrict__ l,
                                                       const double* __restrict__ u,
                                                       double* __restrict__ part) {
  __shared__ double red[NB / 32][4];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
  for (long long j = ((long long)blockIdx.x * NB + threadIdx.x) >> 5; j < n;
       j += (long long)gridDim.x * (NB / 32)) {
    double aty = 0.0;
    for (int k = ptr[j] + lane; k < ptr[j + 1]; k += 32) aty += val[k] * y[row[k]];
    aty = warp_sum_d(aty);
    if (lane == 0) {
      const double lam = c[j] - aty;
      const double lp = fmax(lam, 0.0), lm = fmax(-lam, 0.0);
      const bool lf = isfinite(l[j]), uf = isfinite(u[j]);
      const double rd = (lf ? 0.0 : lp) + (uf ? 0.0 : lm);
      s0 += rd * rd;
      s1 += c[j] * x[j];
      s2 += c[j] * c[j];
      s3 += (lf ? l[j] * lp : 0.0) - (uf ? u[j] * lm : 0.0);
    }
  }
  if (lane == 0) {
    red[wid][0] = s0;
    red[wid][1] = s1;
    red[wid][2] = s2;
    red[wid][3] = s3;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double s = 0.0;
    for (int w = 0; w < NB / 32; ++w) s += red[w][threadIdx.x];
    part[(size_t)blockIdx.x * 4 + threadIdx.x] = s;
  }
}

// out: rel_primal_res, rel_dual_res, rel_gap, rel_kkt.  One block (a single thread took 193 us
// over the 608 blocks' partials of both passes, the block 12 us).
__global__ void __launch_bounds__(NB) k_kkt_start_final(const double* __restrict__ pr, int nbr,
                                                        const double* __restrict__ pc, int nbc,
                                                        double* __restrict__ out) {
  double r[3], cc[4];
  block_columns<3>(pr, nbr, r);
  block_columns<4>(pc, nbc, cc);
  if (threadIdx.x != 0) return;
  const double relp = sqrt(r[0]) / (1.0 + sqrt(r[2]));
  const double reld = sqrt(cc[0]) / (1.0 + sqrt(cc[2]));
  const double pobj = cc[1], dobj = r[1] + cc[3];
  const double relg = fabs(pobj - dobj) / (1.0 + fabs(pobj) + fabs(dobj));
  out[0] = relp;
  out[1] = reld;
  out[2] = relg;
  out[3] = fmax(relp, fmax(reld, relg));
}

// ---------------------------------------------------------------- host side
template <class T>
cudaError_t dalloc(T** p, size_t count) {
  *p = nullptr;
  if (count == 0) count = 1;
  return cudaMalloc((void**)p, count * sizeof(T));
}

struct LpDev {
  int m = 0, n = 0, nnz = 0;
  int64_t* ptr64 = nullptr;
  int *a_ptr = nullptr, *a_col = nullptr, *t_ptr = nullptr, *t_col = nullptr;
  double *a_val = nullptr, *t_val = nullptr;
  double *b = nullptr, *c = nullptr, *l = nullptr, *u = nullptr;
  char* sense = nullptr;
  unsigned char* kind = nullptr;
  // every array above lives in one allocation (one cudaMalloc and one cudaFree per LP, not
  // one each), followed by `extra` bytes the caller asked build_lp_dev for
  void* arena = nullptr;
  unsigned char* extra = nullptr;
  void release() {
    if (arena) cudaFree(arena);
    *this = LpDev{};
  }
};

// byte offsets of consecutive arrays, each 256-byte aligned
struct Carve {
  size_t off = 0;
  size_t take(size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) / 256 * 256;
    return o;
  }
};

int check_host_lp(const pdlp_csr* A, const double* b, const char* sense, const double* c,
                  const double* l, const double* u) {
  if (!A || !b || !sense || !c || !l || !u)
    if (!(A && A->m == 0 && c && l && u))
      return gfail(PDLP_ERR_INVALID_INPUT, "NULL LP array");
  if (A->m < 0 || A->n < 0 || A->nnz < 0 || A->nnz > 0x7fffffffLL)
    return gfail(PDLP_ERR_INVALID_INPUT, "invalid sizes");
  if (A->nnz > 0 && (!A->col || !A->val)) return gfail(PDLP_ERR_INVALID_INPUT, "NULL CSR arrays");
  if (!A->row_ptr) return gfail(PDLP_ERR_INVALID_INPUT, "NULL row_ptr");
  return PDLP_OK;
}

// Copies a host LP to the device, validates it there and builds int32 CSR of A and A^T.
int build_lp_dev(const pdlp_csr* A, const double* b, const char* sense, const double* c,
                 const double* l, const double* u, cudaStream_t s, LpDev* d,
                 size_t extra_bytes = 0) {
  RTRY(check_host_lp(A, b, sense, c, l, u));
  const int m = A->m, n = A->n, nnz = (int)A->nnz;
  const size_t M = (size_t)m, N = (size_t)n, Z = (size_t)nnz;
  d->m = m;
  d->n = n;
  d->nnz = nnz;
  Carve cv;
  const size_t o_ptr64 = cv.take(8 * (M + 1)), o_aptr = cv.take(4 * (M + 1));
  const size_t o_acol = cv.take(4 * Z), o_aval = cv.take(8 * Z);
  const size_t o_tptr = cv.take(4 * (N + 1)), o_tcol = cv.take(4 * Z), o_tval = cv.take(8 * Z);
  const size_t o_b = cv.take(8 * M), o_c = cv.take(8 * N), o_l = cv.take(8 * N), o_u = cv.take(8 * N);
  const size_t o_sense = cv.take(M), o_kind = cv.take(M), o_err = cv.take(sizeof(int));
  const size_t o_extra = cv.take(extra_bytes);
  GTRY(cudaMalloc(&d->arena, cv.off));
  unsigned char* base = (unsigned char*)d->arena;
  d->ptr64 = (int64_t*)(base + o_ptr64);
  d->a_ptr = (int*)(base + o_aptr);
  d->a_col = (int*)(base + o_acol);
  d->a_val = (double*)(base + o_aval);
  d->t_ptr = (int*)(base + o_tptr);
  d->t_col = (int*)(base + o_tcol);
  d->t_val = (double*)(base + o_tval);
  d->b = (double*)(base + o_b);
  d->c = (double*)(base + o_c);
  d->l = (double*)(base + o_l);
  d->u = (double*)(base + o_u);
  d->sense = (char*)(base + o_sense);
  d->kind = base + o_kind;
  d->extra = extra_bytes ? base + o_extra : nullptr;
  GTRY(cudaMemcpyAsync(d->ptr64, A->row_ptr, sizeof(int64_t) * (m + 1), cudaMemcpyHostToDevice, s));
  if (nnz > 0) {
    GTRY(cudaMemcpyAsync(d->a_col, A->col, sizeof(int) * nnz, cudaMemcpyHostToDevice, s));
    GTRY(cudaMemcpyAsync(d->a_val, A->val, sizeof(double) * nnz, cudaMemcpyHostToDevice, s));
  }
  if (m > 0) {
    GTRY(cudaMemcpyAsync(d->b, b, sizeof(double) * m, cudaMemcpyHostToDevice, s));
    GTRY(cudaMemcpyAsync(d->sense, sense, m, cudaMemcpyHostToDevice, s));
  }
  if (n > 0) {
    GTRY(cudaMemcpyAsync(d->c, c, sizeof(double) * n, cudaMemcpyHostToDevice, s));
    GTRY(cudaMemcpyAsync(d->l, l, sizeof(double) * n, cudaMemcpyHostToDevice, s));
    GTRY(cudaMemcpyAsync(d->u, u, sizeof(double) * n, cudaMemcpyHostToDevice, s));
  }
  // the host row pointer decides every later size: check it before any kernel reads it
  if (A->row_ptr[0] != 0 || A->row_ptr[m] != A->nnz)
    return gfail(PDLP_ERR_INVALID_INPUT, "row_ptr must start at 0 and end at nnz");
  for (int i = 0; i < m; ++i)
    if (A->row_ptr[i + 1] < A->row_ptr[i])
      return gfail(PDLP_ERR_INVALID_INPUT, "row_ptr decreases at row " + std::to_string(i));
  int* d_err = (int*)(base + o_err);
  pdlp::SetupIn in{m, n, (long long)nnz, d->ptr64, d->a_col, d->a_val, d->b, d->sense,
                   d->c, d->l, d->u};
  cudaError_t e = pdlp::setup_validate(in, d_err, s);
  int herr = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  GTRY(e);
  if (herr) {
    std::string why;
    if (herr & pdlp::ERR_ROWPTR) why += " row_ptr";
    if (herr & pdlp::ERR_COL) why += " column index";
    if (herr & pdlp::ERR_NONFINITE) why += " non-finite value";
    if (herr & pdlp::ERR_SENSE) why += " sense";
    if (herr & pdlp::ERR_BOUNDS) why += " bounds (l > u or NaN)";
    return gfail(PDLP_ERR_INVALID_INPUT, "invalid LP:" + why);
  }
  const int G = sm_count() * 8;
  k_ptr32<<<grid_rows((long long)m + 1, NB, G), NB, 0, s>>>(m, d->ptr64, d->a_ptr, d->sense, d->kind);
  GTRY(cudaGetLastError());
  int* tmp = nullptr;
  GTRY(dalloc(&tmp, pdlp::transpose_tmp_ints(m, n, nnz)));
  e = pdlp::setup_transpose(m, n, nnz, d->a_ptr, d->a_col, d->a_val, d->t_ptr, d->t_col, d->t_val,
                            tmp, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(tmp);
  GTRY(e);
  return PDLP_OK;
}

// float64 relative KKT of (x, y) (device, projected in place first unless `cold`
// builds the cold start into them); out[4] on the device
int start_kkt(const LpDev& d, double* x, double* y, int cold, double* part, double* out,
              cudaStream_t s) {
  const int G = sm_count() * 4;
  if (d.n + d.m > 0) {
    k_start_project<<<grid_rows((long long)d.n + d.m, NB, G), NB, 0, s>>>(d.n, d.m, x, y, d.l, d.u,
                                                                          d.kind, cold);
    GTRY(cudaGetLastError());
  }
  const int gr = grid_rows(d.m, NB / 32, G), gc = grid_rows(d.n, NB / 32, G);
  double* pr = part;
  double* pc = part + 3 * (size_t)G;
  if (d.m > 0) {
    k_kkt_start_rows<<<gr, NB, 0, s>>>(d.m, d.a_ptr, d.a_col, d.a_val, x, y, d.b, d.kind, pr);
    GTRY(cudaGetLastError());
  }
  if (d.n > 0) {
    k_kkt_start_cols<<<gc, NB, 0, s>>>(d.n, d.t_ptr, d.t_col, d.t_val, x, y, d.c, d.l, d.u, pc);
    GTRY(cudaGetLastError());
  }
  k_kkt_start_final<<<1, NB, 0, s>>>(pr, d.m > 0 ? gr : 0, pc, d.n > 0 ? gc : 0, out);
  GTRY(cudaGetLastError());
  return PDLP_OK;
}

size_t start_kkt_part_doubles() { return (size_t)7 * sm_count() * 4 + 8; }

}  // namespace

// ---------------------------------------------------------------- model / graph structs
struct gnn_model {
  int device = 0;
  cudaStream_t s = nullptr;
  int P = 0;
  float *theta = nullptr, *grad = nullptr, *m1 = nullptr, *m2 = nullptr;
  bf16* w16 = nullptr;
  long long step = 0;
  // activation scratch, sized for the largest graph seen
  long long cap_n = -1, cap_m = -1;
  float *hv[GNN_LAYERS + 1] = {}, *hc[GNN_LAYERS + 1] = {}, *sv[GNN_LAYERS] = {},
        *sc[GNN_LAYERS] = {};
  float *dhv[2] = {}, *dhc[2] = {}, *dsv = nullptr, *dsc = nullptr;
  double *xpred = nullptr, *ypred = nullptr;
  float* part = nullptr;       // per-block gradient partials
  double* lpart = nullptr;     // per-block loss partials (x head, then y head)
  double* loss = nullptr;      // [1]
  int max_blocks = 0;
};

struct gnn_graph {
  gnn_model* owner = nullptr;
  LpDev d;
  float *inv_deg_r = nullptr, *inv_deg_c = nullptr;
  float *a_v32 = nullptr, *t_v32 = nullptr;  // the values of A and A^T as the layers use them
  float *fv = nullptr, *fc = nullptr;
  float *x_star = nullptr, *y_star = nullptr;  // labels: x*, y* (>=-form) / max|c|
  double cmax = 1.0;
  int has_labels = 0;
};

namespace {

void free_scratch(gnn_model* md) {
  std::vector<void*> ps;
  for (int k = 0; k <= GNN_LAYERS; ++k) {
    ps.push_back(md->hv[k]);
    ps.push_back(md->hc[k]);
    md->hv[k] = md->hc[k] = nullptr;
  }
  for (int k = 0; k < GNN_LAYERS; ++k) {
    ps.push_back(md->sv[k]);
    ps.push_back(md->sc[k]);
    md->sv[k] = md->sc[k] = nullptr;
  }
  for (int k = 0; k < 2; ++k) {
    ps.push_back(md->dhv[k]);
    ps.push_back(md->dhc[k]);
    md->dhv[k] = md->dhc[k] = nullptr;
  }
  ps.push_back(md->dsv);
  ps.push_back(md->dsc);
  ps.push_back(md->xpred);
  ps.push_back(md->ypred);
  md->dsv = md->dsc = nullptr;
  md->xpred = md->ypred = nullptr;
  for (void* p : ps)
    if (p) cudaFree(p);
  md->cap_n = md->cap_m = -1;
}

int ensure_scratch(gnn_model* md, int n, int m) {
  if (n <= md->cap_n && m <= md->cap_m) return PDLP_OK;
  GTRY(cudaStreamSynchronize(md->s));
  const long long cn = std::max<long long>(n, md->cap_n), cm = std::max<long long>(m, md->cap_m);
  free_scratch(md);
  for (int k = 0; k <= GNN_LAYERS; ++k) {
    GTRY(dalloc(&md->hv[k], (size_t)cn * H));
    GTRY(dalloc(&md->hc[k], (size_t)cm * H));
  }
  for (int k = 0; k < GNN_LAYERS; ++k) {
    GTRY(dalloc(&md->sv[k], (size_t)cn * H));
    GTRY(dalloc(&md->sc[k], (size_t)cm * H));
  }
  for (int k = 0; k < 2; ++k) {
    GTRY(dalloc(&md->dhv[k], (size_t)cn * H));
    GTRY(dalloc(&md->dhc[k], (size_t)cm * H));
  }
  GTRY(dalloc(&md->dsv, (size_t)cn * H));
  GTRY(dalloc(&md->dsc, (size_t)cm * H));
  GTRY(dalloc(&md->xpred, (size_t)cn));
  GTRY(dalloc(&md->ypred, (size_t)cm));
  md->cap_n = cn;
  md->cap_m = cm;
  return PDLP_OK;
}

const bf16* W(const gnn_model* md, int off) { return md->w16 + off; }

// Forward pass over a graph: activations stay in the model's scratch.
int forward(gnn_model* md, gnn_graph* g, bool want_pred, bool with_label, bool want_dh) {
  const int n = g->d.n, m = g->d.m;
  RTRY(ensure_scratch(md, n, m));
  cudaStream_t s = md->s;
  const int Gs = sm_count() * 8, Gd = sm_count() * 2;
  if (n > 0) {
    k_gnn_embed<GNN_VAR_FEATURES><<<grid_rows((long long)n, NB / 16, Gs), NB, 0, s>>>(
        n, g->fv, W(md, kOff.W_vin), W(md, kOff.b_vin), md->hv[0]);
    GTRY(cudaGetLastError());
  }
  if (m > 0) {
    k_gnn_embed<GNN_CON_FEATURES><<<grid_rows((long long)m, NB / 16, Gs), NB, 0, s>>>(
        m, g->fc, W(md, kOff.W_cin), W(md, kOff.b_cin), md->hc[0]);
    GTRY(cudaGetLastError());
  }
  for (int k = 0; k < GNN_LAYERS; ++k) {
    if (m > 0) {
      k_gnn_spmm<<<grid_rows((long long)m, NB / 16, kAnyGrid), NB, 0, s>>>(
          m, g->d.a_ptr, g->d.a_col, g->a_v32, g->inv_deg_r, nullptr, md->hv[k], md->sc[k], 0);
      GTRY(cudaGetLastError());
      k_gnn_dense<<<grid_rows((long long)m, 128, Gd), NB, 0, s>>>(
          m, md->hc[k], md->sc[k], W(md, kOff.W_cc[k]), W(md, kOff.W_cv[k]), W(md, kOff.b_c[k]),
          md->hc[k + 1]);
      GTRY(cudaGetLastError());
    }
    if (n > 0) {
      k_gnn_spmm<<<grid_rows((long long)n, NB / 16, kAnyGrid), NB, 0, s>>>(
          n, g->d.t_ptr, g->d.t_col, g->t_v32, g->inv_deg_c, nullptr, md->hc[k + 1], md->sv[k], 0);
      GTRY(cudaGetLastError());
      k_gnn_dense<<<grid_rows((long long)n, 128, Gd), NB, 0, s>>>(
          n, md->hv[k], md->sv[k], W(md, kOff.W_vv[k]), W(md, kOff.W_vc[k]), W(md, kOff.b_v[k]),
          md->hv[k + 1]);
      GTRY(cudaGetLastError());
    }
  }
  const int gx = grid_rows((long long)n, kHeadRows, md->max_blocks);
  const int gy = grid_rows((long long)m, kHeadRows, md->max_blocks);
  if (n > 0) {
    k_gnn_head<0><<<gx, NB, 0, s>>>(n, md->hv[GNN_LAYERS], W(md, kOff.w_x), W(md, kOff.b_x),
                                    g->d.l, g->d.u, nullptr, g->cmax,
                                    with_label ? g->x_star : nullptr, 2.f / (float)n,
                                    want_pred ? md->xpred : nullptr, want_dh ? md->dhv[0] : nullptr,
                                    with_label ? md->part : nullptr, md->lpart);
    GTRY(cudaGetLastError());
  }
  if (m > 0) {
    k_gnn_head<1><<<gy, NB, 0, s>>>(m, md->hc[GNN_LAYERS], W(md, kOff.w_y), W(md, kOff.b_y),
                                    nullptr, nullptr, g->d.kind, g->cmax,
                                    with_label ? g->y_star : nullptr, 2.f / (float)m,
                                    want_pred ? md->ypred : nullptr, want_dh ? md->dhc[0] : nullptr,
                                    with_label ? md->part + (size_t)gx * 65 : nullptr,
                                    md->lpart + md->max_blocks);
    GTRY(cudaGetLastError());
  }
  if (with_label) {
    k_gnn_loss<<<1, NB, 0, s>>>(md->lpart, n > 0 ? gx : 0, n > 0 ? 1.0 / n : 0.0,
                                md->lpart + md->max_blocks, m > 0 ? gy : 0, m > 0 ? 1.0 / m : 0.0,
                                md->loss);
    GTRY(cudaGetLastError());
  }
  return PDLP_OK;
}

int reduce_into(gnn_model* md, int nblk, int stride, Seg a, Seg b, Seg c, float scale) {
  const int total = a.len + b.len + c.len;
  k_gnn_reduce<<<(total + 31) / 32, kReduceNB, 0, md->s>>>(md->part, nblk, stride, a, b, c, md->grad,
                                                        scale);
  GTRY(cudaGetLastError());
  return PDLP_OK;
}

// Forward with labels, then backward; adds scale * gradient into md->grad.
int backward(gnn_model* md, gnn_graph* g, float scale) {
  const int n = g->d.n, m = g->d.m;
  RTRY(ensure_scratch(md, n, m));
  cudaStream_t s = md->s;
  const int Gs = sm_count() * 8, Gb = sm_count() * 2;
  // heads (with dH) -- their partials are reduced right after each head
  RTRY(forward(md, g, false, true, true));
  const int gx = grid_rows((long long)n, kHeadRows, md->max_blocks);
  const int gy = grid_rows((long long)m, kHeadRows, md->max_blocks);
  if (n > 0) RTRY(reduce_into(md, gx, 65, Seg{0, 64, kOff.w_x}, Seg{64, 1, kOff.b_x}, Seg{0, 0, 0}, scale));
  if (m > 0) {
    // the y head's partials sit after the x head's in md->part
    k_gnn_reduce<<<3, kReduceNB, 0, s>>>(md->part + (size_t)gx * 65, gy, 65, Seg{0, 64, kOff.w_y},
                                  Seg{64, 1, kOff.b_y}, Seg{0, 0, 0}, md->grad, scale);
    GTRY(cudaGetLastError());
  }
  int cur = 0;
  for (int k = GNN_LAYERS - 1; k >= 0; --k) {
    const int nxt = cur ^ 1;
    if (n > 0) {
      const int gb = grid_rows((long long)n, 64, Gb);
      k_gnn_dense_bwd<<<gb, NB, kBwdSmem, s>>>(n, md->hv[k], md->sv[k], md->hv[k + 1], md->dhv[cur],
                                               W(md, kOff.W_vv[k]), W(md, kOff.W_vc[k]),
                                               md->dhv[nxt], md->dsv, md->part);
      GTRY(cudaGetLastError());
      RTRY(reduce_into(md, gb, kDensePart, Seg{0, 4096, kOff.W_vv[k]}, Seg{4096, 4096, kOff.W_vc[k]},
                       Seg{8192, 64, kOff.b_v[k]}, scale));
      if (m > 0) {
        // dH_c += C dS_v, C_ij = a_ij / deg_j
        k_gnn_spmm<<<grid_rows((long long)m, NB / 16, kAnyGrid), NB, 0, s>>>(
            m, g->d.a_ptr, g->d.a_col, g->a_v32, nullptr, g->inv_deg_c, md->dsv, md->dhc[cur], 1);
        GTRY(cudaGetLastError());
      }
    }
    if (m > 0) {
      const int gb = grid_rows((long long)m, 64, Gb);
      k_gnn_dense_bwd<<<gb, NB, kBwdSmem, s>>>(m, md->hc[k], md->sc[k], md->hc[k + 1], md->dhc[cur],
                                               W(md, kOff.W_cc[k]), W(md, kOff.W_cv[k]),
                                               md->dhc[nxt], md->dsc, md->part);
      GTRY(cudaGetLastError());
      RTRY(reduce_into(md, gb, kDensePart, Seg{0, 4096, kOff.W_cc[k]}, Seg{4096, 4096, kOff.W_cv[k]},
                       Seg{8192, 64, kOff.b_c[k]}, scale));
      if (n > 0) {
        // dH_v += R^T dS_c, R_ij = a_ij / deg_i
        k_gnn_spmm<<<grid_rows((long long)n, NB / 16, kAnyGrid), NB, 0, s>>>(
            n, g->d.t_ptr, g->d.t_col, g->t_v32, nullptr, g->inv_deg_r, md->dsc, md->dhv[nxt], 1);
        GTRY(cudaGetLastError());
      }
    }
    cur = nxt;
  }
  if (n > 0) {
    const int ge = grid_rows((long long)n, 4, Gs);
    k_gnn_embed_bwd<GNN_VAR_FEATURES><<<ge, NB, 0, s>>>(n, g->fv, md->hv[0], md->dhv[cur], md->part);
    GTRY(cudaGetLastError());
    RTRY(reduce_into(md, ge, (GNN_VAR_FEATURES + 1) * H, Seg{0, GNN_VAR_FEATURES * H, kOff.W_vin},
                     Seg{GNN_VAR_FEATURES * H, H, kOff.b_vin}, Seg{0, 0, 0}, scale));
  }
  if (m > 0) {
    const int ge = grid_rows((long long)m, 4, Gs);
    k_gnn_embed_bwd<GNN_CON_FEATURES><<<ge, NB, 0, s>>>(m, g->fc, md->hc[0], md->dhc[cur], md->part);
    GTRY(cudaGetLastError());
    RTRY(reduce_into(md, ge, (GNN_CON_FEATURES + 1) * H, Seg{0, GNN_CON_FEATURES * H, kOff.W_cin},
                     Seg{GNN_CON_FEATURES * H, H, kOff.b_cin}, Seg{0, 0, 0}, scale));
  }
  return PDLP_OK;
}

int adam_step(gnn_model* md, const gnn_adam* a) {
  md->step += 1;
  const double bc1 = 1.0 - std::pow(a->beta1, (double)md->step);
  const double bc2 = 1.0 - std::pow(a->beta2, (double)md->step);
  k_gnn_adam<<<grid_rows(md->P, NB, sm_count() * 4), NB, 0, md->s>>>(
      md->P, md->theta, md->grad, md->m1, md->m2, md->w16, (float)a->lr, (float)a->beta1,
      (float)a->beta2, (float)a->eps, (float)bc1, (float)bc2);
  GTRY(cudaGetLastError());
  return PDLP_OK;
}

int check_model(const gnn_model* md) {
  if (!md) return gfail(PDLP_ERR_INVALID_INPUT, "NULL model");
  int dev = -1;
  GTRY(cudaGetDevice(&dev));
  if (dev != md->device)
    return gfail(PDLP_ERR_INVALID_INPUT, "the model lives on device " + std::to_string(md->device) +
                                             ", current device is " + std::to_string(dev));
  return PDLP_OK;
}

}  // namespace

// ---------------------------------------------------------------- C ABI
extern "C" {

int64_t gnn_param_count(void) { return kOff.total; }

int gnn_create(uint64_t seed, gnn_model** out) {
  if (!out) return gfail(PDLP_ERR_INVALID_INPUT, "NULL output handle");
  *out = nullptr;
  gnn_model* md = new gnn_model();
  auto bail = [&](int code) {
    gnn_free(md);
    return code;
  };
  cudaError_t e = cudaGetDevice(&md->device);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&md->s, cudaStreamNonBlocking);
  if (e != cudaSuccess) return bail(gfail(PDLP_ERR_CUDA, cudaGetErrorString(e)));
  md->P = kOff.total;
  md->max_blocks = sm_count() * 8;
  if (dalloc(&md->theta, md->P) != cudaSuccess || dalloc(&md->grad, md->P) != cudaSuccess ||
      dalloc(&md->m1, md->P) != cudaSuccess || dalloc(&md->m2, md->P) != cudaSuccess ||
      dalloc(&md->w16, md->P) != cudaSuccess || dalloc(&md->lpart, 2 * (size_t)md->max_blocks) != cudaSuccess ||
      dalloc(&md->loss, 1) != cudaSuccess)
    return bail(gfail(PDLP_ERR_OOM, "model allocation failed"));
  const size_t part_floats = std::max<size_t>((size_t)sm_count() * 2 * kDensePart,
                                              (size_t)2 * md->max_blocks * 65);
  if (dalloc(&md->part, std::max<size_t>(part_floats, (size_t)sm_count() * 8 * 7 * H)) != cudaSuccess)
    return bail(gfail(PDLP_ERR_OOM, "model allocation failed"));
  e = cudaFuncSetAttribute(k_gnn_dense_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwdSmem);
  if (e != cudaSuccess) return bail(gfail(PDLP_ERR_CUDA, cudaGetErrorString(e)));
  // Xavier-uniform from SplitMix64, block by block in parameter order
  std::vector<float> th(md->P, 0.f);
  SplitMix64 r{seed};
  auto fill = [&](int off, int rows, int cols, int fan_in, int fan_out) {
    const double lim = std::sqrt(6.0 / (double)(fan_in + fan_out));
    for (int i = 0; i < rows * cols; ++i) th[off + i] = (float)((2.0 * r.uniform() - 1.0) * lim);
  };
  fill(kOff.W_vin, GNN_VAR_FEATURES, H, GNN_VAR_FEATURES, H);
  fill(kOff.W_cin, GNN_CON_FEATURES, H, GNN_CON_FEATURES, H);
  for (int k = 0; k < GNN_LAYERS; ++k) {
    fill(kOff.W_cc[k], H, H, H, H);
    fill(kOff.W_cv[k], H, H, H, H);
    fill(kOff.W_vv[k], H, H, H, H);
    fill(kOff.W_vc[k], H, H, H, H);
  }
  fill(kOff.w_x, 1, H, H, 1);
  fill(kOff.w_y, 1, H, H, 1);
  int rc = gnn_set_params(md, th.data());
  if (rc != PDLP_OK) return bail(rc);
  e = cudaMemsetAsync(md->grad, 0, sizeof(float) * md->P, md->s);
  if (e == cudaSuccess) e = cudaMemsetAsync(md->m1, 0, sizeof(float) * md->P, md->s);
  if (e == cudaSuccess) e = cudaMemsetAsync(md->m2, 0, sizeof(float) * md->P, md->s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(md->s);
  if (e != cudaSuccess) return bail(gfail(PDLP_ERR_CUDA, cudaGetErrorString(e)));
  *out = md;
  return PDLP_OK;
}

int gnn_free(gnn_model* md) {
  if (!md) return PDLP_OK;
  if (md->s) cudaStreamSynchronize(md->s);
  free_scratch(md);
  void* ps[] = {md->theta, md->grad, md->m1, md->m2, md->w16, md->part, md->lpart, md->loss};
  for (void* p : ps)
    if (p) cudaFree(p);
  if (md->s) cudaStreamDestroy(md->s);
  delete md;
  return PDLP_OK;
}

int gnn_get_params(const gnn_model* md, float* out) {
  RTRY(check_model(md));
  if (!out) return gfail(PDLP_ERR_INVALID_INPUT, "NULL output");
  GTRY(cudaMemcpyAsync(out, md->theta, sizeof(float) * md->P, cudaMemcpyDeviceToHost, md->s));
  GTRY(cudaStreamSynchronize(md->s));
  return PDLP_OK;
}

int gnn_set_params(gnn_model* md, const float* in) {
  RTRY(check_model(md));
  if (!in) return gfail(PDLP_ERR_INVALID_INPUT, "NULL input");
  for (int i = 0; i < md->P; ++i)
    if (!std::isfinite(in[i])) return gfail(PDLP_ERR_INVALID_INPUT, "non-finite parameter");
  GTRY(cudaMemcpyAsync(md->theta, in, sizeof(float) * md->P, cudaMemcpyHostToDevice, md->s));
  k_gnn_to_bf16<<<grid_rows(md->P, NB, sm_count() * 4), NB, 0, md->s>>>(md->P, md->theta, md->w16);
  GTRY(cudaGetLastError());
  GTRY(cudaStreamSynchronize(md->s));
  return PDLP_OK;
}

int gnn_get_grad(const gnn_model* md, float* out) {
  RTRY(check_model(md));
  if (!out) return gfail(PDLP_ERR_INVALID_INPUT, "NULL output");
  GTRY(cudaMemcpyAsync(out, md->grad, sizeof(float) * md->P, cudaMemcpyDeviceToHost, md->s));
  GTRY(cudaStreamSynchronize(md->s));
  return PDLP_OK;
}

int gnn_set_grad(gnn_model* md, const float* in) {
  RTRY(check_model(md));
  if (!in) return gfail(PDLP_ERR_INVALID_INPUT, "NULL input");
  GTRY(cudaMemcpyAsync(md->grad, in, sizeof(float) * md->P, cudaMemcpyHostToDevice, md->s));
  GTRY(cudaStreamSynchronize(md->s));
  return PDLP_OK;
}

int gnn_zero_grad(gnn_model* md) {
  RTRY(check_model(md));
  GTRY(cudaMemsetAsync(md->grad, 0, sizeof(float) * md->P, md->s));
  return PDLP_OK;
}

int gnn_save(const gnn_model* md, const char* path) {
  RTRY(check_model(md));
  if (!path) return gfail(PDLP_ERR_INVALID_INPUT, "NULL path");
  std::vector<float> buf(3 * (size_t)md->P);
  GTRY(cudaMemcpyAsync(buf.data(), md->theta, sizeof(float) * md->P, cudaMemcpyDeviceToHost, md->s));
  GTRY(cudaMemcpyAsync(buf.data() + md->P, md->m1, sizeof(float) * md->P, cudaMemcpyDeviceToHost, md->s));
  GTRY(cudaMemcpyAsync(buf.data() + 2 * (size_t)md->P, md->m2, sizeof(float) * md->P,
                       cudaMemcpyDeviceToHost, md->s));
  GTRY(cudaStreamSynchronize(md->s));
  FILE* f = fopen(path, "wb");
  if (!f) return gfail(PDLP_ERR_INVALID_INPUT, std::string("cannot open ") + path);
  const int64_t hdr[2] = {md->P, md->step};
  bool ok = fwrite("PDLPGNN1", 1, 8, f) == 8 && fwrite(hdr, sizeof(hdr), 1, f) == 1 &&
            fwrite(buf.data(), sizeof(float), buf.size(), f) == buf.size();
  ok = (fclose(f) == 0) && ok;
  return ok ? PDLP_OK : gfail(PDLP_ERR_INVALID_INPUT, std::string("write failed: ") + path);
}

int gnn_load(const char* path, gnn_model** out) {
  if (!path || !out) return gfail(PDLP_ERR_INVALID_INPUT, "NULL argument");
  *out = nullptr;
  FILE* f = fopen(path, "rb");
  if (!f) return gfail(PDLP_ERR_INVALID_INPUT, std::string("cannot open ") + path);
  char magic[8];
  int64_t hdr[2];
  std::vector<float> buf(3 * (size_t)kOff.total);
  bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, "PDLPGNN1", 8) == 0 &&
            fread(hdr, sizeof(hdr), 1, f) == 1 && hdr[0] == kOff.total &&
            fread(buf.data(), sizeof(float), buf.size(), f) == buf.size();
  fclose(f);
  if (!ok) return gfail(PDLP_ERR_INVALID_INPUT, std::string("not a model file of this network: ") + path);
  gnn_model* md = nullptr;
  RTRY(gnn_create(0, &md));
  int rc = gnn_set_params(md, buf.data());
  if (rc == PDLP_OK) {
    cudaError_t e = cudaMemcpyAsync(md->m1, buf.data() + md->P, sizeof(float) * md->P,
                                    cudaMemcpyHostToDevice, md->s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(md->m2, buf.data() + 2 * (size_t)md->P, sizeof(float) * md->P,
                          cudaMemcpyHostToDevice, md->s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(md->s);
    if (e != cudaSuccess) rc = gfail(PDLP_ERR_CUDA, cudaGetErrorString(e));
  }
  if (rc != PDLP_OK) {
    gnn_free(md);
    return rc;
  }
  md->step = hdr[1];
  *out = md;
  return PDLP_OK;
}

int gnn_graph_create(gnn_model* md, const pdlp_csr* A, const double* b, const char* sense,
                     const double* c, const double* l, const double* u, gnn_graph** out) {
  RTRY(check_model(md));
  if (!out) return gfail(PDLP_ERR_INVALID_INPUT, "NULL output handle");
  *out = nullptr;
  gnn_graph* g = new gnn_graph();
  g->owner = md;
  cudaStream_t s = md->s;
  // the graph's own arrays and the feature pass's scratch share the LP's allocation
  const size_t M = A ? (size_t)std::max(A->m, 0) : 0, N = A ? (size_t)std::max(A->n, 0) : 0;
  Carve cv;
  const size_t Z = A ? (size_t)std::max<int64_t>(A->nnz, 0) : 0;
  const size_t o_idr = cv.take(4 * M), o_idc = cv.take(4 * N);
  const size_t o_av = cv.take(4 * Z), o_tv = cv.take(4 * Z);
  const size_t o_fv = cv.take(4 * N * GNN_VAR_FEATURES), o_fc = cv.take(4 * M * GNN_CON_FEATURES);
  const size_t o_nr = cv.take(8 * M), o_nc = cv.take(8 * N), o_mx = cv.take(6 * 8);
  int rc = build_lp_dev(A, b, sense, c, l, u, s, &g->d, cv.off);
  if (rc != PDLP_OK) {
    gnn_graph_free(g);
    return rc;
  }
  const int m = g->d.m, n = g->d.n;
  unsigned char* ex = g->d.extra;
  g->inv_deg_r = (float*)(ex + o_idr);
  g->inv_deg_c = (float*)(ex + o_idc);
  g->a_v32 = (float*)(ex + o_av);
  g->t_v32 = (float*)(ex + o_tv);
  g->fv = (float*)(ex + o_fv);
  g->fc = (float*)(ex + o_fc);
  double* nr = (double*)(ex + o_nr);
  double* nc = (double*)(ex + o_nc);
  unsigned long long* mx = (unsigned long long*)(ex + o_mx);
  unsigned long long hmx[6] = {};
  cudaError_t e = cudaMemsetAsync(mx, 0, 6 * sizeof(unsigned long long), s);
  const int G = sm_count() * 8;
  if (e == cudaSuccess && g->d.nnz > 0) {
    k_gnn_values<<<grid_rows(g->d.nnz, NB, G), NB, 0, s>>>(g->d.nnz, g->d.a_val, g->d.t_val, g->a_v32,
                                                           g->t_v32);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && m > 0) {
    k_gnn_stats<<<grid_rows(m, NB, G), NB, 0, s>>>(m, g->d.a_ptr, g->d.a_val, g->d.b, nr,
                                                   g->inv_deg_r, mx);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && n > 0) {
    k_gnn_stats<<<grid_rows(n, NB, G), NB, 0, s>>>(n, g->d.t_ptr, g->d.t_val, g->d.c, nc,
                                                   g->inv_deg_c, mx + 3);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && n > 0) {
    k_gnn_feat_v<<<grid_rows(n, NB, G), NB, 0, s>>>(n, g->d.t_ptr, g->d.c, g->d.l, g->d.u, nc, mx, g->fv);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && m > 0) {
    k_gnn_feat_c<<<grid_rows(m, NB, G), NB, 0, s>>>(m, g->d.a_ptr, g->d.b, g->d.kind, nr, mx, g->fc);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(hmx, mx, sizeof(hmx), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    gnn_graph_free(g);
    return gfail(e == cudaErrorMemoryAllocation ? PDLP_ERR_OOM : PDLP_ERR_CUDA, cudaGetErrorString(e));
  }
  double cm;
  memcpy(&cm, &hmx[3], sizeof(double));
  g->cmax = std::max(cm, 1e-12);
  *out = g;
  return PDLP_OK;
}

int gnn_graph_set_labels(gnn_graph* g, const double* x_star, const double* y_star) {
  if (!g || !x_star || (!y_star && g->d.m > 0)) return gfail(PDLP_ERR_INVALID_INPUT, "NULL argument");
  RTRY(check_model(g->owner));
  const int n = g->d.n, m = g->d.m;
  std::vector<float> xs(std::max(n, 1)), ys(std::max(m, 1));
  std::vector<char> sense(std::max(m, 1));
  cudaStream_t s = g->owner->s;
  if (m > 0) {
    GTRY(cudaMemcpyAsync(sense.data(), g->d.sense, m, cudaMemcpyDeviceToHost, s));
    GTRY(cudaStreamSynchronize(s));
  }
  for (int j = 0; j < n; ++j) {
    if (!std::isfinite(x_star[j])) return gfail(PDLP_ERR_INVALID_INPUT, "non-finite x label");
    xs[j] = (float)x_star[j];
  }
  for (int i = 0; i < m; ++i) {
    if (!std::isfinite(y_star[i])) return gfail(PDLP_ERR_INVALID_INPUT, "non-finite y label");
    ys[i] = (float)((sense[i] == 'L' ? -y_star[i] : y_star[i]) / g->cmax);
  }
  if (!g->x_star) GTRY(dalloc(&g->x_star, n));
  if (!g->y_star) GTRY(dalloc(&g->y_star, m));
  GTRY(cudaMemcpyAsync(g->x_star, xs.data(), sizeof(float) * n, cudaMemcpyHostToDevice, s));
  GTRY(cudaMemcpyAsync(g->y_star, ys.data(), sizeof(float) * m, cudaMemcpyHostToDevice, s));
  GTRY(cudaStreamSynchronize(s));
  g->has_labels = 1;
  return PDLP_OK;
}

int gnn_graph_features(const gnn_graph* g, float* fv, float* fc) {
  if (!g) return gfail(PDLP_ERR_INVALID_INPUT, "NULL graph");
  RTRY(check_model(g->owner));
  cudaStream_t s = g->owner->s;
  if (fv && g->d.n > 0)
    GTRY(cudaMemcpyAsync(fv, g->fv, sizeof(float) * g->d.n * GNN_VAR_FEATURES, cudaMemcpyDeviceToHost, s));
  if (fc && g->d.m > 0)
    GTRY(cudaMemcpyAsync(fc, g->fc, sizeof(float) * g->d.m * GNN_CON_FEATURES, cudaMemcpyDeviceToHost, s));
  GTRY(cudaStreamSynchronize(s));
  return PDLP_OK;
}

int gnn_graph_free(gnn_graph* g) {
  if (!g) return PDLP_OK;
  // cudaFree waits for the device; the owner is not touched (it may be gone).  The degree
  // and feature arrays live in the LP's allocation; the labels have their own.
  g->d.release();
  void* ps[] = {g->x_star, g->y_star};
  for (void* p : ps)
    if (p) cudaFree(p);
  delete g;
  return PDLP_OK;
}

int gnn_forward(gnn_model* md, gnn_graph* g, double* x_out, double* y_out, double* loss) {
  RTRY(check_model(md));
  if (!g || g->owner != md) return gfail(PDLP_ERR_INVALID_INPUT, "graph does not belong to this model");
  const bool lab = g->has_labels != 0;
  RTRY(forward(md, g, true, lab, false));
  cudaStream_t s = md->s;
  if (x_out && g->d.n > 0)
    GTRY(cudaMemcpyAsync(x_out, md->xpred, sizeof(double) * g->d.n, cudaMemcpyDeviceToHost, s));
  if (y_out && g->d.m > 0)
    GTRY(cudaMemcpyAsync(y_out, md->ypred, sizeof(double) * g->d.m, cudaMemcpyDeviceToHost, s));
  double hl = NAN;
  if (lab) GTRY(cudaMemcpyAsync(&hl, md->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
  GTRY(cudaStreamSynchronize(s));
  if (loss) *loss = hl;
  return PDLP_OK;
}

int gnn_backward(gnn_model* md, gnn_graph* g, double scale, double* loss) {
  RTRY(check_model(md));
  if (!g || g->owner != md) return gfail(PDLP_ERR_INVALID_INPUT, "graph does not belong to this model");
  if (!g->has_labels) return gfail(PDLP_ERR_INVALID_INPUT, "graph has no labels");
  RTRY(backward(md, g, (float)scale));
  double hl = NAN;
  GTRY(cudaMemcpyAsync(&hl, md->loss, sizeof(double), cudaMemcpyDeviceToHost, md->s));
  GTRY(cudaStreamSynchronize(md->s));
  if (loss) *loss = hl;
  return PDLP_OK;
}

int gnn_default_adam(gnn_adam* a) {
  if (!a) return gfail(PDLP_ERR_INVALID_INPUT, "NULL argument");
  a->struct_size = sizeof(gnn_adam);
  a->lr = 1e-3;
  a->beta1 = 0.9;
  a->beta2 = 0.999;
  a->eps = 1e-8;
  return PDLP_OK;
}

int gnn_adam_step(gnn_model* md, const gnn_adam* a) {
  RTRY(check_model(md));
  if (!a || a->struct_size != sizeof(gnn_adam)) return gfail(PDLP_ERR_INVALID_INPUT, "bad gnn_adam");
  if (!(a->lr > 0) || !(a->beta1 >= 0 && a->beta1 < 1) || !(a->beta2 >= 0 && a->beta2 < 1) ||
      !(a->eps >= 0))
    return gfail(PDLP_ERR_INVALID_INPUT, "Adam settings out of range");
  RTRY(adam_step(md, a));
  GTRY(cudaStreamSynchronize(md->s));
  return PDLP_OK;
}

int gnn_default_train(gnn_train_params* t) {
  if (!t) return gfail(PDLP_ERR_INVALID_INPUT, "NULL argument");
  t->struct_size = sizeof(gnn_train_params);
  t->epochs = 30;
  t->batch = 4;
  gnn_default_adam(&t->adam);
  t->lr_decay = 0.95;
  t->seed = 1;
  return PDLP_OK;
}

int gnn_train(gnn_model* md, gnn_graph* const* graphs, int count, const gnn_train_params* t,
              double* epoch_loss) {
  RTRY(check_model(md));
  if (!graphs || count <= 0 || !t || t->struct_size != sizeof(gnn_train_params) || t->epochs < 0 ||
      t->batch <= 0 || t->adam.struct_size != sizeof(gnn_adam))
    return gfail(PDLP_ERR_INVALID_INPUT, "bad training arguments");
  for (int i = 0; i < count; ++i)
    if (!graphs[i] || graphs[i]->owner != md || !graphs[i]->has_labels)
      return gfail(PDLP_ERR_INVALID_INPUT, "graph " + std::to_string(i) + " is missing, foreign or unlabelled");
  double* hist = nullptr;
  GTRY(dalloc(&hist, count));
  std::vector<double> h(count);
  std::vector<int> order(count);
  for (int i = 0; i < count; ++i) order[i] = i;
  SplitMix64 r{t->seed};
  gnn_adam a = t->adam;
  int rc = PDLP_OK;
  for (int ep = 0; ep < t->epochs && rc == PDLP_OK; ++ep) {
    for (int i = count - 1; i > 0; --i) {
      const int j = (int)(r.uniform() * (double)(i + 1));
      std::swap(order[i], order[j]);
    }
    for (int b0 = 0; b0 < count && rc == PDLP_OK; b0 += t->batch) {
      const int b1 = std::min(count, b0 + t->batch);
      if (cudaMemsetAsync(md->grad, 0, sizeof(float) * md->P, md->s) != cudaSuccess) {
        rc = gfail(PDLP_ERR_CUDA, "memset");
        break;
      }
      for (int k = b0; k < b1 && rc == PDLP_OK; ++k) {
        rc = backward(md, graphs[order[k]], 1.0f / (float)(b1 - b0));
        if (rc == PDLP_OK &&
            cudaMemcpyAsync(hist + k, md->loss, sizeof(double), cudaMemcpyDeviceToDevice, md->s) != cudaSuccess)
          rc = gfail(PDLP_ERR_CUDA, "loss copy");
      }
      if (rc == PDLP_OK) rc = adam_step(md, &a);
    }
    if (rc == PDLP_OK) {
      if (cudaMemcpyAsync(h.data(), hist, sizeof(double) * count, cudaMemcpyDeviceToHost, md->s) != cudaSuccess ||
          cudaStreamSynchronize(md->s) != cudaSuccess)
        rc = gfail(PDLP_ERR_CUDA, "loss read-back");
      else if (epoch_loss) {
        double s = 0.0;
        for (double v : h) s += v;
        epoch_loss[ep] = s / count;
      }
    }
    a.lr *= t->lr_decay;
  }
  cudaStreamSynchronize(md->s);
  cudaFree(hist);
  return rc;
}

int pdlp_start_kkt(const pdlp_csr* A, const double* b, const char* sense, const double* c,
                   const double* l, const double* u, const double* x0, const double* y0,
                   double* kkt_out) {
  if (!kkt_out || !x0 || (!y0 && A && A->m > 0)) return gfail(PDLP_ERR_INVALID_INPUT, "NULL argument");
  cudaStream_t s = nullptr;
  GTRY(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  LpDev d;
  double *x = nullptr, *y = nullptr, *part = nullptr, *out = nullptr;
  int rc = build_lp_dev(A, b, sense, c, l, u, s, &d);
  cudaError_t e = cudaSuccess;
  if (rc == PDLP_OK) {
    e = dalloc(&x, d.n);
    if (e == cudaSuccess) e = dalloc(&y, d.m);
    if (e == cudaSuccess) e = dalloc(&part, start_kkt_part_doubles());
    if (e == cudaSuccess) e = dalloc(&out, 4);
    if (e == cudaSuccess && d.n > 0)
      e = cudaMemcpyAsync(x, x0, sizeof(double) * d.n, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && d.m > 0)
      e = cudaMemcpyAsync(y, y0, sizeof(double) * d.m, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) rc = gfail(PDLP_ERR_CUDA, cudaGetErrorString(e));
  }
  if (rc == PDLP_OK) rc = start_kkt(d, x, y, 0, part, out, s);
  if (rc == PDLP_OK) {
    e = cudaMemcpyAsync(kkt_out, out, 4 * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) rc = gfail(PDLP_ERR_CUDA, cudaGetErrorString(e));
  }
  cudaStreamSynchronize(s);
  for (void* p : {(void*)x, (void*)y, (void*)part, (void*)out})
    if (p) cudaFree(p);
  d.release();
  cudaStreamDestroy(s);
  return rc;
}

int pdlp_solve_warm(gnn_model* md, const pdlp_csr* A, const double* b, const char* sense,
                    const double* c, const double* l, const double* u, const pdlp_params* p,
                    double* x_out, double* y_out, pdlp_result* r, gnn_warm_info* info) {
  if (!md)
    return pdlp_solve(A, b, sense, c, l, u, p, nullptr, nullptr, x_out, y_out, r, nullptr);
  RTRY(check_model(md));
  if (!r || !x_out || (!y_out && A && A->m > 0)) return gfail(PDLP_ERR_INVALID_INPUT, "NULL output");
  const auto t0 = std::chrono::steady_clock::now();
  gnn_graph* g = nullptr;
  RTRY(gnn_graph_create(md, A, b, sense, c, l, u, &g));
  cudaStream_t s = md->s;
  const int n = g->d.n, m = g->d.m;
  double *xc = nullptr, *yc = nullptr, *part = nullptr, *kk = nullptr, *xo = nullptr, *yo = nullptr;
  double* buf = nullptr;  // the six scratch vectors in one allocation
  double hk[8] = {};
  int rc = forward(md, g, true, false, false);
  cudaError_t e = cudaSuccess;
  if (rc == PDLP_OK) {
    Carve cv;
    const size_t o_xc = cv.take(8 * (size_t)n), o_yc = cv.take(8 * (size_t)m);
    const size_t o_part = cv.take(8 * start_kkt_part_doubles()), o_kk = cv.take(8 * 8);
    const size_t o_xo = cv.take(8 * (size_t)n), o_yo = cv.take(8 * (size_t)m);
    e = cudaMalloc((void**)&buf, cv.off);
    if (e == cudaSuccess) {
      unsigned char* p0 = (unsigned char*)buf;
      xc = (double*)(p0 + o_xc);
      yc = (double*)(p0 + o_yc);
      part = (double*)(p0 + o_part);
      kk = (double*)(p0 + o_kk);
      xo = (double*)(p0 + o_xo);
      yo = (double*)(p0 + o_yo);
    } else {
      rc = gfail(PDLP_ERR_OOM, cudaGetErrorString(e));
    }
  }
  if (rc == PDLP_OK) rc = start_kkt(g->d, md->xpred, md->ypred, 0, part, kk, s);
  if (rc == PDLP_OK) rc = start_kkt(g->d, xc, yc, 1, part, kk + 4, s);
  if (rc == PDLP_OK) {
    e = cudaMemcpyAsync(hk, kk, sizeof(hk), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) rc = gfail(PDLP_ERR_CUDA, cudaGetErrorString(e));
  }
  const double predict_s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  const bool warm = rc == PDLP_OK && hk[3] < hk[7];
  if (rc == PDLP_OK) {
    // the start point is the one chosen above; the primal weight always comes from the
    // projected prediction's norms (pdlp_solve_hinted)
    pdlp_csr Ad{m, n, (int64_t)g->d.nnz, g->d.ptr64, g->d.a_col, g->d.a_val};
    rc = pdlp::solve_device_hint(&Ad, g->d.b, g->d.sense, g->d.c, g->d.l, g->d.u, p,
                                 warm ? md->xpred : nullptr, warm ? md->ypred : nullptr,
                                 md->xpred, md->ypred, xo, yo, r, s);
  }
  if (rc == PDLP_OK) {
    if (n > 0) e = cudaMemcpyAsync(x_out, xo, sizeof(double) * n, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && m > 0 && y_out)
      e = cudaMemcpyAsync(y_out, yo, sizeof(double) * m, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) rc = gfail(PDLP_ERR_CUDA, cudaGetErrorString(e));
  }
  if (info) {
    info->used_warm = warm ? 1 : 0;
    info->warm_rel_kkt = hk[3];
    info->cold_rel_kkt = hk[7];
    info->predict_s = predict_s;
  }
  cudaStreamSynchronize(s);
  if (buf) cudaFree(buf);
  gnn_graph_free(g);
  return rc;
}

}  // extern "C"
