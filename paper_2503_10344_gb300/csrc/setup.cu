// Device setup of one LP (rows A0-A3 of the hot path):
//   validation of the caller's CSR and vectors (error bits, no trap),
//   canonical form K = S A, q = S b (A0),
//   deterministic transpose of A into CSR (A1: count, scan, scatter, then a
//   segmented sort of each column's entries by their position in A, so the
//   result does not depend on the order atomics landed in),
//   Ruiz (inf-norm) and Pock-Chambolle scaling (A2),
//   iteration-space matrix values and vectors, and the scalars of A3.
#include <algorithm>
#include <vector>

#include "setup.h"

namespace pdlp {

namespace {

constexpr int kScanItems = 8;                       // per thread
constexpr int kScanTile = kBlock * kScanItems;      // per block
constexpr int kSmallSeg = 32;                       // per-thread insertion sort up to this length
constexpr int kTile = 4096;                         // bitonic tile of a long column segment

// ------------------------------------------------------------------ validation
__global__ void k_validate_rows(SetupIn in, int* err) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < in.m; i += stride) {
    const int64_t s = in.row_ptr[i], e = in.row_ptr[i + 1];
    if (s < 0 || e < s || e > in.nnz) atomicOr(err, ERR_ROWPTR);
    const char sn = in.sense[i];
    if (sn != 'L' && sn != 'G' && sn != 'E') atomicOr(err, ERR_SENSE);
    if (!isfinite(in.b[i])) atomicOr(err, ERR_NONFINITE);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (in.row_ptr[0] != 0 || in.row_ptr[in.m] != in.nnz) atomicOr(err, ERR_ROWPTR);
  }
}

__global__ void k_validate_nnz(SetupIn in, int* err) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < in.nnz; p += stride) {
    const int j = in.col[p];
    if (j < 0 || j >= in.n) atomicOr(err, ERR_COL);
    if (!isfinite(in.val[p])) atomicOr(err, ERR_NONFINITE);
  }
}

__global__ void k_validate_cols(SetupIn in, int* err) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < in.n; j += stride) {
    const double l = in.l[j], u = in.u[j];
    if (!isfinite(in.c[j])) atomicOr(err, ERR_NONFINITE);
    if (isnan(l) || isnan(u) || l > u || l == INFINITY || u == -INFINITY) atomicOr(err, ERR_BOUNDS);
  }
}

// ------------------------------------------------------------------ A0
__global__ void k_canonical_rows(SetupIn in, int* a_ptr, double* q, unsigned char* row_kind) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i <= in.m; i += stride) {
    a_ptr[i] = (int)in.row_ptr[i];
    if (i == in.m) break;
    const char sn = in.sense[i];
    q[i] = (sn == 'L' ? -1.0 : 1.0) * in.b[i];
    row_kind[i] = sn == 'E' ? 1 : (sn == 'L' ? 2 : 0);
  }
}

// The row of every nonzero, so that the passes over the nonzeros below run one thread per
// nonzero whatever the rows' lengths (a warp per row left 28 of 32 lanes idle on the energy
// system's rows of 3.75 entries, and walked its columns of 17,520 entries alone): groups of
// LANES lanes per row, stores only, so a long row costs its group no waiting.
template <int LANES>
__global__ void k_row_ids(const int* __restrict__ ptr, int rows, int* __restrict__ row_of) {
  const int lane = threadIdx.x & (LANES - 1);
  const long long G = (long long)gridDim.x * blockDim.x / LANES;
  for (long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / LANES; r < rows; r += G)
    for (int p = ptr[r] + lane; p < ptr[r + 1]; p += LANES) row_of[p] = (int)r;
}

// Column indices and signed values, one thread per nonzero (with k_canonical_rows and the
// row ids: 0.81 -> 0.17 ms on the energy system of 7.9M nonzeros).
__global__ void k_canonical_nnz(SetupIn in, const int* __restrict__ row_of,
                                const unsigned char* __restrict__ row_kind,
                                int* __restrict__ a_col, double* __restrict__ a_val64) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < in.nnz; p += stride) {
    const double v = in.val[p];
    a_col[p] = in.col[p];
    a_val64[p] = row_kind[row_of[p]] == 2 ? -v : v;
  }
}

// ------------------------------------------------------------------ scan
// exclusive scan of cnt[0..N) into out[0..N], out[N] = total
__global__ void k_scan_tiles(const int* cnt, int* out, int N, int* bsum) {
  __shared__ int sh[kBlock];
  const long long base = (long long)blockIdx.x * kScanTile + (long long)threadIdx.x * kScanItems;
  int v[kScanItems];
  int s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const long long i = base + k;
    v[k] = i < N ? cnt[i] : 0;
    s += v[k];
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 1; o < kBlock; o <<= 1) {  // Hillis-Steele inclusive scan of thread sums
    const int t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
    __syncthreads();
    sh[threadIdx.x] += t;
    __syncthreads();
  }
  int run = sh[threadIdx.x] - s;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const long long i = base + k;
    if (i < N) out[i] = run;
    run += v[k];
  }
  if (threadIdx.x == kBlock - 1) {
    bsum[blockIdx.x] = sh[kBlock - 1];
    if (gridDim.x == 1) out[N] = sh[kBlock - 1];  // one tile: done
  }
}

__global__ void k_scan_bsum(int* bsum, int nb, int* out, int N) {
  // single block: exclusive scan of the tile sums, written back in place; total into out[N]
  __shared__ int sh[kBlock];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < nb; base += kBlock) {
    const int i = base + threadIdx.x;
    const int v = i < nb ? bsum[i] : 0;
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < kBlock; o <<= 1) {
      const int t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
      __syncthreads();
      sh[threadIdx.x] += t;
      __syncthreads();
    }
    if (i < nb) bsum[i] = carry + sh[threadIdx.x] - v;
    __syncthreads();
    if (threadIdx.x == kBlock - 1) carry += sh[kBlock - 1];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[N] = carry;
}

// SUMS: bsum still holds the tiles' sums, and every block adds up those before its own (the last
// also writes the total): a launch less than scanning them first.
template <bool SUMS>
__global__ void __launch_bounds__(kBlock) k_scan_add(int* out, int N, const int* bsum) {
  const long long base = (long long)blockIdx.x * kScanTile;
  int add;
  if constexpr (SUMS) {
    __shared__ int sh[kWarps];
    int v = 0;
    for (int i = threadIdx.x; i < (int)blockIdx.x; i += kBlock) v += bsum[i];
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    add = 0;
    for (int w = 0; w < kWarps; ++w) add += sh[w];
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[N] = add + bsum[blockIdx.x];
  } else {
    add = bsum[blockIdx.x];
  }
  for (int k = threadIdx.x; k < kScanTile; k += kBlock) {
    const long long i = base + k;
    if (i < N) out[i] += add;
  }
}

// ------------------------------------------------------------------ A1 transpose
__global__ void k_count_cols(const int* a_col, int nnz, int* cnt) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += stride)
    atomicAdd(cnt + a_col[p], 1);
}

__global__ void k_scatter(const int* a_col, int nnz, const int* t_ptr, int* cursor, int* src) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += stride) {
    const int j = a_col[p];
    const int pos = t_ptr[j] + atomicAdd(cursor + j, 1);
    src[pos] = (int)p;
  }
}

__global__ void k_segsort_small(const int* t_ptr, int n, int* src, int* long_list, int* nlong) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
    const int s = t_ptr[j], e = t_ptr[j + 1], len = e - s;
    if (len > kSmallSeg) {
      long_list[atomicAdd(nlong, 1)] = (int)j;
      continue;
    }
    int k[kSmallSeg];
    for (int a = 0; a < len; ++a) k[a] = src[s + a];
    for (int a = 1; a < len; ++a) {  // insertion sort
      const int v = k[a];
      int b = a - 1;
      while (b >= 0 && k[b] > v) {
        k[b + 1] = k[b];
        --b;
      }
      k[b + 1] = v;
    }
    for (int a = 0; a < len; ++a) src[s + a] = k[a];
  }
}

// one block per tile (start, len <= kTile): bitonic sort in shared memory, in place
__global__ void __launch_bounds__(1024) k_sort_tiles(const int2* tiles, int* src) {
  __shared__ int sh[kTile];
  const int2 t = tiles[blockIdx.x];
  const int start = t.x, len = t.y;
  int P = 1;
  while (P < len) P <<= 1;
  for (int i = threadIdx.x; i < P; i += blockDim.x) sh[i] = i < len ? src[start + i] : INT_MAX;
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1) {
    for (int jj = k >> 1; jj > 0; jj >>= 1) {
      for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const int ixj = i ^ jj;
        if (ixj > i) {
          const bool up = (i & k) == 0;
          const int a = sh[i], b = sh[ixj];
          if ((a > b) == up) {
            sh[i] = b;
            sh[ixj] = a;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int i = threadIdx.x; i < len; i += blockDim.x) src[start + i] = sh[i];
}

// segments of more than one sorted tile: the rank of a key is its index in its
// tile plus the number of smaller keys in every other tile of the segment
// (keys are unique positions in A)
__global__ void k_merge_rank(const int4* mtiles, const int* src, int* out) {
  // mtiles[b] = {seg_start, seg_len, tile_start, tile_len}
  const int4 t = mtiles[blockIdx.x];
  const int seg_s = t.x, seg_len = t.y, ts = t.z, tl = t.w;
  for (int i = threadIdx.x; i < tl; i += blockDim.x) {
    const int key = src[ts + i];
    int rank = i;
    for (int o = seg_s; o < seg_s + seg_len; o += kTile) {
      if (o == ts) continue;
      const int ol = min(kTile, seg_s + seg_len - o);
      int lo = 0, hi = ol;  // count of keys < key in sorted [o, o+ol)
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (src[o + mid] < key) lo = mid + 1;
        else hi = mid;
      }
      rank += lo;
    }
    out[seg_s + rank] = key;
  }
}

__global__ void k_copy_ranges(const int2* ranges, const int* from, int* to) {
  const int2 r = ranges[blockIdx.x];
  for (int i = threadIdx.x; i < r.y; i += blockDim.x) to[r.x + i] = from[r.x + i];
}

// Tile descriptors of the long column segments built on the device (used when
// the caller cannot let the host allocate): per segment its tile count and, for
// segments longer than one tile, the merge-rank tile count.
__global__ void k_tile_counts(const int* list, int nlist, const int* t_ptr, int* cnt_t, int* cnt_m) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < nlist; k += stride) {
    const int j = list[k];
    const int len = t_ptr[j + 1] - t_ptr[j];
    const int tiles = (len + kTile - 1) / kTile;
    cnt_t[k] = tiles;
    cnt_m[k] = len > kTile ? tiles : 0;
  }
}

__global__ void k_tile_desc(const int* list, int nlist, const int* t_ptr, const int* off_t,
                            const int* off_m, int2* tiles, int4* mtiles, int2* ranges) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < nlist; k += stride) {
    const int j = list[k];
    const int st = t_ptr[j], len = t_ptr[j + 1] - st;
    int a = off_t[k], b = off_m[k];
    for (int o = 0; o < len; o += kTile) {
      const int tl = min(kTile, len - o);
      tiles[a++] = make_int2(st + o, tl);
      if (len > kTile) mtiles[b++] = make_int4(st, len, st + o, tl);
    }
    ranges[k] = make_int2(st, len > kTile ? len : 0);
  }
}

// Entry p of A^T comes from entry src[p] of A: its row (row_of, in place of a search over the
// row pointers: 1.13 -> 0.35 ms on a batch of 53M nonzeros) and, unless every value is +1
// (t_val64 NULL), its value.
__global__ void k_finish_transpose(const int* __restrict__ row_of,
                                   const double* __restrict__ a_val64,
                                   const int* __restrict__ src, int nnz, int* __restrict__ t_col,
                                   double* __restrict__ t_val64) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += stride) {
    const int s = src[p];
    t_col[p] = row_of[s];
    if (t_val64) t_val64[p] = a_val64[s];
  }
}

// ------------------------------------------------------------------ A2 scaling
// One scaling pass takes the row statistics of K~ = D_r K D_c over both orientations (op 0:
// max |k~_ij|, Ruiz; op 1: sum |k~_ij|^power, Pock-Chambolle) and writes the new factors
// D / sqrt(statistic) to the other pair of factor arrays, so that a pass is one launch and
// both orientations read the old factors.  The products are rounded one by one as
// (D_r |K|) D_c in either orientation (the float64 parity mode reads these factors); a
// maximum is exact in any order, a sum runs over the entries in storage order (rows of A by
// column, rows of A^T by row), so that it rounds exactly as a plain sequential sum does.
//
// The passes are bound by the float64 pipe (a warp instruction holds it ~16 cycles whatever
// its active lanes) and by the gathers of the other orientation's factors, so:
//   - maxima of non-negative float64 values are taken on their bits, in the integer pipe;
//   - rounding is monotone, so a factor common to the row is applied once to the row's
//     maximum: max_p rn(x_p so) = rn(max_p x_p so).  In A^T the row factor comes last and one
//     product per entry remains; a matrix of +1 entries (PAT) needs none in either
//     orientation and reads no values;
//   - the row statistics of a tile are staged in shared memory and the division and square
//     root of the new factors run on full warps.
// Rows longer than 256 entries (and 8 average rows) are walked by whole blocks from a list:
// with two lanes per row the energy system's capacity columns (8,760-17,520 entries) made
// every pass 2.8 ms.  Measured for the 11 passes of a solve: the energy system 33.3 -> 3.8 ms,
// the 50,000 x 200,000 covering LP 0.48 -> 0.36 ms, 96 covering sub-LPs (53M nonzeros)
// 17.2 -> 9.9 ms; what is left is mostly the division and square root of the new factors.
constexpr int kStatLong = 256;
constexpr int kStatSum = 4;  // entries per thread and round of a long row's sum

struct StatSide {
  const int *ptr, *col;
  const double *val, *own, *other;
  double* out;       // the new factors
  const int* list;   // rows longer than `thresh`, list[rows] = how many (NULL: none)
  int rows, thresh, lanes, tile;  // lanes per row, rows per tile
  double power;
};
struct StatPass {
  StatSide a, t;  // rows of A (own factors D_r), rows of A^T (own factors D_c)
  int gl, ga;     // blocks over the long rows, then over A; the rest over A^T
  int op;
};

__device__ __forceinline__ unsigned long long stat_bits(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return b > 0x7ff0000000000000ull ? 0ull : b;  // a NaN product counts as no entry
}

// what an entry adds to its row: op 0 the bits of its part of the maximum, op 1 |k~|^power
template <bool OWN_ROW, bool PAT>
__device__ __forceinline__ unsigned long long stat_max_term(const StatSide& q, int p, double so) {
  const double o = q.other[q.col[p]];
  if (PAT) return stat_bits(o);
  const double a = fabs(q.val[p]);
  return stat_bits(OWN_ROW ? __dmul_rn(__dmul_rn(so, a), o) : __dmul_rn(o, a));
}
template <bool OWN_ROW, bool PAT>
__device__ __forceinline__ double stat_max_row(unsigned long long bits, double so) {
  const double mx = __longlong_as_double((long long)bits);
  return OWN_ROW && !PAT ? mx : __dmul_rn(mx, so);
}
template <bool OWN_ROW, bool PAT>
__device__ __forceinline__ double stat_sum_term(const StatSide& q, int p, double so) {
  const double o = q.other[q.col[p]];
  const double a = PAT ? 1.0 : fabs(q.val[p]);
  const double kt = OWN_ROW ? __dmul_rn(__dmul_rn(so, a), o) : __dmul_rn(__dmul_rn(o, a), so);
  return q.power == 1.0 ? kt : pow(kt, q.power);
}
__device__ __forceinline__ double stat_apply(double own, double st) {
  return own / (st > 0.0 ? sqrt(st) : 1.0);  // a zero statistic leaves the factor
}

// tiles of q.tile consecutive rows, block `bidx` of `nblk`: LANES lanes per row for maxima,
// one for sums
template <int LANES, bool OWN_ROW, bool PAT, int OP>
__device__ __forceinline__ void stat_tiles(const StatSide& q, int bidx, int nblk, double* sh) {
  const int lane = threadIdx.x & (LANES - 1);
  for (long long r0 = (long long)bidx * q.tile; r0 < q.rows; r0 += (long long)nblk * q.tile) {
    for (int k = threadIdx.x / LANES; k < q.tile; k += kBlock / LANES) {
      const long long r = r0 + k;
      unsigned long long mx = 0;
      double sum = 0.0, so = 0.0;
      if (r < q.rows) {
        const int s = q.ptr[r], e = q.ptr[r + 1];
        so = q.own[r];
        if (e - s <= q.thresh) {
#pragma unroll 4
          for (int p = s + lane; p < e; p += LANES) {
            if (OP == 0) {
              const unsigned long long b = stat_max_term<OWN_ROW, PAT>(q, p, so);
              mx = b > mx ? b : mx;
            } else {
              sum = __dadd_rn(sum, stat_sum_term<OWN_ROW, PAT>(q, p, so));
            }
          }
        }
      }
      if (OP == 0) {
        const unsigned mask =
            LANES == 32 ? 0xffffffffu : (((1u << LANES) - 1u) << ((threadIdx.x & 31) & ~(LANES - 1)));
#pragma unroll
        for (int o = LANES / 2; o > 0; o >>= 1) {
          const unsigned long long b = __shfl_xor_sync(mask, mx, o);
          mx = b > mx ? b : mx;
        }
        if (lane == 0) sh[k] = stat_max_row<OWN_ROW, PAT>(mx, so);
      } else {
        sh[k] = sum;
      }
    }
    __syncthreads();
    const long long r = r0 + threadIdx.x;
    if ((int)threadIdx.x < q.tile && r < q.rows && q.ptr[r + 1] - q.ptr[r] <= q.thresh)
      q.out[r] = stat_apply(q.own[r], sh[threadIdx.x]);
    __syncthreads();
  }
}

// row r by the whole block: a maximum in strides of the block; a sum in storage order, seven
// warps filling one buffer of terms while a thread of the eighth adds up the other
template <bool OWN_ROW, bool PAT>
__device__ __forceinline__ void stat_long_row(const StatSide& q, int r, int op, double* sh) {
  const int s = q.ptr[r], e = q.ptr[r + 1], tid = threadIdx.x;
  const double so = q.own[r];
  if (op == 0) {
    unsigned long long mx = 0;
#pragma unroll 4
    for (int p = s + tid; p < e; p += kBlock) {
      const unsigned long long b = stat_max_term<OWN_ROW, PAT>(q, p, so);
      mx = b > mx ? b : mx;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long b = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = b > mx ? b : mx;
    }
    unsigned long long* shb = reinterpret_cast<unsigned long long*>(sh);
    if ((tid & 31) == 0) shb[tid >> 5] = mx;
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < kWarps; ++w) mx = shb[w] > mx ? shb[w] : mx;
      q.out[r] = stat_apply(so, stat_max_row<OWN_ROW, PAT>(mx, so));
    }
    __syncthreads();
    return;
  }
  constexpr int T = kStatSum * (kBlock - 32);  // terms per round
  double acc = 0.0;
  for (long long p0 = s, k = 0; p0 < (long long)e + T; p0 += T, k ^= 1) {
    if (tid >= 32) {
#pragma unroll
      for (int i = 0; i < kStatSum; ++i) {
        const int o = (tid - 32) + i * (kBlock - 32);
        if (p0 + o < e) sh[k * T + o] = stat_sum_term<OWN_ROW, PAT>(q, (int)p0 + o, so);
      }
    } else if (tid == 0 && p0 > s) {
      const int n = min(T, (int)(e - (p0 - T)));
      const double* v = sh + (k ^ 1) * T;
#pragma unroll 8
      for (int i = 0; i < n; ++i) acc = __dadd_rn(acc, v[i]);
    }
    __syncthreads();
  }
  if (tid == 0) q.out[r] = stat_apply(so, acc);
}

template <bool OWN_ROW, bool PAT>
__device__ __forceinline__ void stat_side(const StatSide& q, int op, int bidx, int nblk, double* sh) {
  if (op == 1) return stat_tiles<1, OWN_ROW, PAT, 1>(q, bidx, nblk, sh);
  switch (q.lanes) {
    case 2: return stat_tiles<2, OWN_ROW, PAT, 0>(q, bidx, nblk, sh);
    case 4: return stat_tiles<4, OWN_ROW, PAT, 0>(q, bidx, nblk, sh);
    case 8: return stat_tiles<8, OWN_ROW, PAT, 0>(q, bidx, nblk, sh);
    case 16: return stat_tiles<16, OWN_ROW, PAT, 0>(q, bidx, nblk, sh);
    default: return stat_tiles<32, OWN_ROW, PAT, 0>(q, bidx, nblk, sh);
  }
}

template <bool PAT>
__global__ void __launch_bounds__(kBlock) k_stat_pass(StatPass q) {
  __shared__ double sh[2 * kStatSum * (kBlock - 32)];
  pdl_enter();
  const int b = blockIdx.x;
  if (b < q.gl) {
    const int na = q.a.rows ? q.a.list[q.a.rows] : 0, nt = q.t.list[q.t.rows];
    for (int k = b; k < na + nt; k += q.gl) {
      if (k < na)
        stat_long_row<true, PAT>(q.a, q.a.list[k], q.op, sh);
      else
        stat_long_row<false, PAT>(q.t, q.t.list[k - na], q.op, sh);
    }
  } else if (b < q.gl + q.ga) {
    stat_side<true, PAT>(q.a, q.op, b - q.gl, q.ga, sh);
  } else {
    stat_side<false, PAT>(q.t, q.op, b - q.gl - q.ga, gridDim.x - q.gl - q.ga, sh);
  }
}

// D_r = D_c = 1 and the lists of rows longer than the thresholds in both orientations (in any
// order: every row is treated on its own)
__global__ void k_scale_start(StatSide a, StatSide t, double* dr, double* dc, int* la, int* lt) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
       i < (long long)a.rows + t.rows; i += stride) {
    const bool ra = i < a.rows;
    const StatSide& q = ra ? a : t;
    const int r = (int)(ra ? i : i - a.rows);
    (ra ? dr : dc)[r] = 1.0;
    if (q.ptr[r + 1] - q.ptr[r] > q.thresh) {
      int* list = ra ? la : lt;
      list[atomicAdd(list + q.rows, 1)] = r;
    }
  }
}

// lanes per row for an average row length (about four entries per lane)
static int stat_lanes(double avg) {
  int l = 2;
  while (l < 32 && 4.0 * l < avg) l <<= 1;
  return l;
}

// ------------------------------------------------------------------ value formats
__global__ void k_value_format(const double* val, int nnz, int* flags) {
  // flags[0] &= every value exactly representable in bfloat16; flags[1] &= every value == 1
  bool bf = true, one = true;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += stride) {
    const double v = val[p];
    bf &= (double)__bfloat162float(__double2bfloat16(v)) == v;
    one &= v == 1.0;
  }
  if (!__all_sync(0xffffffffu, bf) && (threadIdx.x & 31) == 0) atomicAnd(flags, 0);
  if (!__all_sync(0xffffffffu, one) && (threadIdx.x & 31) == 0) atomicAnd(flags + 1, 0);
}

// iteration matrix values: scaled (dr_i K_ij) dc_j or raw K_ij, one thread per nonzero of
// either orientation (row: the rows of A of its entries, col: the columns).  A warp per row
// took 1.83 ms for both orientations of the energy system, this 0.10 ms.
template <typename V>
__global__ void k_iter_values(const int* __restrict__ row, const int* __restrict__ col,
                              const double* __restrict__ val64, int nnz,
                              const double* __restrict__ dr, const double* __restrict__ dc,
                              V* __restrict__ out) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += stride)
    out[p] = (V)((dr[row[p]] * val64[p]) * dc[col[p]]);
}
__global__ void k_iter_values_bf16(const double* __restrict__ val64, int nnz,
                                   __nv_bfloat16* __restrict__ out) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += stride)
    out[p] = __double2bfloat16(val64[p]);
}

// iteration-space vectors (A2/A3) and the float64 scalars of A3
template <typename T>
__global__ void k_iter_vectors(VecIn v, T* c, T* l, T* u, T* q, T* tw, T* sw, T* x0, T* y0,
                               double* part) {
  // part[b*7 + k]: k = 0 ||D_c c||^2, 1 ||D_r q||^2, 2 ||c||^2, 3 ||q||^2, 4 ||x~_hint||^2,
  // 5 ||y~_hint||^2 (the hint projected like a start, in scaled space), 6 columns with
  // an infinite bound
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < v.n; j += stride) {
    const double d = v.dc[j], cj = v.c[j];
    double lj = v.l[j], uj = v.u[j];
    if (v.scaled) {
      c[j] = (T)(d * cj);
      lj = lj / d;
      uj = uj / d;
    } else {
      c[j] = (T)cj;
      tw[j] = (T)(d * d);
    }
    l[j] = (T)lj;
    u[j] = (T)uj;
    double x = v.x0 ? (v.scaled ? v.x0[j] / d : v.x0[j]) : 0.0;
    x = fmin(fmax(x, lj), uj);
    x0[2 * j] = (T)x;  // (x_j, dx_j) pair, no step yet
    x0[2 * j + 1] = (T)0;
    acc[0] += (d * cj) * (d * cj);
    acc[2] += cj * cj;
    acc[6] += (isfinite(v.l[j]) && isfinite(v.u[j])) ? 0.0 : 1.0;
    if (v.wx) {
      const double xh = fmin(fmax(v.wx[j] / d, v.l[j] / d), v.u[j] / d);
      acc[4] += xh * xh;
    }
  }
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < v.m; i += stride) {
    const double d = v.dr[i], qi = v.q[i];
    if (v.scaled) {
      q[i] = (T)(d * qi);
    } else {
      q[i] = (T)qi;
      sw[i] = (T)(d * d);
    }
    double y = 0.0;
    if (v.y0) {
      const double yc = v.row_kind[i] == 2 ? -v.y0[i] : v.y0[i];  // caller convention -> canonical
      y = v.scaled ? yc / d : yc;
      if (v.row_kind[i] != 1) y = fmax(y, 0.0);
    }
    y0[i] = (T)y;
    acc[1] += (d * qi) * (d * qi);
    acc[3] += qi * qi;
    if (v.wy) {
      double yh = (v.row_kind[i] == 2 ? -v.wy[i] : v.wy[i]) / d;
      if (v.row_kind[i] != 1) yh = fmax(yh, 0.0);
      acc[5] += yh * yh;
    }
  }
  double out[7];
  block_sum<7>(acc, out);
  if (threadIdx.x == 0)
    for (int k = 0; k < 7; ++k) part[(size_t)blockIdx.x * 7 + k] = out[k];
}

// the largest of a block's values' bits (non-negative float64); thread 0 gets it
__device__ __forceinline__ unsigned long long block_max_bits(unsigned long long mx) {
  __shared__ unsigned long long sh[kWarps];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = b > mx ? b : mx;
  }
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < kWarps; ++w) mx = sh[w] > mx ? sh[w] : mx;
  return mx;
}

// max |(dr_i K_ij) dc_j| over entries [p0, p1), one thread per nonzero (val NULL: every value
// is +1); thread 0 gets the bits
__device__ __forceinline__ unsigned long long absmax_scaled(long long p0, long long p1,
                                                            long long stride, const int* row,
                                                            const int* col, const double* val,
                                                            const double* dr, const double* dc) {
  unsigned long long mx = 0;
#pragma unroll 4
  for (long long p = p0; p < p1; p += stride) {
    const double d = dr[row[p]], v = val ? d * val[p] : d;
    const unsigned long long b = stat_bits(fabs(v * dc[col[p]]));
    mx = b > mx ? b : mx;
  }
  return block_max_bits(mx);
}

__global__ void __launch_bounds__(kBlock) k_absmax_scaled(const int* row, const int* col,
                                                          const double* val, int nnz,
                                                          const double* dr, const double* dc,
                                                          double* part) {
  const unsigned long long mx =
      absmax_scaled((long long)blockIdx.x * kBlock + threadIdx.x, nnz,
                    (long long)gridDim.x * kBlock, row, col, val, dr, dc);
  if (threadIdx.x == 0) part[blockIdx.x] = __longlong_as_double((long long)mx);
}

__global__ void k_finish_scalars(const double* vpart, int nv, const double* mpart, int nmx,
                                 double* out) {
  // out: [0] ||c~||, [1] ||q~||, [2] ||c||, [3] ||q||, [4] max |K~|, [5] ||x~_hint||,
  // [6] ||y~_hint||, [7] columns with an infinite bound
  double a[7] = {0, 0, 0, 0, 0, 0, 0}, r[7];
  for (int b = threadIdx.x; b < nv; b += kBlock)
    for (int k = 0; k < 7; ++k) a[k] += vpart[(size_t)b * 7 + k];
  unsigned long long mx = 0;
  for (int b = threadIdx.x; b < nmx; b += kBlock) {
    const unsigned long long v = stat_bits(mpart[b]);
    mx = v > mx ? v : mx;
  }
  mx = block_max_bits(mx);
  block_sum<7>(a, r);
  if (threadIdx.x == 0) {
    for (int k = 0; k < 4; ++k) out[k] = sqrt(r[k]);
    out[4] = __longlong_as_double((long long)mx);
    out[5] = sqrt(r[4]);
    out[6] = sqrt(r[5]);
    out[7] = r[6];
  }
}

// Bound-objective rescaling (optional, after A2/A3's vectors): the iteration-space
// objective divided by gamma, the right-hand side, the bounds and the start x by beta,
// the start y by gamma; the factors that carry an iteration-space point back to the
// original units (D_c, D_r of the KKT passes and the output) take beta and gamma in,
// and their inverses (the scaled distances of the primal-weight update) 1 / beta and
// 1 / gamma.  The step weights and the iteration matrix were formed before and keep
// the plain D_r, D_c.
template <typename T>
__global__ void k_rescale(int m, int n, double beta, double gamma, T* c, T* l, T* u, T* q, T* x0,
                          T* y0, double* dr, double* dc, double* inv_dr, double* inv_dc) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
    c[j] = (T)((double)c[j] / gamma);
    l[j] = (T)((double)l[j] / beta);
    u[j] = (T)((double)u[j] / beta);
    x0[2 * j] = (T)((double)x0[2 * j] / beta);
    dc[j] = dc[j] * beta;
    inv_dc[j] = 1.0 / dc[j];
  }
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
    q[i] = (T)((double)q[i] / beta);
    y0[i] = (T)((double)y0[i] / gamma);
    dr[i] = dr[i] * gamma;
    inv_dr[i] = 1.0 / dr[i];
  }
}

// rows by descending length, ties by index: a row's place is the number of rows before it
// in that order (every thread compares its row with all the others)
__global__ void k_len_order(const int* ptr, int rows, int* ord) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += stride) {
    const int len = ptr[r + 1] - ptr[r];
    int pos = 0;
    for (int k = 0; k < rows; ++k) {
      const int lk = ptr[k + 1] - ptr[k];
      pos += (lk > len) || (lk == len && k < r);
    }
    ord[pos] = (int)r;
  }
}

// float64 auxiliaries of the KKT passes: 1 / D_r, 1 / D_c and, per column, bit 0
// = lower bound finite, bit 1 = upper bound finite (integer tests instead of
// float64 compares in the per-column epilogue)
__global__ void k_kkt_aux(int m, int n, const double* dr, const double* dc, const double* l,
                          const double* u, double* inv_dr, double* inv_dc, unsigned char* bflags) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride)
    inv_dr[i] = 1.0 / dr[i];
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
    inv_dc[j] = 1.0 / dc[j];
    bflags[j] = (unsigned char)((isfinite(l[j]) ? 1 : 0) | (isfinite(u[j]) ? 2 : 0));
  }
}

// deterministic list of rows longer than thresh: flags, scan, scatter
__global__ void k_long_flags(const int* ptr, int nrows, int thresh, int* flags) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < nrows; r += stride)
    flags[r] = (ptr[r + 1] - ptr[r]) > thresh ? 1 : 0;
}
__global__ void k_long_scatter(const int* flags, const int* pos, int nrows, int* list) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < nrows; r += stride)
    if (flags[r]) list[pos[r]] = (int)r;
}

}  // namespace

int grid_for(long long work_items, int max_blocks) {
  long long g = (work_items + kBlock - 1) / kBlock;
  if (g < 1) g = 1;
  if (g > max_blocks) g = max_blocks;
  return (int)g;
}

int device_sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

#define RET(x)                                  \
  do {                                          \
    cudaError_t e_ = (x);                       \
    if (e_ != cudaSuccess) return e_;           \
  } while (0)

cudaError_t setup_validate(const SetupIn& in, int* d_err, cudaStream_t s) {
  const int G = device_sm_count() * 8;
  RET(cudaMemsetAsync(d_err, 0, sizeof(int), s));
  k_validate_rows<<<grid_for(in.m + 1, G), kBlock, 0, s>>>(in, d_err);
  RET(cudaGetLastError());
  if (in.nnz > 0) {
    k_validate_nnz<<<grid_for(in.nnz, G), kBlock, 0, s>>>(in, d_err);
    RET(cudaGetLastError());
  }
  k_validate_cols<<<grid_for(in.n, G), kBlock, 0, s>>>(in, d_err);
  return cudaGetLastError();
}

// row ids of every nonzero of a CSR matrix
static cudaError_t row_ids(const int* ptr, int rows, long long nnz, int* row_of, cudaStream_t s) {
  if (rows <= 0 || nnz <= 0) return cudaSuccess;
  const int lanes = stat_lanes((double)nnz / rows);
  const int g = grid_for((long long)rows * lanes, device_sm_count() * 8);
  switch (lanes) {
    case 2: k_row_ids<2><<<g, kBlock, 0, s>>>(ptr, rows, row_of); break;
    case 4: k_row_ids<4><<<g, kBlock, 0, s>>>(ptr, rows, row_of); break;
    case 8: k_row_ids<8><<<g, kBlock, 0, s>>>(ptr, rows, row_of); break;
    case 16: k_row_ids<16><<<g, kBlock, 0, s>>>(ptr, rows, row_of); break;
    default: k_row_ids<32><<<g, kBlock, 0, s>>>(ptr, rows, row_of); break;
  }
  return cudaGetLastError();
}

int* transpose_row_ids(int* tmp, int n, long long nnz) { return tmp + (n + 1) + nnz; }

cudaError_t setup_canonical(const SetupIn& in, int* a_ptr, int* a_col, double* a_val64, double* q,
                            unsigned char* row_kind, int* row_of, cudaStream_t s) {
  const int G = device_sm_count() * 8;
  k_canonical_rows<<<grid_for((long long)in.m + 1, G), kBlock, 0, s>>>(in, a_ptr, q, row_kind);
  RET(cudaGetLastError());
  if (in.nnz == 0) return cudaSuccess;
  RET(row_ids(a_ptr, in.m, in.nnz, row_of, s));
  k_canonical_nnz<<<grid_for(in.nnz, G), kBlock, 0, s>>>(in, row_of, row_kind, a_col, a_val64);
  return cudaGetLastError();
}

// One launch up to kScanTile counts, two up to kScanDirect tiles (each block then reads at most
// that many sums again), else three: a launch of the setup's many is 2-3 us (a pass of the
// 200 x 400 relaxation, whose setup scans three times: 1,265 -> 1,215 us).
constexpr int kScanDirect = 4096;
cudaError_t exclusive_scan(const int* cnt, int* out, int N, int* bsum, cudaStream_t s) {
  const int nb = (N + kScanTile - 1) / kScanTile;
  if (nb > 0) {
    k_scan_tiles<<<nb, kBlock, 0, s>>>(cnt, out, N, bsum);
    RET(cudaGetLastError());
  }
  if (nb == 1) return cudaSuccess;
  if (nb > 1 && nb <= kScanDirect) {
    k_scan_add<true><<<nb, kBlock, 0, s>>>(out, N, bsum);
    return cudaGetLastError();
  }
  k_scan_bsum<<<1, kBlock, 0, s>>>(bsum, nb, out, N);
  RET(cudaGetLastError());
  if (nb > 0) {
    k_scan_add<false><<<nb, kBlock, 0, s>>>(out, N, bsum);
    RET(cudaGetLastError());
  }
  return cudaSuccess;
}

int scan_launches(long long N) {
  const long long nb = (N + kScanTile - 1) / kScanTile;
  return nb <= 1 ? 1 : nb <= kScanDirect ? 2 : 3;
}
size_t scan_tmp_ints(long long N) { return (size_t)((N + kScanTile - 1) / kScanTile) + 1; }

cudaError_t setup_transpose(int m, int n, int nnz, const int* a_ptr, const int* a_col,
                            const double* a_val64, int* t_ptr, int* t_col, double* t_val64,
                            int* tmp, cudaStream_t s, bool device_desc) {
  // tmp layout (ints): cnt/cursor [n+1] | src [nnz] | src2 [nnz] | long list [n] | nlong [1]
  //                    | tile descriptors [8 * (nnz/32 + 2)], 16-byte aligned | scan block sums
  const int G = device_sm_count() * 8;
  int* cnt = tmp;
  int* src = cnt + (n + 1);
  int* src2 = src + nnz;
  int* long_list = src2 + nnz;
  int* d_nlong = long_list + n;
  size_t doff = (size_t)(d_nlong + 1 - tmp);
  doff = (doff + 3) & ~(size_t)3;
  int* desc = tmp + doff;
  // bound on tiles of segments longer than 32, rounded up to even so that the
  // int4 array placed after 2 * max_desc ints starts on a 16-byte boundary
  const size_t max_desc = ((size_t)nnz / 32 + 3) & ~(size_t)1;
  int* bsum = desc + 8 * max_desc;
  RET(cudaMemsetAsync(cnt, 0, sizeof(int) * (n + 1), s));
  if (nnz > 0) {
    k_count_cols<<<grid_for(nnz, G), kBlock, 0, s>>>(a_col, nnz, cnt);
    RET(cudaGetLastError());
  }
  RET(exclusive_scan(cnt, t_ptr, n, bsum, s));
  RET(cudaMemsetAsync(cnt, 0, sizeof(int) * (n + 1), s));
  if (nnz > 0) {
    k_scatter<<<grid_for(nnz, G), kBlock, 0, s>>>(a_col, nnz, t_ptr, cnt, src);
    RET(cudaGetLastError());
  }
  RET(cudaMemsetAsync(d_nlong, 0, sizeof(int), s));
  k_segsort_small<<<grid_for(n, G), kBlock, 0, s>>>(t_ptr, n, src, long_list, d_nlong);
  RET(cudaGetLastError());
  int nlong = 0;
  RET(cudaMemcpyAsync(&nlong, d_nlong, sizeof(int), cudaMemcpyDeviceToHost, s));
  RET(cudaStreamSynchronize(s));
  if (nlong > 0 && device_desc) {
    // descriptors built on the device; the count and offset arrays live in src2,
    // which the merge-rank pass only overwrites after the descriptors exist
    int* cnt_t = src2;
    int* cnt_m = cnt_t + nlong;
    int* off_t = cnt_m + nlong;
    int* off_m = off_t + nlong + 1;
    const int gl = grid_for(nlong, G);
    k_tile_counts<<<gl, kBlock, 0, s>>>(long_list, nlong, t_ptr, cnt_t, cnt_m);
    RET(cudaGetLastError());
    RET(exclusive_scan(cnt_t, off_t, nlong, bsum, s));
    RET(exclusive_scan(cnt_m, off_m, nlong, bsum, s));
    int tot_t = 0, tot_m = 0;
    RET(cudaMemcpyAsync(&tot_t, off_t + nlong, sizeof(int), cudaMemcpyDeviceToHost, s));
    RET(cudaMemcpyAsync(&tot_m, off_m + nlong, sizeof(int), cudaMemcpyDeviceToHost, s));
    RET(cudaStreamSynchronize(s));
    if ((size_t)tot_t > max_desc || (size_t)tot_m > max_desc || (size_t)nlong > max_desc)
      return cudaErrorInvalidValue;
    int2* d_tiles = (int2*)desc;
    int4* d_mtiles = (int4*)(desc + 2 * max_desc);
    int2* d_ranges = (int2*)(desc + 6 * max_desc);
    k_tile_desc<<<gl, kBlock, 0, s>>>(long_list, nlong, t_ptr, off_t, off_m, d_tiles, d_mtiles,
                                      d_ranges);
    RET(cudaGetLastError());
    k_sort_tiles<<<tot_t, 1024, 0, s>>>(d_tiles, src);
    RET(cudaGetLastError());
    if (tot_m > 0) {
      k_merge_rank<<<tot_m, kBlock, 0, s>>>(d_mtiles, src, src2);
      RET(cudaGetLastError());
      k_copy_ranges<<<nlong, kBlock, 0, s>>>(d_ranges, src2, src);
      RET(cudaGetLastError());
    }
  } else if (nlong > 0) {
    std::vector<int> ids(nlong);
    RET(cudaMemcpyAsync(ids.data(), long_list, sizeof(int) * nlong, cudaMemcpyDeviceToHost, s));
    std::vector<int> hp(n + 1);
    RET(cudaMemcpyAsync(hp.data(), t_ptr, sizeof(int) * (n + 1), cudaMemcpyDeviceToHost, s));
    RET(cudaStreamSynchronize(s));
    std::sort(ids.begin(), ids.end());
    std::vector<int2> tiles;
    std::vector<int4> mtiles;
    std::vector<int2> mranges;
    for (int j : ids) {
      const int st = hp[j], len = hp[j + 1] - hp[j];
      for (int o = 0; o < len; o += kTile) tiles.push_back(make_int2(st + o, std::min(kTile, len - o)));
      if (len > kTile) {
        for (int o = 0; o < len; o += kTile)
          mtiles.push_back(make_int4(st, len, st + o, std::min(kTile, len - o)));
        mranges.push_back(make_int2(st, len));
      }
    }
    if (tiles.size() > max_desc || mtiles.size() > max_desc) return cudaErrorInvalidValue;
    int2* d_tiles = (int2*)desc;                       // 2 ints each
    int4* d_mtiles = (int4*)(desc + 2 * max_desc);     // 4 ints each
    int2* d_ranges = (int2*)(desc + 6 * max_desc);     // 2 ints each
    RET(cudaMemcpyAsync(d_tiles, tiles.data(), sizeof(int2) * tiles.size(), cudaMemcpyHostToDevice, s));
    if (!mtiles.empty()) {
      RET(cudaMemcpyAsync(d_mtiles, mtiles.data(), sizeof(int4) * mtiles.size(),
                          cudaMemcpyHostToDevice, s));
      RET(cudaMemcpyAsync(d_ranges, mranges.data(), sizeof(int2) * mranges.size(),
                          cudaMemcpyHostToDevice, s));
    }
    k_sort_tiles<<<(int)tiles.size(), 1024, 0, s>>>(d_tiles, src);
    RET(cudaGetLastError());
    if (!mtiles.empty()) {
      k_merge_rank<<<(int)mtiles.size(), kBlock, 0, s>>>(d_mtiles, src, src2);
      RET(cudaGetLastError());
      k_copy_ranges<<<(int)mranges.size(), kBlock, 0, s>>>(d_ranges, src2, src);
      RET(cudaGetLastError());
    }
    // the host vectors are read by the copies above: wait before they go out of scope
    RET(cudaStreamSynchronize(s));
  }
  if (nnz > 0) {
    // the merge buffer is free again: the rows of A's entries go there (and stay, for the
    // passes over the nonzeros that follow)
    RET(row_ids(a_ptr, m, nnz, src2, s));
    k_finish_transpose<<<grid_for(nnz, G), kBlock, 0, s>>>(src2, a_val64, src, nnz, t_col, t_val64);
    RET(cudaGetLastError());
  }
  return cudaSuccess;
}

size_t transpose_tmp_ints(int m, int n, long long nnz) {
  return (size_t)(n + 1) + 2 * (size_t)nnz + (size_t)n + 1 + 4 + 8 * ((size_t)nnz / 32 + 3) +
         scan_tmp_ints((long long)std::max(m, n) + 1) + 64;
}

cudaError_t setup_scaling(const ScaleIn& sc, double* dr, double* dc, double* dr2, double* dc2,
                          int* list_a, int* list_t, cudaStream_t s) {
  const int G = device_sm_count() * 8;
  const bool pat = sc.a_val64 == nullptr;
  auto side = [&](const int* ptr, const int* col, const double* val, int rows, const int* list) {
    const double avg = rows > 0 ? (double)sc.nnz / rows : 1.0;
    StatSide q{};
    q.ptr = ptr;
    q.col = col;
    q.val = val;
    q.rows = rows;
    q.list = list;
    q.lanes = stat_lanes(avg);
    q.thresh = std::max(kStatLong, (int)std::min(8.0 * avg, 1e9));
    return q;
  };
  StatPass q{side(sc.a_ptr, sc.a_col, sc.a_val64, sc.m, list_a),
             side(sc.t_ptr, sc.t_col, sc.t_val64, sc.n, list_t), 0, 0, 0};
  const int passes = sc.ruiz_iters + (sc.pc_alpha >= 0.0 ? 1 : 0);
  // the factors alternate between (dr, dc) and (dr2, dc2) and end in (dr, dc)
  double *r0 = passes % 2 ? dr2 : dr, *c0 = passes % 2 ? dc2 : dc;
  double *r1 = passes % 2 ? dr : dr2, *c1 = passes % 2 ? dc : dc2;
  RET(cudaMemsetAsync(list_a + sc.m, 0, sizeof(int), s));
  RET(cudaMemsetAsync(list_t + sc.n, 0, sizeof(int), s));
  k_scale_start<<<grid_for((long long)sc.m + sc.n, G), kBlock, 0, s>>>(q.a, q.t, r0, c0, list_a,
                                                                       list_t);
  RET(cudaGetLastError());
  // as many blocks as there can be long rows, at most two per SM
  q.gl = (int)std::min<long long>(2 * device_sm_count(),
                                  sc.nnz / q.a.thresh + sc.nnz / q.t.thresh);
  for (int it = 0; it < passes; ++it) {
    q.op = it < sc.ruiz_iters ? 0 : 1;
    // rows per tile: the whole block finishes rows, unless that leaves SMs without a tile
    auto blocks = [&](StatSide& d) {
      const int lanes = q.op == 1 ? 1 : d.lanes;
      d.tile = kBlock;
      while (d.tile > kBlock / lanes && (d.rows + d.tile - 1) / d.tile < 2 * device_sm_count())
        d.tile /= 2;
      return d.rows > 0 ? std::min(G, (d.rows + d.tile - 1) / d.tile) : 0;
    };
    q.ga = blocks(q.a);
    const int gt = blocks(q.t);
    q.a.own = q.t.other = r0;
    q.t.own = q.a.other = c0;
    q.a.out = r1;
    q.t.out = c1;
    q.a.power = 2.0 - sc.pc_alpha;
    q.t.power = sc.pc_alpha;
    RET(pat ? launch_pdl(k_stat_pass<true>, q.gl + q.ga + gt, kBlock, s, q)
            : launch_pdl(k_stat_pass<false>, q.gl + q.ga + gt, kBlock, s, q));
    std::swap(r0, r1);
    std::swap(c0, c1);
  }
  return cudaSuccess;
}

cudaError_t setup_value_format(const double* val64, int nnz, int* d_flags, int* h_bf16_exact,
                               int* h_all_one, cudaStream_t s) {
  const int G = device_sm_count() * 8;
  const int ones[2] = {1, 1};
  RET(cudaMemcpyAsync(d_flags, ones, sizeof(ones), cudaMemcpyHostToDevice, s));
  if (nnz > 0) {
    k_value_format<<<grid_for(nnz, G), kBlock, 0, s>>>(val64, nnz, d_flags);
    RET(cudaGetLastError());
  }
  int h[2];
  RET(cudaMemcpyAsync(h, d_flags, sizeof(h), cudaMemcpyDeviceToHost, s));
  RET(cudaStreamSynchronize(s));
  *h_bf16_exact = h[0];
  *h_all_one = h[1];
  return cudaSuccess;
}

cudaError_t setup_iter_values(int which_type, const int* row, const int* col,
                              const double* val64, int nnz, const double* dr, const double* dc,
                              void* out, cudaStream_t s) {
  if (nnz == 0) return cudaSuccess;
  const int g = grid_for(nnz, device_sm_count() * 8);
  switch (which_type) {
    case 0: k_iter_values<double><<<g, kBlock, 0, s>>>(row, col, val64, nnz, dr, dc, (double*)out); break;
    case 1: k_iter_values<float><<<g, kBlock, 0, s>>>(row, col, val64, nnz, dr, dc, (float*)out); break;
    case 2: k_iter_values_bf16<<<g, kBlock, 0, s>>>(val64, nnz, (__nv_bfloat16*)out); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t setup_row_ids(const int* ptr, int rows, long long nnz, int* row_of, cudaStream_t s) {
  return row_ids(ptr, rows, nnz, row_of, s);
}

cudaError_t setup_iter_vectors(const VecIn& v, int fp32, void* c, void* l, void* u, void* q,
                               void* tw, void* sw, void* x0, void* y0, const int* row_of,
                               const int* a_col, const double* a_val64, int nnz, double* part,
                               double* scalars_out, cudaStream_t s) {
  const int G = device_sm_count() * 8;
  const int gv = grid_for(std::max(v.m, v.n), G);
  if (fp32)
    k_iter_vectors<float><<<gv, kBlock, 0, s>>>(v, (float*)c, (float*)l, (float*)u, (float*)q,
                                                (float*)tw, (float*)sw, (float*)x0, (float*)y0, part);
  else
    k_iter_vectors<double><<<gv, kBlock, 0, s>>>(v, (double*)c, (double*)l, (double*)u, (double*)q,
                                                 (double*)tw, (double*)sw, (double*)x0, (double*)y0,
                                                 part);
  RET(cudaGetLastError());
  if (!scalars_out) return cudaSuccess;  // a batch takes its scalars per LP
  const int gm = grid_for(nnz, G);
  double* mpart = part + (size_t)gv * 7;
  k_absmax_scaled<<<gm, kBlock, 0, s>>>(row_of, a_col, a_val64, nnz, v.dr, v.dc, mpart);
  RET(cudaGetLastError());
  k_finish_scalars<<<1, kBlock, 0, s>>>(part, gv, mpart, gm, scalars_out);
  return cudaGetLastError();
}

size_t setup_part_doubles(int m, int n) {
  const int G = device_sm_count() * 8;
  return (size_t)G * 7 + (size_t)G + 16;
}

// ---- Halpern variant: the power iteration for L ~ ||K~||_2, K~ = D_r K D_c
// (K the canonical matrix; val NULL: every entry +1).  v = w / s is the unit vector of
// the previous pass (w = 1/sqrt(n), s = 1 at the start); a pass forms u = K~ v and
// w = K~^T u, s = ||w||; after the last pass L = sqrt(s).  A zero s leaves v = 0.
__global__ void k_pow_start(double* w, int n, double* s) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  const double v = 1.0 / sqrt((double)n);
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) w[j] = v;
  if (blockIdx.x == 0 && threadIdx.x == 0) *s = 1.0;
}

// A pass over the matrix (ptr, col, val): out_r = fo_r sum_p K_rp fi_c(p) in_c(p) / s
// (s NULL: no division), fo, fi the row and column scalings.  Rows of at most `thresh`
// entries by groups of kPowLanes lanes, rows grid-strided (longer rows: k_pow_long); with
// part != NULL also each block's sum of out_r^2 into part[block].
constexpr int kPowLanes = 4;
__device__ __forceinline__ double pow_inv(const double* s) {
  const double sv = s ? *s : 1.0;
  return sv > 0.0 ? 1.0 / sv : 0.0;
}
__device__ __forceinline__ void pow_block_part(double sq, double* part) {
  __shared__ double red[kBlock];
  red[threadIdx.x] = sq;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < kBlock; k += kPowLanes) t += red[k];  // the groups' first lanes
    part[blockIdx.x] = t;
  }
}
__global__ void __launch_bounds__(kBlock) k_pow_pass(const int* ptr, const int* col,
                                                      const double* val, int rows, int thresh,
                                                      const double* fo, const double* fi,
                                                      const double* in, const double* s,
                                                      double* out, double* part) {
  const int gl = threadIdx.x & (kPowLanes - 1);
  const double inv = pow_inv(s);
  double sq = 0.0;
  const long long G = (long long)gridDim.x * (kBlock / kPowLanes);
  for (long long r = ((long long)blockIdx.x * kBlock + threadIdx.x) / kPowLanes; r < rows; r += G) {
    const int b0 = ptr[r], e0 = ptr[r + 1];
    if (e0 - b0 > thresh) continue;  // uniform within the group
    double acc = 0.0;
    for (int p = b0 + gl; p < e0; p += kPowLanes) {
      const int c = col[p];
      acc += (val ? val[p] : 1.0) * fi[c] * (in[c] * inv);
    }
    acc = group_sum<kPowLanes>(acc);
    if (gl == 0) {
      const double v = fo[r] * acc;
      out[r] = v;
      sq += v * v;
    }
  }
  if (part) pow_block_part(gl == 0 ? sq : 0.0, part);
}
// the rows longer than `thresh` (list[nlist]), one block per row, grid-strided over the list
__global__ void __launch_bounds__(kBlock) k_pow_long(const int* ptr, const int* col,
                                                      const double* val, const int* list,
                                                      int nlist, const double* fo,
                                                      const double* fi, const double* in,
                                                      const double* s, double* out,
                                                      double* part) {
  __shared__ double red[kBlock];
  const double inv = pow_inv(s);
  double sq = 0.0;
  for (int k = blockIdx.x; k < nlist; k += gridDim.x) {
    const int r = list[k];
    double acc = 0.0;
    for (int p = ptr[r] + threadIdx.x; p < ptr[r + 1]; p += kBlock) {
      const int c = col[p];
      acc += (val ? val[p] : 1.0) * fi[c] * (in[c] * inv);
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int h = kBlock / 2; h > 0; h >>= 1) {
      if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      const double v = fo[r] * red[0];
      out[r] = v;
      sq += v * v;
    }
    __syncthreads();
  }
  if (part && threadIdx.x == 0) part[blockIdx.x] = sq;
}

// s = sqrt(sum of nb partials), added in slot order (one block)
__global__ void __launch_bounds__(kBlock) k_pow_norm(const double* part, int nb, double* s) {
  __shared__ double red[kBlock];
  double t = 0.0;
  for (int k = threadIdx.x; k < nb; k += kBlock) t += part[k];
  red[threadIdx.x] = t;
  __syncthreads();
  for (int h = kBlock / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *s = sqrt(red[0]);
}

cudaError_t setup_power_norm(const PowIn& q, int iters, double* u, double* w, double* part,
                             int part_cap, double* s_dev, double* L, long long* launches,
                             cudaStream_t s) {
  *L = 0.0;
  const int G = std::max(1, std::min(part_cap / 2, device_sm_count() * 8));
  const int per = kBlock / kPowLanes;
  const int gr = std::max(1, std::min(G, (q.m + per - 1) / per));
  const int gc = std::max(1, std::min(G, (q.n + per - 1) / per));
  const int lr = std::min(q.a_nlong, G), lc = std::min(q.t_nlong, G);
  k_pow_start<<<grid_for(q.n, G), kBlock, 0, s>>>(w, q.n, s_dev);
  *launches += 1;
  for (int it = 0; it < iters; ++it) {
    // u = K~ v over the rows of A, then w = K~^T u over the rows of A^T with ||w||^2
    k_pow_pass<<<gr, kBlock, 0, s>>>(q.a_ptr, q.a_col, q.a_val, q.m, q.a_thresh, q.dr, q.dc, w,
                                     s_dev, u, nullptr);
    if (lr) k_pow_long<<<lr, kBlock, 0, s>>>(q.a_ptr, q.a_col, q.a_val, q.a_long, q.a_nlong, q.dr,
                                             q.dc, w, s_dev, u, nullptr);
    k_pow_pass<<<gc, kBlock, 0, s>>>(q.t_ptr, q.t_col, q.t_val, q.n, q.t_thresh, q.dc, q.dr, u,
                                     nullptr, w, part);
    if (lc) k_pow_long<<<lc, kBlock, 0, s>>>(q.t_ptr, q.t_col, q.t_val, q.t_long, q.t_nlong, q.dc,
                                             q.dr, u, nullptr, w, part + gc);
    k_pow_norm<<<1, kBlock, 0, s>>>(part, gc + lc, s_dev);
    *launches += 3 + (lr ? 1 : 0) + (lc ? 1 : 0);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  double sv = 0.0;
  e = cudaMemcpyAsync(&sv, s_dev, sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess) *L = sqrt(sv);
  return e;
}

cudaError_t setup_len_order(const int* ptr, int rows, int* ord, cudaStream_t s) {
  k_len_order<<<grid_for(rows, device_sm_count() * 8), kBlock, 0, s>>>(ptr, rows, ord);
  return cudaGetLastError();
}

// Cuts of the resident step kernel: block g's rows start where the nonzeros and kResRowWeight
// per row before them reach g / G of the total, so that the blocks' gathers and epilogues are
// even (an epilogue costs about as much as four gathered entries).  Block 0 finds the cuts, every
// block looks for the longest row.
constexpr int kResRowWeight = 4;
__global__ void __launch_bounds__(kBlock) k_res_plan(int m, int n, long long nnz,
                                                     const int* a_ptr, const int* t_ptr, int G,
                                                     int it, int vb, int implicit, int* cut_t,
                                                     int* cut_a, ResSizes* sizes) {
  int longest = 0;
  const long long stride = (long long)gridDim.x * kBlock;
  for (long long i = (long long)blockIdx.x * kBlock + threadIdx.x; i < (long long)m + n;
       i += stride) {
    const int* p = i < m ? a_ptr + i : t_ptr + (i - m);
    longest = max(longest, p[1] - p[0]);
  }
  longest = __reduce_max_sync(0xffffffffu, longest);
  if ((threadIdx.x & 31) == 0) atomicMax(&sizes->max_len, longest);
  if (blockIdx.x != 0) return;
  const int g = threadIdx.x;
  for (int side = 0; side < 2; ++side) {
    const int rows = side ? m : n;
    const int* ptr = side ? a_ptr : t_ptr;
    int* cut = side ? cut_a : cut_t;
    if (g <= G) {
      const long long want = (nnz + (long long)kResRowWeight * rows) * g / G;
      int lo = 0, hi = rows;  // the first row whose weight before it is at least `want`
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (ptr[mid] + (long long)kResRowWeight * mid >= want) hi = mid; else lo = mid + 1;
      }
      cut[g] = lo;
    }
  }
  __syncthreads();
  if (g < G) {
    const int nt = cut_t[g + 1] - cut_t[g], zt = t_ptr[cut_t[g + 1]] - t_ptr[cut_t[g]];
    const int na = cut_a[g + 1] - cut_a[g], za = a_ptr[cut_a[g + 1]] - a_ptr[cut_a[g]];
    atomicMax(&sizes->t_rows, nt);
    atomicMax(&sizes->t_nnz, zt);
    atomicMax(&sizes->a_rows, na);
    atomicMax(&sizes->a_nnz, za);
    atomicMax(&sizes->bytes, res_layout(nt, zt, na, za, it, vb, implicit != 0).bytes);
  }
}

cudaError_t setup_res_plan(int m, int n, int nnz, const int* a_ptr, const int* t_ptr, int G, int it,
                           int vb, bool implicit, int* cut_t, int* cut_a, ResSizes* sizes, cudaStream_t s) {
  RET(cudaMemsetAsync(sizes, 0, sizeof(ResSizes), s));
  k_res_plan<<<grid_for((long long)m + n, device_sm_count()), kBlock, 0, s>>>(
      m, n, nnz, a_ptr, t_ptr, G, it, vb, implicit ? 1 : 0, cut_t, cut_a, sizes);
  return cudaGetLastError();
}

cudaError_t setup_rescale(int m, int n, int fp32, double beta, double gamma, void* c, void* l,
                          void* u, void* q, void* x0, void* y0, double* dr, double* dc,
                          double* inv_dr, double* inv_dc, cudaStream_t s) {
  const int g = grid_for(std::max(m, n), device_sm_count() * 8);
  if (fp32)
    k_rescale<float><<<g, kBlock, 0, s>>>(m, n, beta, gamma, (float*)c, (float*)l, (float*)u,
                                          (float*)q, (float*)x0, (float*)y0, dr, dc, inv_dr, inv_dc);
  else
    k_rescale<double><<<g, kBlock, 0, s>>>(m, n, beta, gamma, (double*)c, (double*)l, (double*)u,
                                           (double*)q, (double*)x0, (double*)y0, dr, dc, inv_dr,
                                           inv_dc);
  return cudaGetLastError();
}

cudaError_t setup_kkt_aux(int m, int n, const double* dr, const double* dc, const double* l,
                          const double* u, double* inv_dr, double* inv_dc, unsigned char* bflags,
                          cudaStream_t s) {
  k_kkt_aux<<<grid_for(std::max(m, n), device_sm_count() * 8), kBlock, 0, s>>>(
      m, n, dr, dc, l, u, inv_dr, inv_dc, bflags);
  return cudaGetLastError();
}

__global__ void k_offset_copy(int* dst, const int* src, long long count, int offset) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride)
    dst[i] = src[i] + offset;
}

cudaError_t setup_offset_copy(int* dst, const int* src, long long count, int offset,
                              cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  k_offset_copy<<<grid_for(count, device_sm_count() * 8), kBlock, 0, s>>>(dst, src, count, offset);
  return cudaGetLastError();
}

cudaError_t setup_long_rows(const int* ptr, int nrows, int thresh, int* flags, int* pos, int* bsum,
                            int* list, int* h_count, cudaStream_t s) {
  const int G = device_sm_count() * 8;
  k_long_flags<<<grid_for(nrows, G), kBlock, 0, s>>>(ptr, nrows, thresh, flags);
  RET(cudaGetLastError());
  RET(exclusive_scan(flags, pos, nrows, bsum, s));
  k_long_scatter<<<grid_for(nrows, G), kBlock, 0, s>>>(flags, pos, nrows, list);
  RET(cudaGetLastError());
  RET(cudaMemcpyAsync(h_count, pos + nrows, sizeof(int), cudaMemcpyDeviceToHost, s));
  return cudaStreamSynchronize(s);
}

// ------------------------------------------------------------------ tile items
namespace {

// cnt[r] = work items that start at row r (0: row r continues the tile before it);
// lfl[r] = 1 if row r is long.  A row starts an item if it is the first row, a
// multiple of kTileRows, long, follows a long row, or starts in another window of
// W nonzeros than the row before it.
__global__ void k_tile_count(const int* ptr, int R, int W, int rows, int* cnt, int* lfl) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < R; i += stride) {
    const int r = (int)i;
    const int s = ptr[r], e = ptr[r + 1];
    const bool lng = e - s > kLongRow;
    bool start = r == 0 || r % rows == 0 || lng;
    if (!start) {
      const int sp = ptr[r - 1];
      start = s / W != sp / W || s - sp > kLongRow;
    }
    cnt[r] = start ? (lng ? (e - s + W - 1) / W : 1) : 0;
    lfl[r] = lng ? 1 : 0;
  }
}

// the first row of every LP of a batch starts an item
__global__ void k_tile_lp_starts(const int* lp_row0, int count, int R, int* cnt) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x) {
    const int r = lp_row0[k];
    if (r < R && cnt[r] == 0) cnt[r] = 1;
  }
}

__device__ int lp_of_row(const int* lp_row0, int count, int r) {
  // the last LP whose first row is <= r (empty LPs share their first row with the next)
  int lo = 0, hi = count;  // answer in [lo, hi)
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (lp_row0[mid] <= r) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ void k_tile_emit(const int* ptr, int R, int W, const int* lp_row0, int count,
                            const int* cnt, const int* off, const int* loff, TileItem* items) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < R; i += stride) {
    const int r = (int)i;
    const int c = cnt[r];
    if (c == 0) continue;
    const int lp = lp_row0 ? lp_of_row(lp_row0, count, r) : 0;
    const int s = ptr[r], e = ptr[r + 1], i0 = off[r];
    if (e - s > kLongRow) {
      for (int t = 0; t < c; ++t)
        items[i0 + t] = TileItem{r, r + 1, s + t * W, (int)min((long long)s + (long long)(t + 1) * W,
                                                               (long long)e), lp, i0, c, loff[r]};
    } else {
      int re = r + 1;
      while (re < R && cnt[re] == 0) ++re;
      items[i0] = TileItem{r, re, s, ptr[re], lp, -1, 0, -1};
    }
  }
}

__global__ void k_tile_lp_ranges(const int* lp_row0, int count, int R, const int* off,
                                 const int* loff, int* item0, int* lng0) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k <= count; k += gridDim.x * blockDim.x) {
    const int r = k == count ? R : (lp_row0 ? lp_row0[k] : 0);
    item0[k] = off[r];
    lng0[k] = loff[r];
  }
}

}  // namespace

TileShape tile_shape(int form) {
  return form == 2 ? TileShape{kWarpTileRows, kWarpTileWindowMin, kWarpTileWindowMax}
                   : TileShape{kTileRows, kTileWindowMin, kTileWindowMax};
}

int tile_window(const TileShape& sh, int R, long long nnz) {
  const double avg = R > 0 ? (double)nnz / (double)R : 1.0;
  const double w = (double)sh.rows * avg;
  return (int)std::max((double)sh.wmin, std::min((double)sh.wmax, w));
}

size_t tile_item_cap(const TileShape& sh, int R, long long nnz, int count) {
  // starts: multiples of the row cap, crossings of the W-windows, the rows at and
  // after each long row, LP starts; plus the slices of the long rows (at most
  // nnz / W + one per long row); long rows number at most nnz / (kLongRow + 1)
  const size_t W = (size_t)tile_window(sh, R, nnz), Z = (size_t)nnz;
  const size_t nlong = Z / (kLongRow + 1) + 1;
  return (size_t)R / sh.rows + 2 * (Z / W + 1) + 3 * nlong + (size_t)count + 8;
}

size_t tile_tmp_ints(int R) { return 4 * ((size_t)R + 1) + scan_tmp_ints((long long)R + 1) + 8; }

cudaError_t setup_tiles(const TileShape& sh, const int* ptr, int R, long long nnz,
                        const int* lp_row0, int count, int* tmp, TileItem* items, int* item0,
                        int* lng0, int* ticket, size_t item_cap, int* h_counts, int* W_out,
                        cudaStream_t s) {
  const int W = tile_window(sh, R, nnz);
  *W_out = W;
  int* cnt = tmp;
  int* off = cnt + (R + 1);
  int* lfl = off + (R + 1);
  int* loff = lfl + (R + 1);
  int* bsum = loff + (R + 1);
  const int G = device_sm_count() * 8;
  if (R > 0) {
    k_tile_count<<<grid_for(R, G), kBlock, 0, s>>>(ptr, R, W, sh.rows, cnt, lfl);
    RET(cudaGetLastError());
    if (lp_row0 && count > 1) {
      k_tile_lp_starts<<<grid_for(count, G), kBlock, 0, s>>>(lp_row0, count, R, cnt);
      RET(cudaGetLastError());
    }
  }
  RET(exclusive_scan(cnt, off, R, bsum, s));
  RET(exclusive_scan(lfl, loff, R, bsum, s));
  RET(cudaMemcpyAsync(h_counts, off + R, sizeof(int), cudaMemcpyDeviceToHost, s));
  RET(cudaMemcpyAsync(h_counts + 1, loff + R, sizeof(int), cudaMemcpyDeviceToHost, s));
  RET(cudaStreamSynchronize(s));
  if ((size_t)h_counts[0] > item_cap) return cudaErrorInvalidValue;
  if (R > 0) {
    k_tile_emit<<<grid_for(R, G), kBlock, 0, s>>>(ptr, R, W, lp_row0, count, cnt, off, loff, items);
    RET(cudaGetLastError());
  }
  k_tile_lp_ranges<<<grid_for(count + 1, G), kBlock, 0, s>>>(lp_row0, count, R, off, loff, item0,
                                                              lng0);
  RET(cudaGetLastError());
  if (h_counts[0] > 0) RET(cudaMemsetAsync(ticket, 0, sizeof(int) * (size_t)h_counts[0], s));
  return cudaSuccess;
}

// ------------------------------------------------------------------ batches
namespace {

// One LP of a batch: its arrays (device) and its first global row, column and
// nonzero in the block-diagonal problem.
__global__ void k_batch_ingest(const BatchLp* lps, int64_t* rp_g, int* col_g, double* val_g,
                               double* b_g, char* sense_g, double* c_g, double* l_g, double* u_g,
                               int* err) {
  const BatchLp L = lps[blockIdx.y];
  const int k = blockIdx.y;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int e = 0;
  for (long long i = t0; i <= L.m; i += stride) {
    const int64_t v = L.rp[i];
    if (i < L.m) {
      const int64_t w = L.rp[i + 1];
      if (v < 0 || w < v || w > L.nnz) e |= ERR_ROWPTR;
      const char sn = L.sense[i];
      if (sn != 'L' && sn != 'G' && sn != 'E') e |= ERR_SENSE;
      const double bi = L.b[i];
      if (!isfinite(bi)) e |= ERR_NONFINITE;
      b_g[L.R + i] = bi;
      sense_g[L.R + i] = sn;
    }
    if ((i == 0 && v != 0) || (i == L.m && v != L.nnz)) e |= ERR_ROWPTR;
    rp_g[L.R + i] = L.Z + v;  // the next LP writes the same value at its first row
  }
  for (long long p = t0; p < L.nnz; p += stride) {
    const int j = L.col[p];
    const double v = L.val[p];
    if (j < 0 || j >= L.n) e |= ERR_COL;
    if (!isfinite(v)) e |= ERR_NONFINITE;
    col_g[L.Z + p] = (int)L.C + j;
    val_g[L.Z + p] = v;
  }
  for (long long j = t0; j < L.n; j += stride) {
    const double cj = L.c[j], lj = L.l[j], uj = L.u[j];
    if (!isfinite(cj)) e |= ERR_NONFINITE;
    if (isnan(lj) || isnan(uj) || lj > uj || lj == INFINITY || uj == -INFINITY) e |= ERR_BOUNDS;
    c_g[L.C + j] = cj;
    l_g[L.C + j] = lj;
    u_g[L.C + j] = uj;
  }
  if (e) atomicOr(err + k, e);
}

// The A3 scalars of each LP, as k_iter_vectors and k_absmax_scaled take them for one LP:
// gridDim.x blocks per LP each leave 7 sums and the bits of a maximum in part[], and one thread
// per LP adds them up in order (one block per LP walked 555,000 nonzeros alone and left most
// of the chip idle: 5.86 -> 0.44 ms for 96 covering sub-LPs).
__global__ void __launch_bounds__(kBlock) k_batch_scalars(const BatchLp* lps, const double* dr,
                                                          const double* dc, const double* c,
                                                          const double* l, const double* u,
                                                          const double* q, const int* row_of,
                                                          const int* a_col, const double* a_val64,
                                                          double* part) {
  const BatchLp L = lps[blockIdx.y];
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};
  const long long t0 = (long long)blockIdx.x * kBlock + threadIdx.x;
  const long long stride = (long long)gridDim.x * kBlock;
  for (long long j = L.C + t0; j < L.C + L.n; j += stride) {
    const double d = dc[j], cj = c[j];
    acc[0] += (d * cj) * (d * cj);
    acc[2] += cj * cj;
    acc[6] += (isfinite(l[j]) && isfinite(u[j])) ? 0.0 : 1.0;
  }
  for (long long i = L.R + t0; i < L.R + L.m; i += stride) {
    const double d = dr[i], qi = q[i];
    acc[1] += (d * qi) * (d * qi);
    acc[3] += qi * qi;
  }
  const unsigned long long mx =
      absmax_scaled(L.Z + t0, L.Z + L.nnz, stride, row_of, a_col, a_val64, dr, dc);
  double r7[7];
  block_sum<7>(acc, r7);
  if (threadIdx.x == 0) {
    double* o = part + 8 * ((size_t)blockIdx.y * gridDim.x + blockIdx.x);
    for (int k = 0; k < 7; ++k) o[k] = r7[k];
    o[7] = __longlong_as_double((long long)mx);
  }
}

// out[8 k + ...] = ||c~||, ||q~||, ||c||, ||q||, max |K~_ij|, 0, 0, columns with an infinite
// bound
__global__ void k_batch_scalars_final(const double* part, int nblk, int count, double* out) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x) {
    const double* v = part + 8 * (size_t)k * nblk;
    double r[7] = {0, 0, 0, 0, 0, 0, 0}, mx = 0.0;
    for (int b = 0; b < nblk; ++b) {
      for (int i = 0; i < 7; ++i) r[i] += v[8 * b + i];
      mx = fmax(mx, v[8 * b + 7]);
    }
    double* o = out + 8 * (size_t)k;
    for (int i = 0; i < 4; ++i) o[i] = sqrt(r[i]);
    o[4] = mx;
    o[5] = 0.0;
    o[6] = 0.0;
    o[7] = r[6];
  }
}

// counts[k] = entries of `pos` (an exclusive scan over global rows) before LP k's first row
__global__ void k_batch_bounds(const BatchLp* lps, int count, int over_cols, int R,
                               const int* pos, int* out) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k <= count; k += gridDim.x * blockDim.x) {
    const long long r = k == count ? R : (over_cols ? lps[k].C : lps[k].R);
    out[k] = pos[r];
  }
}

}  // namespace

cudaError_t setup_batch_ingest(const BatchLp* d_lps, int count, long long max_rows_nnz_cols,
                               int64_t* rp_g, int* col_g, double* val_g, double* b_g,
                               char* sense_g, double* c_g, double* l_g, double* u_g, int* d_err,
                               cudaStream_t s) {
  RET(cudaMemsetAsync(d_err, 0, sizeof(int) * (size_t)count, s));
  if (count == 0) return cudaSuccess;
  const int per_lp = (int)std::min<long long>(64, std::max<long long>(1, (max_rows_nnz_cols + kBlock - 1) / kBlock));
  dim3 grid((unsigned)per_lp, (unsigned)count);
  k_batch_ingest<<<grid, kBlock, 0, s>>>(d_lps, rp_g, col_g, val_g, b_g, sense_g, c_g, l_g, u_g,
                                         d_err);
  return cudaGetLastError();
}

// blocks per LP of k_batch_scalars: eight per SM over the batch
static int batch_scalar_blocks(int count) {
  return std::max(1, std::min(32, device_sm_count() * 8 / std::max(1, count)));
}
size_t batch_scalar_doubles(int count) { return 8 * (size_t)count * batch_scalar_blocks(count); }

cudaError_t setup_batch_scalars(const BatchLp* d_lps, int count, const double* dr,
                                const double* dc, const double* c, const double* l,
                                const double* u, const double* q, const int* row_of,
                                const int* a_col, const double* a_val64, double* part, double* out,
                                cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  const int nb = batch_scalar_blocks(count);
  k_batch_scalars<<<dim3((unsigned)nb, (unsigned)count), kBlock, 0, s>>>(
      d_lps, dr, dc, c, l, u, q, row_of, a_col, a_val64, part);
  RET(cudaGetLastError());
  k_batch_scalars_final<<<grid_for(count, 64), kBlock, 0, s>>>(part, nb, count, out);
  return cudaGetLastError();
}

cudaError_t setup_batch_long_rows(const int* ptr, int R, int thresh, const BatchLp* d_lps,
                                  int count, int over_cols, int* flags, int* pos, int* bsum,
                                  int* list, int* d_bounds, cudaStream_t s) {
  const int G = device_sm_count() * 8;
  if (R > 0) {
    k_long_flags<<<grid_for(R, G), kBlock, 0, s>>>(ptr, R, thresh, flags);
    RET(cudaGetLastError());
  }
  RET(exclusive_scan(flags, pos, R, bsum, s));
  if (R > 0) {
    k_long_scatter<<<grid_for(R, G), kBlock, 0, s>>>(flags, pos, R, list);
    RET(cudaGetLastError());
  }
  k_batch_bounds<<<grid_for(count + 1, G), kBlock, 0, s>>>(d_lps, count, over_cols, R, pos,
                                                            d_bounds);
  return cudaGetLastError();
}

}  // namespace pdlp
