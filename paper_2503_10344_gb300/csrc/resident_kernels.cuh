// Step attempts of one LP held in the shared memory of all SMs (rows A4-A7 of the hot path; LPs
// of up to ~30 MB).
//
// An LP such as the 50,000 x 200,000 covering LP has 22 MB of step data: it sits in L2, and an
// attempt of three dependent launches spends its 20 us on launch boundaries and on chains of
// dependent loads (row pointer, column index, gathered entry), not on bytes.  Here one
// cooperative launch runs a whole check period.  Block b of G owns a run of columns (rows of
// A^T) and a run of rows of A, cut so that every block has about the same work (k_res_plan).
// It copies their indices, values and vectors to shared memory once per launch; an attempt
// then reads nothing from global memory but the gathered entries of y and of the (x', dx)
// pairs:
//   primal: the entries of y that the block's columns need, staged in shared memory, all loads
//           in flight at once; then each column is summed in storage order (LANES lanes per
//           row, rows beyond kResLong entries by a warp) and finished, its (x', dx) published;
//   dual:   the same over the block's rows, y' published;
//   the step decision (A6) by one thread of every block, from the same sums in the same order,
//   so that all blocks hold bit-identical copies of the step state.
// There is no grid barrier.  A published entry carries the number of the attempt that made it
// (in float32 y and its tag in 8 bytes, x', dx and theirs in 16; in float64 every number and its
// tag in 16: single accesses), a gather reads an entry
// again until the tag is the one it needs, and the blocks' partial sums travel the same way, one
// 16-byte word per block.  So a phase starts on each entry as it arrives, without the four trips
// to L2 that a fence, an arrival, a poll and a fence take (measured: 4,000-5,000 cycles per
// barrier, two of them half of an attempt of the 2,000-row covering LP).  While one warp
// collects the sums and decides, the others already gather the y' of this attempt: the next
// primal step needs them if the step is accepted (a rejected step gathers the old y again).
// No entry is overwritten while a block may still need it: x'(k + 1) is published after the
// decision of attempt k, which has every block's sums, posted when its gathers of x'(k) were
// done; y alternates between two buffers, and so do the posted sums (res_slot).
// Every wait is bounded as in the cooperative kernel of iter_kernels.cuh.
//
// Measured per attempt on a GB300: see the table above one_block_nnz() in solver.cu, where the form
// is chosen.
#pragma once

#include "internal.h"
#include "iter_kernels.cuh"

namespace pdlp {

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ ulonglong2 ld_relaxed_u128(const ulonglong2* p) {
  ulonglong2 v;
  asm volatile(
      "{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
      : "=l"(v.x), "=l"(v.y)
      : "l"(p)
      : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_u128(ulonglong2* p, ulonglong2 v) {
  asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p),
               "l"(v.x), "l"(v.y)
               : "memory");
}
__device__ __forceinline__ unsigned long long pack2(unsigned hi, float lo) {
  return ((unsigned long long)hi << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ float low_f(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ unsigned high_u(unsigned long long v) { return (unsigned)(v >> 32); }
// whether what carries `tag` is older than `want`
__device__ __forceinline__ bool res_old(unsigned tag, unsigned want) { return (int)(tag - want) < 0; }

// What is published and gathered: an entry of y, a pair (x', dx), a block's three sums, each
// with its tag in every word that a single access moves.  float32: y in 8 bytes (tag | y), a
// pair in 16 (dx | x', tag), the sums in 16; float64: a 16-byte word (value, tag) per number.
template <typename T> struct ResY;
template <typename T> struct ResX;
template <typename T> struct ResS;
template <> struct ResY<float> {
  using Word = unsigned long long;
  using Acc = float;
  static constexpr int kInFlight = kResGatherY;
  static __device__ __forceinline__ Word load(const Word* p) { return ld_relaxed_u64(p); }
  static __device__ __forceinline__ void post(Word* p, float y, unsigned tag) {
    st_relaxed_u64(p, pack2(tag, y));
  }
  static __device__ __forceinline__ bool old(const Word& w, unsigned tag) { return res_old(high_u(w), tag); }
  static __device__ __forceinline__ Acc value(const Word& w) { return low_f(w); }
};
template <> struct ResX<float> {
  using Word = ulonglong2;
  using Acc = P2<float>;
  static constexpr int kInFlight = kResGatherX;
  static __device__ __forceinline__ Word load(const Word* p) { return ld_relaxed_u128(p); }
  static __device__ __forceinline__ void post(Word* p, float x, float dx, unsigned tag) {
    st_relaxed_u128(p, ulonglong2{pack2(__float_as_uint(dx), x), tag});
  }
  static __device__ __forceinline__ bool old(const Word& w, unsigned tag) {
    return res_old((unsigned)w.y, tag);
  }
  static __device__ __forceinline__ Acc value(const Word& w) {
    return Acc{low_f(w.x), __uint_as_float(high_u(w.x))};
  }
};
template <> struct ResS<float> {
  using Word = ulonglong2;
  static __device__ __forceinline__ Word load(const Word* p) { return ld_relaxed_u128(p); }
  static __device__ __forceinline__ void post(Word* p, const float (&v)[3], unsigned tag) {
    st_relaxed_u128(p, ulonglong2{pack2(tag, v[0]), pack2(__float_as_uint(v[2]), v[1])});
  }
  static __device__ __forceinline__ bool is(const Word& w, unsigned tag) { return high_u(w.x) == tag; }
  static __device__ __forceinline__ float value(const Word& w, int k) {
    return k == 0 ? low_f(w.x) : k == 1 ? low_f(w.y) : __uint_as_float(high_u(w.y));
  }
};
__device__ __forceinline__ ulonglong2 tagged(double v, unsigned tag) {
  return ulonglong2{(unsigned long long)__double_as_longlong(v), tag};
}
__device__ __forceinline__ double untagged(const ulonglong2& w) {
  return __longlong_as_double((long long)w.x);
}
template <> struct ResY<double> {
  using Word = ulonglong2;
  using Acc = double;
  static constexpr int kInFlight = kResGatherY / 2;  // as many bytes
  static __device__ __forceinline__ Word load(const Word* p) { return ld_relaxed_u128(p); }
  static __device__ __forceinline__ void post(Word* p, double y, unsigned tag) {
    st_relaxed_u128(p, tagged(y, tag));
  }
  static __device__ __forceinline__ bool old(const Word& w, unsigned tag) {
    return res_old((unsigned)w.y, tag);
  }
  static __device__ __forceinline__ Acc value(const Word& w) { return untagged(w); }
};
template <> struct ResX<double> {
  struct alignas(32) Word {
    ulonglong2 x, dx;
  };
  using Acc = P2<double>;
  static constexpr int kInFlight = kResGatherX / 2;
  static __device__ __forceinline__ Word load(const Word* p) {
    return Word{ld_relaxed_u128(&p->x), ld_relaxed_u128(&p->dx)};
  }
  static __device__ __forceinline__ void post(Word* p, double x, double dx, unsigned tag) {
    st_relaxed_u128(&p->x, tagged(x, tag));
    st_relaxed_u128(&p->dx, tagged(dx, tag));
  }
  static __device__ __forceinline__ bool old(const Word& w, unsigned tag) {
    return res_old((unsigned)w.x.y, tag) || res_old((unsigned)w.dx.y, tag);
  }
  static __device__ __forceinline__ Acc value(const Word& w) {
    return Acc{untagged(w.x), untagged(w.dx)};
  }
};
template <> struct ResS<double> {
  struct Word {
    ulonglong2 v[3];
  };
  static __device__ __forceinline__ Word load(const Word* p) {
    return Word{{ld_relaxed_u128(p->v), ld_relaxed_u128(p->v + 1), ld_relaxed_u128(p->v + 2)}};
  }
  static __device__ __forceinline__ void post(Word* p, const double (&v)[3], unsigned tag) {
    for (int k = 0; k < 3; ++k) st_relaxed_u128(p->v + k, tagged(v[k], tag));
  }
  static __device__ __forceinline__ bool is(const Word& w, unsigned tag) {
    return (unsigned)w.v[0].y == tag && (unsigned)w.v[1].y == tag && (unsigned)w.v[2].y == tag;
  }
  static __device__ __forceinline__ double value(const Word& w, int k) { return untagged(w.v[k]); }
};

// a bounded wait: false once the limit has passed or another block has given up
struct ResWait {
  DevState* st;
  int limit, polls;
  __device__ __forceinline__ bool more() {
    if (++polls > limit) {
      atomicExch(&st->bar_err, 1);
      return false;
    }
    return (polls & 255) != 0 || *(volatile int*)&st->bar_err == 0;
  }
};

// Fault-handling tests: a block that does not begin until another one has given up waiting for it
// (or for 16 limits).  Outside the loop over the attempts: a test and a call in there made an attempt
// of the 720-hour energy system 8 % slower.
__device__ __forceinline__ void res_hold(DevState* st, int limit) {
  for (int polls = 0; polls < 16 * limit && *(volatile int*)&st->bar_err == 0; ++polls) {}
}

// n / d for n >= 0, d > 0 without the division's branch to its rare cases: the hardware's approximate
// reciprocal r and one residual correction of the quotient (Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", 1990).  r is within an ulp, so n r is within
// 1.5 2^-23 of the quotient; the residual is exact but for its last bit, and what is left before the
// final rounding is of relative size 2^-45: an error of (1/2 + 2^-20) ulp, where n is above 2^-90
// (below, that of n as the square of a float32 number is larger).  A d whose reciprocal is no normal
// number (0 / d would be 0 times infinity) is first scaled, with n, by a power of two.
// n / d itself in the loops over the rows: 0.35 us more per attempt (covering LP of 2,000 rows
// 4.3 -> 4.6, 10,000 rows 5.4 -> 5.7, 50,000 rows 12.6 -> 13.1, 200 x 400 relaxation 2.2 -> 2.55).
__device__ __forceinline__ float div_pos(float n, float d) {
  const float s = d < 0x1p-100f ? 0x1p64f : d > 0x1p100f ? 0x1p-64f : 1.0f;
  n *= s;
  d *= s;
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(d));
  const float q = n * r;
  return fmaf(fmaf(-q, d, n), r, q);
}

// N sums over a warp whose lanes other than the multiples of `step` (a power of two) below `used`
// hold zeros, in every lane that is such a multiple (lane 0 among them).  In float64, where an
// addition takes some 100 cycles and holds the SM's one pipe for 16, the levels that would add zeros
// only are left out, and all of them where every lane holds zeros (rows that did not move, warps
// without rows); in float32 the tests would cost more than the levels.  The sums advance level by
// level together: shuffles stay in program order, so sum after sum waits for each addition.
template <int N, typename T>
__device__ __forceinline__ void res_warp_sums(T (&v)[N], int step, int used) {
  constexpr bool F64 = std::is_same<T, double>::value;
  if constexpr (F64) {
    bool any = false;
#pragma unroll
    for (int k = 0; k < N; ++k) any |= __double_as_longlong(v[k]) << 1 != 0;  // (not +0, not -0)
    if (!__any_sync(0xffffffffu, any)) return;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (F64 && (o < step || o >= used)) continue;
    T w[N];
#pragma unroll
    for (int k = 0; k < N; ++k) w[k] = __shfl_xor_sync(0xffffffffu, v[k], o);
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] += w[k];
  }
}

// This block's three sums (of lane 0) posted to every replica under `tag`, and the sums over
// all blocks in slot order per lane, then a fixed shuffle tree (in lane 0).  Called by one whole warp.
// (Replicas: all blocks polling one copy of the slots queued at a few L2 lines.  A second set of
// slots: a block whose rows need no x' of another block waits for nobody between its decision and
// its next posting, so it may be an attempt ahead of a block that still reads.)
// `meanwhile` runs between the posting and the polling.
template <typename T, typename F>
__device__ __forceinline__ bool res_sums(DevState* st, typename ResS<T>::Word* slot, int reps,
                                         int G, unsigned tag, int limit, T (&sum)[3], F meanwhile) {
  using S = ResS<T>;
  constexpr int kPoll = sizeof(T) == 8 ? 2 : kResPoll;
  const int lane = threadIdx.x & 31, b = blockIdx.x;
  if constexpr (std::is_same<T, double>::value)
#pragma unroll
    for (int k = 0; k < 3; ++k) sum[k] = __shfl_sync(0xffffffffu, sum[k], 0);
  if (lane < reps) S::post(slot + res_slot(tag, reps, lane, G, b), sum, tag);
  meanwhile();
  const typename S::Word* mine = slot + res_slot(tag, reps, b & (reps - 1), G, 0);
  bool ok = true;
  sum[0] = sum[1] = sum[2] = (T)0;
  ResWait wait{st, limit, 0};
  for (int b0 = 0; b0 < G; b0 += 32 * kPoll) {
    typename S::Word w[kPoll];
#pragma unroll
    for (int i = 0; i < kPoll; ++i)
      if (b0 + i * 32 + lane < G) w[i] = S::load(mine + b0 + i * 32 + lane);
    bool miss = true;
    while (miss) {
      miss = false;
#pragma unroll
      for (int i = 0; i < kPoll; ++i)
        if (b0 + i * 32 + lane < G && !S::is(w[i], tag)) {
          miss = true;
          w[i] = S::load(mine + b0 + i * 32 + lane);
        }
      if (miss && !wait.more()) {
        ok = false;
        break;
      }
    }
#pragma unroll
    for (int i = 0; i < kPoll; ++i)
      if (b0 + i * 32 + lane < G) {
#pragma unroll
        for (int k = 0; k < 3; ++k) sum[k] += S::value(w[i], k);
      }
  }
  ok = __all_sync(0xffffffffu, ok);
  res_warp_sums(sum, 1, G);
  return ok;
}

// One side's rows of the block.
template <typename V>
struct ResSide {
  const int* ptr;       // [rows + 1] relative to the block's first nonzero
  const unsigned* key;  // [nnz] the gathers: index | (place in the chunk << bits)
  const V* val;         // [nnz] values in storage order (none for a pattern); with GV in global
                        // memory, staged with the entries that they multiply
  const int* lng;       // [nlong] rows longer than kResLong
  int rows, nlong, bits, cap;
};

template <typename T, typename V>
__device__ __forceinline__ T res_val(const V* v, int p) {
  if constexpr (std::is_same<V, Pattern>::value) return (T)1;
  else if constexpr (std::is_same<V, T>::value) return v[p];
  else return __bfloat162float(v[p]);
}

// The chunk of whole rows from row ra: at most `cap` nonzeros (every thread finds its end).
__device__ __forceinline__ int res_chunk_end(const int* ptr, int rows, int cap, int ra) {
  const int p0 = ptr[ra];
  if (ptr[rows] - p0 <= cap) return rows;
  int lo = ra + 1, hi = rows;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (ptr[mid] - p0 <= cap) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The gathers of a chunk in the order of the entries they read, to 2^shift entries: a warp's
// loads then share cache lines (unordered, each lane's load is a line of its own and the SM
// looks up one a cycle: 8,900 gathers of the covering LP's y per SM took 12,300 cycles).
// hist[kResBuckets]: scratch.  The order within a bucket is whatever the counters give: it does
// not enter any result.
__device__ __forceinline__ void res_sort_keys(const int* __restrict__ col, int n, int shift,
                                              int bits, int* hist, unsigned* key) {
  __shared__ int wsum[32];
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
  for (int i = tid; i < kResBuckets; i += T) hist[i] = 0;
  __syncthreads();
  for (int p = tid; p < n; p += T) atomicAdd(hist + (__ldg(col + p) >> shift), 1);
  __syncthreads();
  // exclusive scan: each thread a run of kResBuckets / T buckets
  const int per = kResBuckets / T;
  int s = 0;
  for (int k = 0; k < per; ++k) s += hist[tid * per + k];
  int inc = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) wsum[tid >> 5] = inc;
  __syncthreads();
  int base = inc - s;
  for (int w = 0; w < (tid >> 5); ++w) base += wsum[w];
  for (int k = 0; k < per; ++k) {
    const int c = hist[tid * per + k];
    hist[tid * per + k] = base;
    base += c;
  }
  __syncthreads();
  for (int p = tid; p < n; p += T) {
    const int c = __ldg(col + p);
    key[atomicAdd(hist + (c >> shift), 1)] = (unsigned)c | ((unsigned)p << bits);
  }
  __syncthreads();
}

// Sums over the staged entries of rows [ra, rb) of the chunk that starts at nonzero p0, and
// their epilogues: LANES lanes per row, then a warp per long row.
template <int LANES, typename T, typename Acc, typename V, typename Fin>
__device__ __forceinline__ void res_rows(const ResSide<V>& s, const V* val, const Acc* stage, int p0,
                                         int ra, int rb, Fin fin) {
  const int lane = threadIdx.x & (LANES - 1), NT = blockDim.x;
  auto add = [&](Acc& acc, int p) {
    const T v = res_val<T, V>(val, p);
    const Acc t = stage[p - p0];
    if constexpr (std::is_same<Acc, T>::value) acc += v * t;
    else acc += Acc{v * t.a, v * t.b};
  };
  for (int r = ra + (int)threadIdx.x / LANES; r < rb; r += NT / LANES) {
    const int b = s.ptr[r], e = s.ptr[r + 1];
    if (e - b > kResLong) continue;  // uniform within the group
    Acc acc{};
#pragma unroll 4
    for (int p = b + lane; p < e; p += LANES) add(acc, p);
    acc = group_sum<LANES>(acc);
    if (lane == 0) fin(r, acc);
  }
  const int wl = threadIdx.x & 31;
  for (int k = threadIdx.x >> 5; k < s.nlong; k += NT >> 5) {
    const int r = s.lng[k];
    if (r < ra || r >= rb) continue;
    const int b = s.ptr[r], e = s.ptr[r + 1];
    Acc acc{};
#pragma unroll 4
    for (int p = b + wl; p < e; p += 32) add(acc, p);
    acc = group_sum<32>(acc);
    if (wl == 0) fin(r, acc);
  }
}

template <typename T, typename Acc, typename V, typename Fin>
__device__ __forceinline__ void res_rows_lanes(int lanes, const ResSide<V>& s, const V* val,
                                               const Acc* stage, int p0, int ra, int rb, Fin fin) {
  switch (lanes) {
    case 1: return res_rows<1, T>(s, val, stage, p0, ra, rb, fin);
    case 2: return res_rows<2, T>(s, val, stage, p0, ra, rb, fin);
    case 4: return res_rows<4, T>(s, val, stage, p0, ra, rb, fin);
    case 8: return res_rows<8, T>(s, val, stage, p0, ra, rb, fin);
    default: return res_rows<16, T>(s, val, stage, p0, ra, rb, fin);
  }
}

// The entries that the rows of a chunk need, into the stage: threads t, t + nt, ... of the
// block, E::kInFlight loads in flight each.  Returns false when a wait gave up.
// (A newer tag ends the wait too: only the y gathered ahead of a step that is then rejected can
// meet one, and it is dropped.)
template <bool GV, typename E, typename V>
__device__ __forceinline__ bool res_gather(const ResSide<V>& s, int p0, int n,
                                           const typename E::Word* __restrict__ from, unsigned tag,
                                           typename E::Acc* stage, int t, int nt, ResWait wait) {
  constexpr int U = E::kInFlight;
  if constexpr (GV) {  // the chunk's values, behind its entries
    V* vst = (V*)(stage + s.cap);
#pragma unroll 4
    for (int i = t; i < n; i += nt) vst[i] = __ldg(s.val + p0 + i);
  }
  const unsigned mask = (1u << s.bits) - 1u;
  const unsigned* key = s.key + p0;
  for (int i0 = t; i0 < n; i0 += nt * U) {
    unsigned c[U];
    typename E::Word w[U];
#pragma unroll
    for (int k = 0; k < U; ++k) c[k] = i0 + k * nt < n ? key[i0 + k * nt] : 0u;
#pragma unroll
    for (int k = 0; k < U; ++k)
      if (i0 + k * nt < n) w[k] = E::load(from + (c[k] & mask));
    bool miss = true;
    while (miss) {
      miss = false;
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (i0 + k * nt < n && E::old(w[k], tag)) {
          miss = true;
          w[k] = E::load(from + (c[k] & mask));
        }
      if (miss && !wait.more()) return false;
    }
#pragma unroll
    for (int k = 0; k < U; ++k)
      if (i0 + k * nt < n) stage[c[k] >> s.bits] = E::value(w[k]);
  }
  return true;
}

// A side's product: chunk by chunk the entries its rows need, then the rows' sums.  The first
// chunk may have been gathered ahead (`ahead`).
template <typename T, bool GV, typename E, typename V, typename Fin>
__device__ __forceinline__ void res_product(int lanes, const ResSide<V>& s,
                                            const typename E::Word* from, unsigned tag,
                                            typename E::Acc* stage, bool ahead, ResWait wait,
                                            int* fail, Fin fin) {
  int ra = 0;
  while (ra < s.rows) {
    const int p0 = s.ptr[ra], rb = res_chunk_end(s.ptr, s.rows, s.cap, ra);
    if (ra > 0) __syncthreads();  // the chunk before is summed
    if (ra > 0 || !ahead)
      if (!res_gather<GV, E>(s, p0, s.ptr[rb] - p0, from, tag, stage, threadIdx.x, blockDim.x, wait))
        *fail = 1;
    __syncthreads();
    res_rows_lanes<T, typename E::Acc>(lanes, s, GV ? (const V*)(stage + s.cap) - p0 : s.val, stage, p0, ra, rb, fin);
    ra = rb;
  }
}

// The step decision (decide_step, the same operations in the iterate type) in two halves: what the
// next attempt reads, which every thread of the block waits for, and the rest of the state, written
// later in the shadow of something else (700-970 cycles of a thread that nobody waits for; at the
// start of the next attempt they delayed its whole block: a tenth of an attempt).
template <typename T>
struct ResDecision {
  T eta, eta_bar, eta_next;
  bool accept, numerical;
};
template <typename T>
__device__ __forceinline__ ResDecision<T> res_decide(DevState* st, T dx2, T dy2, T dkd, T fd, T fi,
                                                     int& left) {
  constexpr bool F64 = std::is_same<T, double>::value;
  const T eta = F64 ? (T)st->eta : (T)st->eta_f;
  ResDecision<T> r{eta, (T)INFINITY, eta, true, false};
  if (!isfinite(dx2) || !isfinite(dy2) || !isfinite(dkd)) {
    st->status = 4;  // PDLP_NUMERICAL
    r.numerical = true;
    return r;
  }
  const T om = F64 ? (T)st->omega : (T)st->omega_f, iom = F64 ? (T)0 : (T)st->inv_omega_f;
  if (st->adaptive || st->tr_cap > 0) {  // (a fixed step needs the bound for the trace alone)
    const T den = (T)2 * fabs(dkd);
    const T num = F64 ? om * dx2 + dy2 / om : om * dx2 + dy2 * iom;
    r.eta_bar = den > (T)0 ? num / den : (T)INFINITY;
  }
  if (st->adaptive) {
    r.eta_next = fmin(fd * r.eta_bar, fi * r.eta);
    r.accept = !(r.eta > r.eta_bar);
  }
  if (r.accept) {
    st->cur ^= 1;
    if (--left == 0) st->check_due = 1;
  }
  const T pw = r.accept ? r.eta : (T)0;
  if constexpr (F64) {
    st->pending_w = pw;
    st->pw_f = (float)pw;
    if (r.eta_next != r.eta) {  // (else the quotient that is there already)
      st->eta = r.eta_next;
      st->tau_d = r.eta_next / om;
      st->sigma_d = r.eta_next * om;
    }
  } else {
    st->pw_f = pw;
    st->eta_f = r.eta_next;
    st->tau_f = r.eta_next * iom;
    st->sigma_f = r.eta_next * om;
  }
  return r;
}
template <typename T>
__device__ __forceinline__ void res_record(DevState* st, const ResDecision<T>& r) {
  const long long t = st->attempts;
  st->attempts = t + 1;
  if (r.numerical) return;
  if (t < st->tr_cap) {
    st->tr_eta[t] = (double)r.eta;
    st->tr_eta_bar[t] = (double)r.eta_bar;
    st->tr_accepted[t] = r.accept ? 1 : 0;
  }
  if (r.accept) {
    st->sum_w += (double)r.eta;
    st->iters += 1;
  }
  if constexpr (std::is_same<T, float>::value) {
    st->pending_w = r.accept ? (double)r.eta : 0.0;
    st->eta = (double)r.eta_next;
  }
}

// GV: the matrix values stay in global memory (L2) and are copied with each chunk.
template <typename T, typename V, bool IMPLICIT, bool GV>
__global__ void __launch_bounds__(kResBlock, 1) k_resident(IterData<T, V> d, ResPlan R,
                                                           int max_attempts) {
  using EY = ResY<T>;
  using EX = ResX<T>;
  constexpr bool VALS = !std::is_same<V, Pattern>::value;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ DevState ls;
  __shared__ T red[3][32];  // the warps' sums (0 beyond the block's warps)
  __shared__ int nlong[2], stop, fail;
  DevState* gst = d.st;
  const int tid = threadIdx.x, NT = blockDim.x, G = R.G, b = blockIdx.x;
  if (tid == 0) {
    ls = *gst;
    if (b != 0) ls.tr_cap = 0;  // one block writes the trace
    stop = (ls.status != 0 || ls.check_due) ? 1 : 0;
    fail = 0;
  }
  if (tid < 32) red[0][tid] = red[1][tid] = red[2][tid] = (T)0;
  __syncthreads();
  if (stop) return;
  // ---- the block's columns [t0, t1) and rows [a0, a1)
  const int t0 = R.cut_t[b], t1 = R.cut_t[b + 1], a0 = R.cut_a[b], a1 = R.cut_a[b + 1];
  const int nt = t1 - t0, na = a1 - a0;
  const int tz0 = __ldg(d.t_ptr + t0), az0 = __ldg(d.a_ptr + a0);
  const int tz = __ldg(d.t_ptr + t1) - tz0, az = __ldg(d.a_ptr + a1) - az0;
  const ResLayout L = res_layout(nt, tz, na, az, (int)sizeof(T), VALS && !GV ? (int)sizeof(V) : 0, IMPLICIT);
  int* tp = (int*)(sm + L.t_ptr);
  unsigned* tk = (unsigned*)(sm + L.t_col);
  V* tv = VALS ? (V*)(sm + L.t_val) : nullptr;
  int* tl = (int*)(sm + L.t_lng);
  int* ap = (int*)(sm + L.a_ptr);
  unsigned* ak = (unsigned*)(sm + L.a_col);
  V* av = VALS ? (V*)(sm + L.a_val) : nullptr;
  int* al = (int*)(sm + L.a_lng);
  T* c = (T*)(sm + L.c);
  T* l = (T*)(sm + L.l);
  T* u = (T*)(sm + L.u);
  T* tw = IMPLICIT ? (T*)(sm + L.tw) : nullptr;
  T* q = (T*)(sm + L.q);
  T* sw = IMPLICIT ? (T*)(sm + L.sw) : nullptr;
  unsigned char* kind = sm + L.kind;
  T* xs[2] = {(T*)(sm + L.x0), (T*)(sm + L.x1)};
  T* ys[2] = {(T*)(sm + L.y0), (T*)(sm + L.y1)};
  T* sx = (T*)(sm + L.sx);
  T* sy = (T*)(sm + L.sy);
  P2<T>* stage2 = (P2<T>*)(sm + L.bytes);
  T* stage1 = (T*)(sm + L.bytes);
  typename EX::Word* const ex_x = (typename EX::Word*)R.ex_x;
  auto ex_y = [&](int k) { return (typename EY::Word*)R.ex_y[k]; };
  // ---- copy in (iterates with ordinary loads: the KKT block of the same graph wrote them);
  // the y of this launch is published under a tag of its own
  for (int i = tid; i <= nt; i += NT) tp[i] = __ldg(d.t_ptr + t0 + i) - tz0;
  for (int i = tid; i <= na; i += NT) ap[i] = __ldg(d.a_ptr + a0 + i) - az0;
  const int cur0 = ls.cur;
  const unsigned tag0 = 2u * (unsigned)ls.attempts;
  for (int i = tid; i < na; i += NT) {
    const T y = d.y[cur0][a0 + i];
    EY::post(ex_y(cur0) + a0 + i, y, tag0 + 1u);
    ys[cur0][i] = y;
    q[i] = __ldg(d.q + a0 + i);
    if constexpr (IMPLICIT) sw[i] = __ldg(d.sw + a0 + i);
    kind[i] = __ldg(d.row_kind + a0 + i);
    sy[i] = d.sum_y[a0 + i];
  }
  for (int j = tid; j < nt; j += NT) {
    c[j] = __ldg(d.c + t0 + j);
    l[j] = __ldg(d.l + t0 + j);
    u[j] = __ldg(d.u + t0 + j);
    if constexpr (IMPLICIT) tw[j] = __ldg(d.tw + t0 + j);
    xs[cur0][j] = d.x[cur0][t0 + j].x;
    sx[j] = d.sum_x[t0 + j];
  }
  if constexpr (VALS && !GV) {
    for (int p = tid; p < tz; p += NT) tv[p] = d.t_val[tz0 + p];
    for (int p = tid; p < az; p += NT) av[p] = d.a_val[az0 + p];
  }
  __syncthreads();
  // the gathers of every chunk, ordered
  int* hist = (int*)stage1;
  for (int ra = 0; ra < nt;) {
    const int rb = res_chunk_end(tp, nt, R.cap_t, ra), p0 = tp[ra];
    res_sort_keys(d.t_col + tz0 + p0, tp[rb] - p0, R.shift_t, R.bits_t, hist, tk + p0);
    ra = rb;
  }
  for (int ra = 0; ra < na;) {
    const int rb = res_chunk_end(ap, na, R.cap_a, ra), p0 = ap[ra];
    res_sort_keys(d.a_col + az0 + p0, ap[rb] - p0, R.shift_a, R.bits_a, hist, ak + p0);
    ra = rb;
  }
  // the long rows of each side in order (one warp per side)
  if (tid < 64) {
    const int side = tid >> 5, lane = tid & 31, n = side ? na : nt;
    const int* ptr = side ? ap : tp;
    int* lst = side ? al : tl;
    int cnt = 0;
    for (int r0 = 0; r0 < n; r0 += 32) {
      const int r = r0 + lane;
      const bool lg = r < n && ptr[r + 1] - ptr[r] > kResLong;
      const unsigned m = __ballot_sync(0xffffffffu, lg);
      if (lg) lst[cnt + __popc(m & ((1u << lane) - 1u))] = r;
      cnt += __popc(m);
    }
    if (lane == 0) nlong[side] = cnt;
  }
  // accepted steps to the next check (thread 0)
  int left = 0;
  if (tid == 0) {
    const long long p = ls.period - ls.iters % ls.period, q = ls.iter_limit - ls.iters;
    left = (int)(p < q ? p : q > 1 ? q : 1);
  }
  __syncthreads();
  const ResSide<V> st{tp, tk, GV ? d.t_val + tz0 : tv, tl, nt, nlong[0], R.bits_t, R.cap_t};
  const ResSide<V> sa{ap, ak, GV ? d.a_val + az0 : av, al, na, nlong[1], R.bits_a, R.cap_a};
  const int ahead_n = nt ? tp[res_chunk_end(tp, nt, R.cap_t, 0)] : 0;  // the first chunk of st
  const ResWait wait{gst, (int)ls.spin_limit, 0};
  ResDecision<T> dec{};
  const long long first_attempt = ls.attempts;
  unsigned ytag = tag0 + 1u;
  if (b == 0 && G > 1 && ls.bar_skip != 0) res_hold(gst, wait.limit);
  bool ahead = false;  // the first chunk of the next primal step is staged
  for (int att = 0; att < max_attempts; ++att) {
    const int cur = ls.cur;
    const T pw = StepT<T>::pw(&ls), tau = StepT<T>::tau(&ls), sigma = StepT<T>::sigma(&ls);
    const unsigned tag = tag0 + 2u * (unsigned)(att + 1);
    T fd = 0, fi = 0;
    if (tid == 0) step_factors(&ls, first_attempt + att + 1, &fd, &fi);
    // ---- A4: primal step over the block's columns
    {
      const T* xo = xs[cur];
      T* xn = xs[cur ^ 1];
      T dx2 = 0;
      auto fin = [&](int j, T aty) {
        const T x = xo[j];
        const T w = IMPLICIT ? tw[j] : (T)1;
        const T step = IMPLICIT ? tau * w : tau;
        const T xv = clampv(x - step * (c[j] - aty), l[j], u[j]);
        const T dd = xv - x;
        xn[j] = xv;
        EX::post(ex_x + t0 + j, xv, dd, tag);
        if (pw != (T)0) sx[j] += pw * x;  // A7: add the iterate whose weight is pending
        if constexpr (IMPLICIT) dx2 += div_pos(dd * dd, w);
        else dx2 += dd * dd;
      };
      res_product<T, GV, EY>(R.lanes_t, st, ex_y(cur), ytag, stage1, ahead, wait, &fail, fin);
      T v[1] = {dx2};
      res_warp_sums(v, R.lanes_t, 32);
      if ((tid & 31) == 0) red[0][tid >> 5] = v[0];
    }
    __syncthreads();  // the stage is free
    // ---- A5: dual step over the block's rows
    {
      const T* yo = ys[cur];
      T* yn = ys[cur ^ 1];
      typename EY::Word* gy = ex_y(cur ^ 1);
      T dy2 = 0, dkd = 0;
      auto fin = [&](int i, P2<T> acc) {  // acc.a = (K x')_i, acc.b = (K dx)_i
        const T y = yo[i];
        const T w = IMPLICIT ? sw[i] : (T)1;
        const T step = IMPLICIT ? sigma * w : sigma;
        T yv = y + step * (q[i] - (acc.a + acc.b));
        if (kind[i] != 1) yv = maxv(yv, (T)0);
        EY::post(gy + a0 + i, yv, tag);
        yn[i] = yv;
        if (pw != (T)0) sy[i] += pw * y;
        const T dd = yv - y;
        if constexpr (IMPLICIT) dy2 += div_pos(dd * dd, w);
        else dy2 += dd * dd;
        dkd += dd * acc.b;
      };
      res_product<T, GV, EX>(R.lanes_a, sa, ex_x, tag, stage2, false, wait, &fail, fin);
      T v[2] = {dy2, dkd};
      res_warp_sums(v, R.lanes_a, 32);
      if ((tid & 31) == 0) {
        red[1][tid >> 5] = v[0];
        red[2][tid >> 5] = v[1];
      }
    }
    __syncthreads();  // the stage is free, the warps' sums are there
    if (tid < 32) {
      T s[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) s[k] = red[k][tid];
      res_warp_sums(s, 1, NT >> 5);
      bool ok = fail == 0;
      auto record = [&] {  // of the attempt before, while the sums travel
        if (tid == 0 && att > 0) res_record(&ls, dec);
      };
      if (G > 1)
        ok = res_sums<T>(gst, (typename ResS<T>::Word*)R.slot, R.replicas, G, tag, wait.limit, s,
                         record) && ok;
      else
        record();
      // ---- A6: the same decision in every block
      if (tid == 0) {
        dec = res_decide<T>(&ls, s[0], s[1], s[2], fd, fi, left);
        stop = !ok ? 2 : (ls.status != 0 || ls.check_due) ? 1 : 0;
      }
    } else if (!res_gather<GV, EY>(st, 0, ahead_n, ex_y(cur ^ 1), tag, stage1, tid - 32, NT - 32,
                                 wait)) {
      fail = 1;
    }
    __syncthreads();
    if (stop || fail) break;
    ahead = ls.cur != cur;  // accepted: what was gathered ahead is the y of the next step
    if (ahead) ytag = tag;
    if (!ahead) __syncthreads();  // the stage is gathered anew
  }
  if (stop == 2 || fail) {  // a wait gave up: so do the others', before long
    if (tid == 0) {
      atomicExch(&gst->bar_err, 1);
      atomicExch(&gst->status, kStatusWaitFailed);
    }
    return;
  }
  if (tid == 0 && max_attempts > 0) res_record(&ls, dec);  // of the last attempt
  // ---- copy out: the iterate (its step is not needed any more) and the running sums
  const int cur = ls.cur;
  for (int j = tid; j < nt; j += NT) {
    vec2_t<T> o;
    o.x = xs[cur][j];
    o.y = (T)0;
    d.x[cur][t0 + j] = o;
    d.sum_x[t0 + j] = sx[j];
  }
  for (int i = tid; i < na; i += NT) {
    d.y[cur][a0 + i] = ys[cur][i];
    d.sum_y[a0 + i] = sy[i];
  }
  if (b == 0 && tid == 0) {
    store_step_state(gst, ls);
    // others may have given up on this block's last sums and left without their part of the
    // iterate (they flag bar_err before the status, which was overwritten just now)
    __threadfence();
    if (*(volatile int*)&gst->bar_err != 0) atomicExch(&gst->status, kStatusWaitFailed);
  }
}

}  // namespace pdlp
