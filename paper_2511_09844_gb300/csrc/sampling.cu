// Speculative acceptance (Sec. 3.1; Leviathan et al. 2023) and token sampling over the
// vocabulary.
//
// Decisions are integers (token ids, accept/reject), so every floating-point step that feeds one
// is a correctly rounded fp32 operation in a fixed order (common.cuh: exp_cw, log_at), and every
// reduction across threads and CTAs is exact: maxima and arg-maxima through atomicMax on
// order-preserving packed keys (ties to the lowest index), the softmax normaliser through 64-bit
// integer sums of floor(e * 2^45). The outcome therefore does not depend on how the vocabulary
// is split across CTAs. Acceptance of many rows first takes an approximate normaliser with a proven bound, and
// the exact ones only for the decisions within it and the rows drawn from.
//
//   p = softmax(z / T):  s = z * fl(1/T), m = max s, e = exp(s - m), S = fl(sum floor(e 2^45)) 2^-45,
//                        p = e / S
//   accept draft i  iff  u_i * q_i(x_i) <= p_{i-1}(x_i)              (u_i from Philox)
//   replacement         argmax_v max(0, p_j - q_{j+1})_v / E_v, E_v = -ln u_v; if that residual is 0
//                        everywhere, argmax_v (s_v - ln E_v) on row j
//   bonus / draft       argmax_v (s_v - ln E_v)   (exponential race in log form)
//   T = 0               accept iff x_i = argmax z_{i-1}; emit argmax of the row
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace sd2 {
namespace {

constexpr int kThreads = 256;
constexpr int kPerCta = kThreads * 4 * 8;   // most vocabulary entries per CTA (8 passes of 4 per thread)
constexpr int kRacePerCta = kThreads * 4 * 32; // the acceptance race (longer spans: more of it is skipped)
constexpr int kStatsPerCta = kThreads * 8 * 8;   // the row-statistics passes: at most 8 passes of 8
enum { MODE_NONE = 0, MODE_DONE = 1, MODE_RESIDUAL = 2, MODE_BONUS = 3 };

// Vocabulary entries per CTA for `rows` rows: enough CTAs per row to fill the GPU about twice over,
// in whole passes of `gran` entries per thread, at most max_span (few rows: more, shorter CTAs; a
// large batch keeps long ones). Every decision is independent of how the vocabulary is split.
int vocab_span(int V, int rows, int gran, int max_span) {
  const int pass = kThreads * gran;
  const int want = std::max(1, (2 * sm_count_cached() + rows - 1) / std::max(1, rows));
  const int span = (((V + want - 1) / want + pass - 1) / pass) * pass;
  return std::min(max_span, std::max(pass, span));
}

template <typename T>
__device__ __forceinline__ void load4(const T* row, int v, float z[4]);
template <>
__device__ __forceinline__ void load4<float>(const float* row, int v, float z[4]) {
  const float4 t = *reinterpret_cast<const float4*>(row + v);
  z[0] = t.x; z[1] = t.y; z[2] = t.z; z[3] = t.w;
}
template <>
__device__ __forceinline__ void load4<bf16>(const bf16* row, int v, float z[4]) {
  const uint2 t = *reinterpret_cast<const uint2*>(row + v);
  z[0] = bf_lo(t.x); z[1] = bf_hi(t.x); z[2] = bf_lo(t.y); z[3] = bf_hi(t.y);
}
// 8 consecutive entries from v (n < 8 of them at the row's end; rows start 16-byte (f32) or 8-byte
// (bf16) aligned)
template <typename T>
__device__ __forceinline__ void load8(const T* row, int v, int n, float z[8]);
template <>
__device__ __forceinline__ void load8<float>(const float* row, int v, int n, float z[8]) {
  if (n >= 8) {
    const float4 a = *reinterpret_cast<const float4*>(row + v), b = *reinterpret_cast<const float4*>(row + v + 4);
    z[0] = a.x; z[1] = a.y; z[2] = a.z; z[3] = a.w; z[4] = b.x; z[5] = b.y; z[6] = b.z; z[7] = b.w;
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) z[j] = j < n ? row[v + j] : 0.f;
  }
}
template <>
__device__ __forceinline__ void load8<bf16>(const bf16* row, int v, int n, float z[8]) {
  if (n >= 8) {    // rows are 8-byte aligned (V % 4 == 0): two 8-byte loads
    const uint2 t = *reinterpret_cast<const uint2*>(row + v), u = *reinterpret_cast<const uint2*>(row + v + 4);
    z[0] = bf_lo(t.x); z[1] = bf_hi(t.x); z[2] = bf_lo(t.y); z[3] = bf_hi(t.y);
    z[4] = bf_lo(u.x); z[5] = bf_hi(u.x); z[6] = bf_lo(u.y); z[7] = bf_hi(u.y);
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) z[j] = j < n ? bf2f(row[v + j]) : 0.f;
  }
}
template <typename T>
__device__ __forceinline__ float load1(const T* row, int v);
template <>
__device__ __forceinline__ float load1<float>(const float* row, int v) { return row[v]; }
template <>
__device__ __forceinline__ float load1<bf16>(const bf16* row, int v) { return bf2f(row[v]); }

__device__ __forceinline__ float inv_temp(float t) { return __fdiv_rn(1.0f, t); }

__device__ __forceinline__ unsigned long long block_max_u64(unsigned long long v, unsigned long long* red) {
  v = warp_max_u64(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  v = (l < (int)(blockDim.x >> 5)) ? red[l] : 0ull;
  return warp_max_u64(v);
}
__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long v, unsigned long long* red) {
  v = warp_sum_u64(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  v = (l < (int)(blockDim.x >> 5)) ? red[l] : 0ull;
  return warp_sum_u64(v);
}

struct RowRef {
  int b;
  bool is_draft;
  size_t offset;  // element offset of the row
};
// Row r of the stats table: target rows b*(k+1)+i first, then draft rows b*k+i.
__device__ __forceinline__ RowRef row_ref(int r, int B, int k, int V) {
  RowRef rr;
  const int nt = B * (k + 1);
  if (r < nt) {
    rr.b = r / (k + 1); rr.is_draft = false; rr.offset = static_cast<size_t>(r) * V;
  } else {
    rr.b = (r - nt) / k; rr.is_draft = true; rr.offset = static_cast<size_t>(r - nt) * V;
  }
  return rr;
}

__device__ __forceinline__ unsigned step_value(const int* step_ptr, unsigned step) {
  return step_ptr ? static_cast<unsigned>(*step_ptr) : step;
}
__device__ __forceinline__ unsigned long long seed_value(const Seed& s) { return s.ptr ? *s.ptr : s.value; }

// A row's key in the stats table: the packed (max of s, first index of it) of pack_key with bit 31
// of its low word (set for every index) cleared when the row held a non-finite logit.
constexpr unsigned long long kKeyFinite = 0x80000000ull;
__device__ __forceinline__ unsigned long long row_key(unsigned long long key, bool bad) {
  return bad ? key & ~kKeyFinite : key | kKeyFinite;
}
__device__ __forceinline__ bool key_bad(unsigned long long key) { return !(key & kKeyFinite); }
__device__ __forceinline__ int key_index(unsigned long long key) { return static_cast<int>(packed_index(key | kKeyFinite)); }

// What the first kernel of an acceptance prepares for the last: a sequence's race slots and its
// counter (done by the CTA that holds the sequence's first target row), the error word of a
// standalone call.
__device__ __forceinline__ void prepare_race(int r, int B, int k, const AcceptScratch& s, unsigned* err, int reset_err) {
  if (threadIdx.x) return;
  if (r == 0 && reset_err) *err = 0u;
  if (r < B * (k + 1) && r % (k + 1) == 0) {
    const int b = r / (k + 1);
    s.slot[2 * b] = 0ull;
    s.slot[2 * b + 1] = 0ull;
    s.counter[b] = 0;
  }
}

// This thread's packed (max, first index of it) of s = z/T (z when greedy) over entries lo .. hi - 1,
// and whether it met a non-finite one. Its entries come in increasing index order, so a strictly
// greater value is the only update (+0 and -0 compare equal, as the packed key folds them). Each
// group of 8 is reduced with fmaxf first; only a group that beats the running maximum is searched
// for the first index of its maximum. Non-finite entries show as a NaN in sum(z - z).
template <typename T>
__device__ __forceinline__ unsigned long long max_of(const T* row, int lo, int hi, bool greedy, float invT, bool& bad) {
  float best_s = -INFINITY;
  int best_i = -1;
  float nf = 0.f;
#pragma unroll 2
  for (int v = lo + threadIdx.x * 8; v < hi; v += blockDim.x * 8) {
    float z[8];
    const int n = min(8, hi - v);
    load8<T>(row, v, n, z);
    float s[8];
    if (n == 8) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        nf += __fsub_rn(z[j], z[j]);
        s[j] = greedy ? z[j] : __fmul_rn(z[j], invT);
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        nf += j < n ? __fsub_rn(z[j], z[j]) : 0.f;
        s[j] = j < n ? (greedy ? z[j] : __fmul_rn(z[j], invT)) : -INFINITY;
      }
    }
    const float g = fmaxf(fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3])), fmaxf(fmaxf(s[4], s[5]), fmaxf(s[6], s[7])));
    if (g > best_s || best_i < 0) {
      int jj = 7;
#pragma unroll
      for (int j = 7; j >= 0; --j) jj = (j < n && s[j] == g) ? j : jj;
      best_s = g;
      best_i = v + jj;
    }
  }
  bad = !(nf == 0.f);
  return best_i < 0 ? 0ull : pack_key(best_s, static_cast<uint32_t>(best_i));
}

// sum floor(exp(s - m) 2^45) of the first n of 8 logits.
__device__ __forceinline__ unsigned long long fixed_sum8(const float (&z)[8], int n, float invT, float m, f32x2 mz) {
  uint32_t ah = 0, al = 0;
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    float e0, e1;
    exp_cw2(__fsub_rn(__fmul_rn(z[j], invT), m), __fsub_rn(__fmul_rn(z[j + 1], invT), m), mz, e0, e1);
    uint32_t ph, pl;
    fixed45_parts(j < n ? e0 : 0.f, ph, pl);
    ah += ph;
    al += pl;
    fixed45_parts(j + 1 < n ? e1 : 0.f, ph, pl);
    ah += ph;
    al += pl;
  }
  return (static_cast<unsigned long long>(ah) << 23) + al;
}
// This thread's part of the exact fixed-point normaliser over entries lo .. hi - 1.
template <typename T>
__device__ __forceinline__ unsigned long long sum_of(const T* row, int lo, int hi, float invT, float m, f32x2 mz) {
  unsigned long long acc = 0;
#pragma unroll 2
  for (int v = lo + threadIdx.x * 8; v < hi; v += blockDim.x * 8) {
    float z[8];
    const int n = min(8, hi - v);
    load8<T>(row, v, n, z);
    acc += fixed_sum8(z, n, invT, m, mz);
  }
  return acc;
}

// ------------------------------------------------------------------------------ few rows
// Row statistics of a few rows (small batches): one cluster of C CTAs per row (16 while that is what it
// takes to fill the GPU, else 8), which exchange their maxima, then their exact normalisers, through
// distributed shared memory, so the maximum and the normaliser are one launch. Bound by latency: a
// thread holds its entries (up to kHeld groups of 8) in registers between the two, so the row is
// loaded once, all loads in flight at once; longer rows are read again.
constexpr int kRowThreads = 512;
constexpr int kHeld = 3;
template <typename T, int C>
__global__ void __launch_bounds__(kRowThreads) row_stats_kernel(const T* target, const T* draft, int B, int k, int V,
                                                                const float* temp, const int* stopped,
                                                                AcceptScratch sc, unsigned* err, int reset_err) {
  pdl_trigger();
  cluster_arrive_relaxed();                          // waited for before the first store into another CTA
  pdl_wait();
  __shared__ unsigned long long red[32];
  __shared__ __align__(16) float4 sMax[C];           // from every CTA: key (two words), non-finite flag
  __shared__ __align__(16) float4 sSum[C];           // rank 0's: every CTA's normaliser (two words)
  const int r = blockIdx.x / C, rank = static_cast<int>(cluster_rank());
  const RowRef rr = row_ref(r, B, k, V);
  const T* row = (rr.is_draft ? draft : target) + rr.offset;
  const int span = ((V + C * 8 - 1) / (C * 8)) * 8;
  const int lo = rank * span, hi = min(V, lo + span);
  const bool held = span <= kHeld * kRowThreads * 8;
  float z[kHeld][8];
  if (held)
#pragma unroll
    for (int u = 0; u < kHeld; ++u) {
      const int v = lo + (u * kRowThreads + static_cast<int>(threadIdx.x)) * 8;
      load8<T>(row, v, max(0, hi - v), z[u]);
    }
  if (rank == 0) prepare_race(r, B, k, sc, err, reset_err);
  const float t = temp[rr.b];
  const bool greedy = !(t > 0.f);
  if ((stopped && stopped[rr.b]) || (greedy && rr.is_draft)) {   // uniform over the cluster
    __syncwarp();
    cluster_wait();
    return;
  }
  const float invT = greedy ? 1.f : inv_temp(t);
  bool bad;
  unsigned long long best;
  if (held) {
    float best_s = -INFINITY, nf = 0.f;
    int best_i = -1;
#pragma unroll
    for (int u = 0; u < kHeld; ++u) {
      const int v = lo + (u * kRowThreads + static_cast<int>(threadIdx.x)) * 8;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        nf += __fsub_rn(z[u][j], z[u][j]);
        const float s = greedy ? z[u][j] : __fmul_rn(z[u][j], invT);
        const bool up = v + j < hi && (s > best_s || best_i < 0);   // increasing index: only a greater value moves it
        best_s = up ? s : best_s;
        best_i = up ? v + j : best_i;
      }
    }
    bad = !(nf == 0.f);
    best = best_i < 0 ? 0ull : pack_key(best_s, static_cast<uint32_t>(best_i));
  } else {
    best = max_of<T>(row, lo, hi, greedy, invT, bad);
  }
  best = block_max_u64(best, red);
  const int any_bad = __syncthreads_or(bad ? 1 : 0);
  // Every CTA of the cluster runs: a store into the shared memory of one that has not started would be lost (a
  // short vocabulary leaves slices empty, whose CTAs are here at once).
  cluster_wait();
  if (threadIdx.x < C)
    st_dsmem_v4(static_cast<uint32_t>(__cvta_generic_to_shared(&sMax[rank])), threadIdx.x,
                __uint_as_float(static_cast<uint32_t>(best)), __uint_as_float(static_cast<uint32_t>(best >> 32)),
                __uint_as_float(static_cast<uint32_t>(any_bad)), 0.f);
  cluster_sync_all();
  best = 0ull;
  bad = false;
#pragma unroll
  for (int q = 0; q < C; ++q) {
    const float4 w = sMax[q];
    const unsigned long long key = (static_cast<unsigned long long>(__float_as_uint(w.y)) << 32) | __float_as_uint(w.x);
    best = key > best ? key : best;
    bad |= __float_as_uint(w.z) != 0u;
  }
  if (rank == 0 && threadIdx.x == 0) sc.rowkey[r] = row_key(best, bad);
  if (greedy) return;                                // no remote access follows: free to leave
  const float m = packed_key(best);
  unsigned long long acc = 0;
  if (held) {
#pragma unroll
    for (int u = 0; u < kHeld; ++u) {
      const int n = hi - (lo + (u * kRowThreads + static_cast<int>(threadIdx.x)) * 8);
      if (n > 0) acc += fixed_sum8(z[u], n, invT, m, sc.minus_zero2);
    }
  } else {
    acc = sum_of<T>(row, lo, hi, invT, m, sc.minus_zero2);
  }
  acc = block_sum_u64(acc, red);
  if (threadIdx.x == 0)
    st_dsmem_v4(static_cast<uint32_t>(__cvta_generic_to_shared(&sSum[rank])), 0u,
                __uint_as_float(static_cast<uint32_t>(acc)), __uint_as_float(static_cast<uint32_t>(acc >> 32)), 0.f, 0.f);
  cluster_sync_all();
  if (rank == 0 && threadIdx.x == 0) {
    acc = 0;
#pragma unroll
    for (int q = 0; q < C; ++q)
      acc += (static_cast<unsigned long long>(__float_as_uint(sSum[q].y)) << 32) | __float_as_uint(sSum[q].x);
    sc.rowsum[r] = acc;
  }
}

// ------------------------------------------------------------------------------ many rows
// Row statistics of many rows: one CTA per row, one pass over the logits: the exact maximum and an
// approximate normaliser (hardware ex2, fp32 sums about each thread's running maximum), written as a
// float into rowsum. An acceptance test needs the exact normalisers only where u q and p are closer
// than the approximation's error, and the replacement only those of one target and one draft row, so
// the fixed-sequence exponentials (about 25 operations a logit) run on the rows that need them
// instead of on all 2k + 1 of a sequence. What is left per logit, about 6 operations and one ex2,
// fits under the one read of the logits: 256 sequences x 33 rows of 152064 bf16 take 462 us in all for
// 2.57 GB (5.6 TB/s), 1928 us with two passes and the exact exponential of every logit.
// Relative error of the approximate normaliser against the exact one (accept_norm_margin), with u = 2^-24:
//   exponents    three roundings of the distance t from the maximum (the exact side's subtraction; a subtraction,
//                and the product with a rounded log2 e, here; a chain of references splits t, not the errors'
//                sum), weighted by the mass at t, whose mean is at most ln V: 13 (3 u + 2^-26) < 3e-6
//   ex2, exp_cw  4e-7
//   sums         u for every entry of a thread's accumulator (V / (4 threads)) and for the block's tree
//   rescales     ex2 (2^-22) and a product (u) for every raise of a thread's reference, at most one a pass of 32
//                entries a thread, one for the last 4 entries and one to the block's maximum
constexpr int kManyThreads = 256;

constexpr float kLog2e = 0x1.715476p+0f;

// max and min of two values, NaN if either is (max) or the number (min)
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// 32 entries of one thread's pass, in groups of G consecutive ones (16 bytes); the groups of a pass
// lie kManyThreads groups apart, so a warp's loads are contiguous.
template <typename T>
struct Chunk;
template <>
struct Chunk<bf16> {
  static constexpr int G = 8;
  uint4 w[4];
  // groups 0 .. ng - 1 exist, ng >= 1; the others repeat group 0, which changes no max or min
  __device__ __forceinline__ void load(const bf16* p, bool wide, int ng) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const bf16* q = p + (i < ng ? i : 0) * kManyThreads * G;
      if (wide) {
        w[i] = __ldg(reinterpret_cast<const uint4*>(q));
      } else {                             // rows are 8-byte aligned
        const uint2 a = __ldg(reinterpret_cast<const uint2*>(q)), b = __ldg(reinterpret_cast<const uint2*>(q) + 1);
        w[i] = make_uint4(a.x, a.y, b.x, b.y);
      }
    }
  }
  __device__ __forceinline__ void range(float& mx, float& mn) const {
    auto h = [](uint32_t v) { return *reinterpret_cast<const __nv_bfloat162*>(&v); };
    __nv_bfloat162 a = h(w[0].x), b = a;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t q[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        a = __hmax2_nan(a, h(q[j]));
        b = __hmin2(b, h(q[j]));
      }
    }
    mx = max_nan(__low2float(a), __high2float(a));
    mn = fminf(__low2float(b), __high2float(b));
  }
  __device__ __forceinline__ void pair(int i, float& lo, float& hi) const {   // pair i of 16
    const uint4 v = w[i >> 2];
    const uint32_t q[4] = {v.x, v.y, v.z, v.w};
    lo = bf_lo(q[i & 3]);
    hi = bf_hi(q[i & 3]);
  }
};
template <>
struct Chunk<float> {
  static constexpr int G = 4;
  float4 w[8];
  __device__ __forceinline__ void load(const float* p, bool, int ng) {
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = __ldg(reinterpret_cast<const float4*>(p + (i < ng ? i : 0) * kManyThreads * G));
  }
  __device__ __forceinline__ void range(float& mx, float& mn) const {
    mx = w[0].x;
    mn = w[0].x;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      mx = max_nan(mx, max_nan(max_nan(w[i].x, w[i].y), max_nan(w[i].z, w[i].w)));
      mn = fminf(mn, fminf(fminf(w[i].x, w[i].y), fminf(w[i].z, w[i].w)));
    }
  }
  __device__ __forceinline__ void pair(int i, float& lo, float& hi) const {
    const float4 v = w[i >> 1];
    lo = (i & 1) ? v.z : v.x;
    hi = (i & 1) ? v.w : v.y;
  }
};

template <typename T>
__global__ void __launch_bounds__(kManyThreads) row_scan_kernel(const T* target, const T* draft, int B, int k, int V,
                                                                const float* temp, const int* stopped,
                                                                AcceptScratch sc, unsigned* err, int reset_err) {
  pdl_trigger();
  pdl_wait();
  __shared__ unsigned long long red[32];
  __shared__ float redf[32];
  const int r = blockIdx.x;
  const RowRef rr = row_ref(r, B, k, V);
  prepare_race(r, B, k, sc, err, reset_err);
  if (stopped && stopped[rr.b]) return;
  const float t = temp[rr.b];
  const bool greedy = !(t > 0.f);
  if (greedy && rr.is_draft) return;
  const T* row = (rr.is_draft ? draft : target) + rr.offset;
  bool bad;
  if (greedy) {
    unsigned long long best = block_max_u64(max_of<T>(row, 0, V, true, 1.f, bad), red);
    const int any_bad = __syncthreads_or(bad ? 1 : 0);
    if (threadIdx.x == 0) sc.rowkey[r] = row_key(best, any_bad != 0);
    return;
  }
  constexpr int G = Chunk<T>::G, NG = 32 / G;
  const float invT = inv_temp(t);
  const bool wide = (reinterpret_cast<uintptr_t>(row) & 15) == 0;
  float m = -INFINITY, zx = -INFINITY, zn = INFINITY;   // reference of the sums; largest and smallest logit
  f32x2 s0 = 0ull, s1 = 0ull;                        // pairs of running sums of 2^((s - m) log2 e)
  const f32x2 iT = pk2(invT, invT), l2e = pk2(kLog2e, kLog2e);
  auto reference = [&](float cx) {                   // logits up to cx follow
    zx = max_nan(zx, cx);
    const float sx = __fmul_rn(cx, invT);
    if (sx > m) {
      const float f = exp2_approx(__fmul_rn(m - sx, kLog2e));
      s0 = mul2(s0, pk2(f, f));
      s1 = mul2(s1, pk2(f, f));
      m = sx;
    }
  };
  const int Vg = V - V % G;                          // whole groups; at most 4 entries follow
  for (int v = threadIdx.x * G; v < Vg; v += kManyThreads * 32) {
    Chunk<T> c;
    const int ng = min(NG, (Vg - v - 1) / (kManyThreads * G) + 1);
    c.load(row + v, wide, ng);
    float cx, cn;
    c.range(cx, cn);
    zn = fminf(zn, cn);
    reference(cx);
    const f32x2 nm = pk2(-m, -m);
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      if (2 * i / G < ng) {
        float z0, z1, z2, z3, e0, e1, e2, e3;
        c.pair(i, z0, z1);
        c.pair(i + 1, z2, z3);
        un2(mul2(add2(prod2(pk2(z0, z1), iT, sc.minus_zero2), nm), l2e), e0, e1);
        un2(mul2(add2(prod2(pk2(z2, z3), iT, sc.minus_zero2), nm), l2e), e2, e3);
        s0 = add2(s0, pk2(exp2_approx(e0), exp2_approx(e1)));
        s1 = add2(s1, pk2(exp2_approx(e2), exp2_approx(e3)));
      }
    }
  }
  if (Vg + static_cast<int>(threadIdx.x) < V) {      // the row's last 4 entries (bf16, V % 8 == 4)
    const float z = load1<T>(row, Vg + threadIdx.x);
    zn = fminf(zn, z);
    reference(z);
    s0 = add2(s0, pk2(exp2_approx(__fmul_rn(__fmul_rn(z, invT) - m, kLog2e)), 0.f));
  }
  float a0, a1, a2, a3;
  un2(s0, a0, a1);
  un2(s1, a2, a3);
  const float sum = (a0 + a1) + (a2 + a3);
  const unsigned long long key = block_max_u64(pack_key(m, 0u), red);
  const float M = packed_key(key);
  // (a thread without entries has m = -inf and an empty sum)
  bad = zn == -INFINITY || zx == INFINITY || !(zx == zx);
  const float total = block_sum(m == -INFINITY ? 0.f : sum * exp2_approx(__fmul_rn(m - M, kLog2e)), redf);
  const int any_bad = __syncthreads_or(bad ? 1 : 0);
  if (threadIdx.x == 0) {
    sc.rowkey[r] = row_key(key, any_bad != 0);
    sc.rowsum[r] = __float_as_uint(total);
  }
}

// ------------------------------------------------------------------------------ decisions
struct RowDist {  // what p(x) needs for one row
  float m, S;
};
__device__ __forceinline__ RowDist row_dist(const unsigned long long* rowkey, const unsigned long long* rowsum, int r) {
  RowDist d;
  d.m = packed_key(rowkey[r]);
  d.S = __fmul_rn(__ull2float_rn(rowsum[r]), 0x1p-45f);
  return d;
}
__device__ __forceinline__ float prob(float z, float invT, RowDist d) {
  return __fdiv_rn(exp_cw(__fsub_rn(__fmul_rn(z, invT), d.m)), d.S);
}
__device__ __forceinline__ float accept_u01(int i, int b, unsigned stp, uint32_t k0, uint32_t k1) {
  return bits_to_u01(philox4x32_10(make_uint4(0u, (RNG_ACCEPT << 16) | i, static_cast<uint32_t>(b), stp), k0, k1).x);
}
// ERR_NONFINITE if any of sequence b's rows held a non-finite logit (a greedy sequence reads no draft
// row). By the lanes of one warp.
__device__ __forceinline__ void report_bad_rows(int b, int B, int k, bool greedy, const AcceptScratch& s, unsigned* err) {
  bool bad = false;
  for (int i = threadIdx.x & 31; i <= k; i += 32) {
    bad |= key_bad(s.rowkey[b * (k + 1) + i]);
    if (!greedy && i < k) bad |= key_bad(s.rowkey[B * (k + 1) + b * k + i]);
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(err, static_cast<unsigned>(ERR_NONFINITE));
}
// First draft of sequence b that is not its row's argmax: the kept prefix j (k: all kept), at T = 0.
// By the lanes of one warp.
__device__ __forceinline__ int greedy_prefix(const int* xb, const unsigned long long* keys, int k) {
  for (int i0 = 0; i0 < k; i0 += 32) {
    const int i = i0 + (threadIdx.x & 31);
    const unsigned miss = __ballot_sync(0xffffffffu, i < k && xb[i] != key_index(keys[i]));
    if (miss) return i0 + __ffs(miss) - 1;
  }
  return k;
}

// ------------------------------------------------------------------------------ the race
struct Race {
  int j;
  bool resid;        // residual race (a draft was rejected), else the log-form race on row j
  float invT;
  RowDist dp, dq;    // residual: the exact distributions of target row j and draft row j + 1
};
// Replacement or bonus token of sequence b over slice entries lo .. hi - 1, the whole block; the
// sequence's last slice to finish emits the token. A thread skips the exact arithmetic of an entry
// that cannot win: with E = -ln u >= 1 - u, its key is at most p_hi / (1 - u) (residual race; p_hi is
// the hardware ex2's p, 0.1% up, far beyond its error) or s - ln(1 - u) + slack (log form), compared
// with the best exact key the block has published so far. Skipped keys are strictly smaller, so the
// winner, ties included, is that of the full evaluation. What is left per entry is the Philox word
// and a few operations. The log-form race that replaces an all-zero residual (rounding only) is run
// by the last slice, alone.
template <typename T>
__device__ void race_slice(const T* target, const T* draft, int b, int B, int k, int V, const Race& ra, int lo, int hi,
                           int n_slices, unsigned stp, uint32_t k0, uint32_t k1, int* tokens, int* n,
                           const AcceptScratch& s) {
  __shared__ unsigned long long red[32];
  __shared__ unsigned sBest;                 // ord_f32 of the best key published
  __shared__ int sLast;
  const T* trow = target + static_cast<size_t>(b * (k + 1) + ra.j) * V;
  const T* drow = draft + static_cast<size_t>(b * k + ra.j) * V;     // read in the residual race only
  const float invT = ra.invT;
  volatile unsigned* vbest = &sBest;
  auto words = [&](int v) {
    return philox4x32_10(make_uint4(static_cast<uint32_t>(v >> 2), (RNG_RESAMPLE << 16) | ra.j, static_cast<uint32_t>(b), stp),
                         k0, k1);
  };
  auto log_race = [&](int from, int to) {
    if (threadIdx.x == 0) sBest = 0u;
    __syncthreads();
    unsigned long long best = 0;
    for (int v = from + threadIdx.x * 4; v < to; v += blockDim.x * 4) {
      const uint4 c = words(v);
      const uint32_t w[4] = {c.x, c.y, c.z, c.w};
      float z[4];
      load4<T>(trow, v, z);
      const unsigned bo = *vbest;
      const float bk = bo ? unord_f32(bo) : -INFINITY;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float u = bits_to_u01(w[e]), st = __fmul_rn(z[e], invT);
        const float hi_key = st - 0x1.62e43p-1f * __log2f(1.f - u);
        if (hi_key + (1e-4f + 1e-6f * fabsf(hi_key)) < bk) continue;
        const float E = -log_at(u);
        const unsigned long long kl = pack_key(__fsub_rn(st, log_at(E)), v + e);
        if (kl > best) {
          best = kl;
          atomicMax(&sBest, static_cast<unsigned>(kl >> 32));
        }
      }
    }
    return block_max_u64(best, red);
  };
  unsigned long long best = 0;
  if (ra.resid) {
    if (threadIdx.x == 0) sBest = 0u;
    __syncthreads();
    const float up = __fdiv_rn(1.001f, ra.dp.S);
    for (int v = lo + threadIdx.x * 4; v < hi; v += blockDim.x * 4) {
      const uint4 c = words(v);
      const uint32_t w[4] = {c.x, c.y, c.z, c.w};
      float zt[4], zd[4];
      load4<T>(trow, v, zt);
      load4<T>(drow, v, zd);
      const unsigned bo = *vbest;
      const float bk = bo > 0x80000000u ? unord_f32(bo) : 0.f;     // a key above +0
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float u = bits_to_u01(w[e]), t = __fsub_rn(__fmul_rn(zt[e], invT), ra.dp.m);
        if (exp2_approx(t * kLog2e) * up < bk * (1.f - u)) continue;
        const float p = __fdiv_rn(exp_cw(t), ra.dp.S);
        const float q = __fdiv_rn(exp_cw(__fsub_rn(__fmul_rn(zd[e], invT), ra.dq.m)), ra.dq.S);
        const float r = fmaxf(__fsub_rn(p, q), 0.0f);
        if (r == 0.f) continue;                                    // cannot be drawn
        const unsigned long long kr = pack_key(__fdiv_rn(r, -log_at(u)), v + e);
        if (kr > best) {
          best = kr;
          atomicMax(&sBest, static_cast<unsigned>(kr >> 32));
        }
      }
    }
    best = block_max_u64(best, red);
  } else {
    best = log_race(lo, hi);
  }
  if (threadIdx.x == 0) {
    atomicMax(&s.slot[2 * b], best);
    __threadfence();
    sLast = atomicAdd(&s.counter[b], 1) == n_slices - 1;
  }
  __syncthreads();
  if (!sLast) return;
  __shared__ unsigned long long sWin;
  if (threadIdx.x == 0) sWin = atomicMax(&s.slot[2 * b], 0ull);
  __syncthreads();
  unsigned long long win = sWin;
  if (ra.resid && !(static_cast<uint32_t>(win >> 32) > 0x80000000u)) win = log_race(0, V);   // no key above +0
  if (threadIdx.x == 0) {
    tokens[static_cast<size_t>(b) * (k + 1) + ra.j] = static_cast<int>(packed_index(win));
    n[b] = ra.j + 1;
    s.counter[b] = 0;
  }
}

// Few rows: every slice of a sequence takes the sequence's decisions itself (a lane per draft, from
// the exact row statistics), then races over its slice.
template <typename T>
__global__ void __launch_bounds__(kThreads) decide_race_kernel(const T* target, const T* draft, const int* xhat,
                                                               const float* temp, int B, int k, int V, Seed seed_arg,
                                                               const int* step_ptr, unsigned step, const int* stopped,
                                                               int* tokens, int* n, AcceptScratch s, unsigned* err, int span) {
  pdl_trigger();
  pdl_wait();
  __shared__ int sJ;
  const int b = blockIdx.x;
  const bool first = blockIdx.y == 0;
  if (stopped && stopped[b]) {
    if (first && threadIdx.x == 0) n[b] = 0;
    return;
  }
  const int* xb = xhat + static_cast<size_t>(b) * k;
  int* out = tokens + static_cast<size_t>(b) * (k + 1);
  const float t = temp[b];
  const bool greedy = !(t > 0.f);
  const unsigned long long* keys = s.rowkey + b * (k + 1);
  if (greedy && !first) return;
  const float invT = greedy ? 1.f : inv_temp(t);
  const unsigned stp = step_value(step_ptr, step);
  const unsigned long long seed = seed_value(seed_arg);
  const uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
  const int nt = B * (k + 1);
  if (threadIdx.x < 32) {
    if (first) report_bad_rows(b, B, k, greedy, s, err);
    int j = k;
    if (greedy) {
      j = greedy_prefix(xb, keys, k);
    } else {
      for (int i0 = 0; i0 < k && j == k; i0 += 32) {
        const int i = i0 + threadIdx.x;
        bool rej = false;
        if (i < k) {
          const int x = min(max(xb[i], 0), V - 1);
          const int rt = b * (k + 1) + i, rd = nt + b * k + i;
          const float p = prob(load1<T>(target + static_cast<size_t>(rt) * V, x), invT, row_dist(s.rowkey, s.rowsum, rt));
          const float q = prob(load1<T>(draft + static_cast<size_t>(rd - nt) * V, x), invT, row_dist(s.rowkey, s.rowsum, rd));
          rej = !(__fmul_rn(accept_u01(i + 1, b, stp, k0, k1), q) <= p);
        }
        const unsigned m = __ballot_sync(0xffffffffu, rej);
        if (m) j = i0 + __ffs(m) - 1;
      }
    }
    if (first)
      for (int i = threadIdx.x; i < j; i += 32) out[i] = xb[i];
    if (threadIdx.x == 0) {
      sJ = j;
      if (greedy) {
        out[j] = key_index(keys[j]);
        n[b] = j + 1;
      }
    }
  }
  if (greedy) return;
  __syncthreads();
  Race ra;
  ra.j = sJ;
  ra.resid = ra.j < k;
  ra.invT = invT;
  if (ra.resid) {
    ra.dp = row_dist(s.rowkey, s.rowsum, b * (k + 1) + ra.j);
    ra.dq = row_dist(s.rowkey, s.rowsum, nt + b * k + ra.j);
  }
  const int lo = blockIdx.y * span;
  race_slice<T>(target, draft, b, B, k, V, ra, lo, min(V, lo + span), gridDim.y, stp, k0, k1, tokens, n, s);
}

// Many rows: the decisions of one sequence from the approximate normalisers. Draft i is certain when
// u q and p differ by more than their error bound (margin, relative); the first draft that is not is
// settled by its two exact normalisers, summed by the whole block (a few in 10^4 drafts).
template <typename T>
__global__ void __launch_bounds__(kRowThreads) decide_kernel(const T* target, const T* draft, const int* xhat,
                                                             const float* temp, int B, int k, int V, Seed seed_arg,
                                                             const int* step_ptr, unsigned step, const int* stopped,
                                                             int* tokens, int* n, AcceptScratch s, unsigned* err,
                                                             float margin) {
  pdl_trigger();
  pdl_wait();
  __shared__ unsigned long long red[32];
  __shared__ int sI, sKind;
  const int b = blockIdx.x, lane = threadIdx.x & 31;
  if (stopped && stopped[b]) {
    if (threadIdx.x == 0) {
      n[b] = 0;
      s.jmode[2 * b] = 0;
      s.jmode[2 * b + 1] = MODE_NONE;
    }
    return;
  }
  const int* xb = xhat + static_cast<size_t>(b) * k;
  int* out = tokens + static_cast<size_t>(b) * (k + 1);
  const float t = temp[b];
  const bool greedy = !(t > 0.f);
  if (threadIdx.x < 32) report_bad_rows(b, B, k, greedy, s, err);
  if (greedy) {
    if (threadIdx.x < 32) {
      const unsigned long long* keys = s.rowkey + b * (k + 1);
      const int j = greedy_prefix(xb, keys, k);
      for (int i = lane; i < j; i += 32) out[i] = xb[i];
      if (lane == 0) {
        out[j] = key_index(keys[j]);
        n[b] = j + 1;
        s.jmode[2 * b] = j;
        s.jmode[2 * b + 1] = MODE_DONE;
      }
    }
    return;
  }
  const float invT = inv_temp(t);
  const unsigned stp = step_value(step_ptr, step);
  const unsigned long long seed = seed_value(seed_arg);
  const uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
  const int nt = B * (k + 1);
  enum { ACCEPT = 0, REJECT = 1, UNSURE = 2 };
  int j = k;
  for (int from = 0; from < k;) {
    if (threadIdx.x < 32) {                // the first draft from `from` on that is not surely kept
      int at = k, kind = ACCEPT;
      for (int i0 = from; i0 < k && at == k; i0 += 32) {
        const int i = i0 + lane;
        int kd = ACCEPT;
        if (i < k) {
          const int x = min(max(xb[i], 0), V - 1);
          const int rt = b * (k + 1) + i, rd = nt + b * k + i;
          const float ep = exp_cw(__fsub_rn(__fmul_rn(load1<T>(target + static_cast<size_t>(rt) * V, x), invT), packed_key(s.rowkey[rt])));
          const float eq = exp_cw(__fsub_rn(__fmul_rn(load1<T>(draft + static_cast<size_t>(rd - nt) * V, x), invT), packed_key(s.rowkey[rd])));
          const float p = ep / __uint_as_float(static_cast<uint32_t>(s.rowsum[rt]));
          const float uq = accept_u01(i + 1, b, stp, k0, k1) * (eq / __uint_as_float(static_cast<uint32_t>(s.rowsum[rd])));
          // far above the denormals on the larger side, so roundings stay relative
          kd = UNSURE;
          if (eq == 0.f) kd = ACCEPT;                                  // u 0 <= p
          else if (p > 1e-30f && uq * (1.f + margin) < p) kd = ACCEPT;
          else if (uq > 1e-30f && p * (1.f + margin) < uq) kd = REJECT;
        }
        const unsigned m = __ballot_sync(0xffffffffu, kd != ACCEPT);
        if (m) {
          at = i0 + __ffs(m) - 1;
          kind = __shfl_sync(0xffffffffu, kd, __ffs(m) - 1);
        }
      }
      if (lane == 0) { sI = at; sKind = kind; }
    }
    __syncthreads();
    const int i = sI, kind = sKind;
    __syncthreads();
    if (i >= k) break;
    if (kind == UNSURE) {
      const int rt = b * (k + 1) + i, rd = nt + b * k + i, x = min(max(xb[i], 0), V - 1);
      const T* tr = target + static_cast<size_t>(rt) * V;
      const T* dr = draft + static_cast<size_t>(rd - nt) * V;
      RowDist dp, dq;
      dp.m = packed_key(s.rowkey[rt]);
      dq.m = packed_key(s.rowkey[rd]);
      dp.S = __fmul_rn(__ull2float_rn(block_sum_u64(sum_of<T>(tr, 0, V, invT, dp.m, s.minus_zero2), red)), 0x1p-45f);
      dq.S = __fmul_rn(__ull2float_rn(block_sum_u64(sum_of<T>(dr, 0, V, invT, dq.m, s.minus_zero2), red)), 0x1p-45f);
      if (__fmul_rn(accept_u01(i + 1, b, stp, k0, k1), prob(load1<T>(dr, x), invT, dq)) <= prob(load1<T>(tr, x), invT, dp)) {
        from = i + 1;
        continue;
      }
    }
    j = i;
    break;
  }
  for (int i = threadIdx.x; i < j; i += blockDim.x) out[i] = xb[i];
  if (threadIdx.x == 0) {
    s.jmode[2 * b] = j;
    s.jmode[2 * b + 1] = j < k ? MODE_RESIDUAL : MODE_BONUS;
    if (j < k) {                           // summed exactly by the next kernel
      s.rowsum[b * (k + 1) + j] = 0ull;
      s.rowsum[nt + b * k + j] = 0ull;
    }
  }
}

// Many rows: the exact normalisers of the two rows each replacement is drawn from.
template <typename T>
__global__ void __launch_bounds__(kThreads) resid_sum_kernel(const T* target, const T* draft, int B, int k, int V,
                                                             const float* temp, AcceptScratch s, int span) {
  pdl_trigger();
  pdl_wait();
  __shared__ unsigned long long red[32];
  const int b = blockIdx.x >> 1;
  const bool is_draft = blockIdx.x & 1;
  if (s.jmode[2 * b + 1] != MODE_RESIDUAL) return;
  const int j = s.jmode[2 * b];
  const int lr = is_draft ? b * k + j : b * (k + 1) + j;          // row of its tensor
  const int r = is_draft ? B * (k + 1) + lr : lr;
  const T* row = (is_draft ? draft : target) + static_cast<size_t>(lr) * V;
  const int lo = blockIdx.y * span;
  const unsigned long long acc =
      block_sum_u64(sum_of<T>(row, lo, min(V, lo + span), inv_temp(temp[b]), packed_key(s.rowkey[r]), s.minus_zero2), red);
  if (threadIdx.x == 0 && acc) atomicAdd(&s.rowsum[r], acc);
}

// Many rows: the race of the sequences whose decisions decide_kernel took.
template <typename T>
__global__ void __launch_bounds__(kThreads) race_kernel(const T* target, const T* draft, const float* temp, int B, int k,
                                                        int V, Seed seed_arg, const int* step_ptr, unsigned step,
                                                        int* tokens, int* n, AcceptScratch s, int span) {
  pdl_trigger();
  pdl_wait();
  const int b = blockIdx.x;
  const int mode = s.jmode[2 * b + 1];
  if (mode != MODE_RESIDUAL && mode != MODE_BONUS) return;
  Race ra;
  ra.j = s.jmode[2 * b];
  ra.resid = mode == MODE_RESIDUAL;
  ra.invT = inv_temp(temp[b]);
  if (ra.resid) {
    ra.dp = row_dist(s.rowkey, s.rowsum, b * (k + 1) + ra.j);
    ra.dq = row_dist(s.rowkey, s.rowsum, B * (k + 1) + b * k + ra.j);
  }
  const unsigned long long seed = seed_value(seed_arg);
  const int lo = blockIdx.y * span;
  race_slice<T>(target, draft, b, B, k, V, ra, lo, min(V, lo + span), gridDim.y, step_value(step_ptr, step),
                static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32), tokens, n, s);
}

// One token per row: argmax (T = 0) or the log-form exponential race.
__global__ void __launch_bounds__(kThreads) sample_kernel(const float* logits, long long ld, int V, const float* temp,
                                                          Seed seed_arg, int purpose, int i,
                                                          const int* step_ptr, unsigned step, int* out, int ld_out,
                                                          int* out2, int ld_out2, unsigned long long* slot,
                                                          int* counter, unsigned* err, int span) {
  pdl_trigger();
  __shared__ unsigned long long red[32];
  __shared__ bool last;
  extern __shared__ float4 race[];         // ln E of the span's entries after the first pass's, a thread's own
  float4 first = make_float4(0.f, 0.f, 0.f, 0.f);      // the first pass's
  const int b = blockIdx.x;
  const float* row = logits + static_cast<size_t>(b) * ld;
  // Temperature, seed and step lie since before the step, so the race's random half, which is most of the
  // arithmetic, is done while the logits are still being computed (only the logits are waited for): a step of 8
  // drafts at batch 16 11.88 -> 11.72 ms, of 5 at batch 1 6.555 -> 6.530. The first pass's values stay in registers,
  // so that a one-pass launch (batch 1) fits beside the lm_head's CTAs.
  const float t = temp[b];
  const bool greedy = !(t > 0.f);
  const float invT = greedy ? 1.f : inv_temp(t);
  const unsigned stp = step_value(step_ptr, step);
  const unsigned long long seed = seed_value(seed_arg);
  const uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
  const int lo = blockIdx.y * span, hi = min(V, lo + span);
  for (int v = lo + threadIdx.x * 4; !greedy && v < hi; v += kThreads * 4) {
    const uint4 c = philox4x32_10(make_uint4(static_cast<uint32_t>(v >> 2), (static_cast<uint32_t>(purpose) << 16) | i,
                                             static_cast<uint32_t>(b), stp), k0, k1);
    const float4 g = make_float4(log_at(-log_at(bits_to_u01(c.x))), log_at(-log_at(bits_to_u01(c.y))),
                                 log_at(-log_at(bits_to_u01(c.z))), log_at(-log_at(bits_to_u01(c.w))));
    if (v < lo + kThreads * 4) first = g;
    else race[((v - lo) >> 2) - kThreads] = g;
  }
  pdl_wait();
  unsigned long long best = 0;
  bool bad = false;
#pragma unroll 4
  for (int v = lo + threadIdx.x * 4; v < hi; v += kThreads * 4) {
    float z[4];
    load4<float>(row, v, z);
    const float4 g4 = greedy ? make_float4(0.f, 0.f, 0.f, 0.f) : v < lo + kThreads * 4 ? first : race[((v - lo) >> 2) - kThreads];
    const float g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      bad |= !isfinite(z[e]);
      const float key = greedy ? z[e] : __fsub_rn(__fmul_rn(z[e], invT), g[e]);
      const unsigned long long pk = pack_key(key, v + e);
      best = pk > best ? pk : best;
    }
  }
  best = block_max_u64(best, red);
  const int any_bad = __syncthreads_or(bad ? 1 : 0);
  if (threadIdx.x == 0) {
    atomicMax(&slot[b], best);
    if (any_bad) atomicOr(err, static_cast<unsigned>(ERR_NONFINITE));
    __threadfence();
    last = (atomicAdd(&counter[b], 1) == static_cast<int>(gridDim.y) - 1);
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    const unsigned long long r = atomicExch(&slot[b], 0ull);
    const int tok = static_cast<int>(packed_index(r));
    out[static_cast<size_t>(b) * ld_out] = tok;
    if (out2) out2[static_cast<size_t>(b) * ld_out2] = tok;
    counter[b] = 0;
  }
}

// Rows (2k + 1 a sequence) up to which the acceptance runs as two latency-bound launches with every
// normaliser exact; above, as four whose exact arithmetic covers only the rows that need it. One CTA
// per row fills the GPU from about as many rows as it has SMs on. Measured (us, few / many rows path):
// 132 rows of 128256 f32 51.7 / 59.5, 176 rows 67.7 / 70.1, 264 rows 88.0 / 68.7; 176 rows of 32000
// bf16 38.4 / 27.7; 11 rows of 128256 f32 15.7 / 29.0. A short vocabulary's rows are read sooner: 32000 bf16,
// 80 rows 24.7 / 24.3, 112 rows 29.2 / 25.0, 144 rows 34.3 / 26.2 (152064: 43 / 58, 53 / 68, 62 / 74).
constexpr int kFewRows = 152, kFewRowsShort = 96, kShortVocab = 1 << 16;
int few_rows(int V) { return V <= kShortVocab ? kFewRowsShort : kFewRows; }

// Whether the 16-CTA clusters of row_stats_kernel can be scheduled (a non-portable size: the attribute
// is set for the current context on every call, the device's answer is remembered).
template <typename T>
bool clusters_of_16() {
  const auto f = row_stats_kernel<T, 16>;
  if (cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  static const bool fits = [f] {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(kRowThreads);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    const bool ok = cudaOccupancyMaxActiveClusters(&n, f, &cfg) == cudaSuccess && n > 0;
    cudaGetLastError();
    return ok;
  }();
  return fits;
}

template <typename T>
cudaError_t accept_typed(const T* target, const T* draft, const int* xhat, const float* temp, int B, int k, int V,
                         Seed seed, unsigned step, const int* step_ptr, const int* stopped, int* tokens,
                         int* n, const AcceptScratch& s, unsigned* err, bool reset_err, cudaStream_t st) {
  const int R = B * (2 * k + 1), reset = reset_err ? 1 : 0;
  const int span = vocab_span(V, B, 4, kRacePerCta), S = (V + span - 1) / span;
  cudaError_t e;
  if (R <= few_rows(V)) {
    e = R * 8 < sm_count_cached() && clusters_of_16<T>()
            ? launch_pdl_cluster(row_stats_kernel<T, 16>, dim3(R * 16), dim3(kRowThreads), 0, st, 16, target, draft, B, k, V,
                                 temp, stopped, s, err, reset)
            : launch_pdl_cluster(row_stats_kernel<T, 8>, dim3(R * 8), dim3(kRowThreads), 0, st, 8, target, draft, B, k, V,
                                 temp, stopped, s, err, reset);
    if (e != cudaSuccess) return e;
    return launch_pdl(decide_race_kernel<T>, dim3(B, S), dim3(kThreads), 0, st, target, draft, xhat, temp, B, k, V, seed,
                      step_ptr, step, stopped, tokens, n, s, err, span);
  }
  e = launch_pdl(row_scan_kernel<T>, dim3(R), dim3(kManyThreads), 0, st, target, draft, B, k, V, temp, stopped, s, err, reset);
  if (e != cudaSuccess) return e;
  // p and u q each carry one normaliser's error; a few fp32 roundings on top
  const float margin = 2.f * accept_norm_margin(V) + 1e-6f;
  e = launch_pdl(decide_kernel<T>, dim3(B), dim3(kRowThreads), 0, st, target, draft, xhat, temp, B, k, V, seed, step_ptr,
                 step, stopped, tokens, n, s, err, margin);
  if (e != cudaSuccess) return e;
  const int rspan = vocab_span(V, 2 * B, 8, kStatsPerCta), RS = (V + rspan - 1) / rspan;
  e = launch_pdl(resid_sum_kernel<T>, dim3(2 * B, RS), dim3(kThreads), 0, st, target, draft, B, k, V, temp, s, rspan);
  if (e != cudaSuccess) return e;
  return launch_pdl(race_kernel<T>, dim3(B, S), dim3(kThreads), 0, st, target, draft, temp, B, k, V, seed, step_ptr, step,
                    tokens, n, s, span);
}

}  // namespace

float accept_norm_margin(int V) {
  const int passes = (V + 32 * kManyThreads - 1) / (32 * kManyThreads);
  return 6e-6f + 6.0e-8f * (static_cast<float>(V) / (4.f * kManyThreads) + 24.f) + 3.1e-7f * static_cast<float>(passes + 2);
}

size_t accept_scratch_bytes(int B, int k) {
  const size_t R = static_cast<size_t>(B) * (2 * k + 1);
  return 8 * (2 * R) + 8 * (2 * static_cast<size_t>(B)) + 4 * static_cast<size_t>(B) + 4 * 2 * static_cast<size_t>(B) + 64;
}

AcceptScratch accept_scratch_carve(void* base, int B, int k) {
  const size_t R = static_cast<size_t>(B) * (2 * k + 1);
  AcceptScratch s;
  s.minus_zero2 = kMinusZero2;
  unsigned long long* p = static_cast<unsigned long long*>(base);
  s.rowkey = p;
  s.rowsum = p + R;
  s.slot = p + 2 * R;
  s.counter = reinterpret_cast<int*>(p + 2 * R + 2 * B);
  s.jmode = s.counter + B;
  return s;
}

cudaError_t accept_blocks(const void* target, const void* draft, int dtype, const int* xhat, const float* temp, int B,
                          int k, int V, Seed seed, unsigned step, const int* step_ptr, const int* stopped,
                          int* tokens, int* n, const AcceptScratch& s, unsigned* err, bool reset_err, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  if (dtype == 1)
    return accept_typed<bf16>(static_cast<const bf16*>(target), static_cast<const bf16*>(draft), xhat, temp, B, k, V,
                              seed, step, step_ptr, stopped, tokens, n, s, err, reset_err, st);
  return accept_typed<float>(static_cast<const float*>(target), static_cast<const float*>(draft), xhat, temp, B, k, V,
                             seed, step, step_ptr, stopped, tokens, n, s, err, reset_err, st);
}

cudaError_t sample_rows(const float* logits, long long ld, int B, int V, const float* temp, Seed seed,
                        int purpose, int i, const int* step_ptr, unsigned step, int* out, int ld_out, int* out2,
                        int ld_out2, unsigned long long* slot, int* counter, unsigned* err, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  const int span = vocab_span(V, B, 4, kPerCta), S = (V + span - 1) / span;
  { const cudaError_t e_ = launch_pdl(sample_kernel, dim3(dim3(B, S)), dim3(kThreads), static_cast<size_t>(span - kThreads * 4) * 4, st, logits, ld, V, temp, seed, purpose, i, step_ptr, step, out, ld_out,
                                                 out2, ld_out2, slot, counter, err, span); if (e_ != cudaSuccess) return e_; }
  return cudaGetLastError();
}

}  // namespace sd2
