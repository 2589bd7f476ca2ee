// Causal decode attention of few query vectors over many sequences (heads of 64): the drafter steps of a
// batch, 1 or 2 rows of every sequence.
//
// With at most 16 query vectors per (sequence, KV head) the products are small and what counts is how soon
// the K/V rows arrive. The kernel of attention.cu walks 64-position tiles with all its warps, three block
// barriers a tile, and merges its context splits through a cluster; here one CTA per (sequence, KV head)
// gives each of 8 warps a range of the positions, staged by cp.async six sub-tiles of 16 (a cache block) ahead
// (three where two CTAs share an SM), and nothing synchronises before the warps' partials are merged. Each
// warp is a flash-decoding pass on mma.sync m16n8k16 (16 query vectors x 8 positions, then x 8 dimensions).
// Bound by latency: the first rows' arrival, then about 1100 cycles of dependent products, exponentials and
// shuffles a sub-tile (16 warps of three sub-tiles: 3.2 us where 8 take 2.9 at 128 positions, 13.9 for 14.6 at
// 2500). 16 sequences of 145 to 700 positions, 8 KV heads: 9.3 -> 5.2 us.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "kernels.h"
#include "tc.cuh"

namespace sd2 {
namespace {

using tc::smem_u32;

constexpr int kHd = 64;
constexpr int kQv = 16;                    // query vectors of a group: the MMA's M side
constexpr int kSub = 16;                   // positions per sub-tile: one cache block
constexpr int kStride = kHd + 8;           // K/V/Q row stride (bf16)
constexpr int kAcc = kHd + 4;              // a warp's partial accumulators, row stride (f32)
constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
// BUF: sub-tiles in flight per warp. 6 fill an SM's shared memory, 3 leave room for a second CTA.
template <int BUF>
struct FewCfg {
  static constexpr int WARP = BUF * 2 * kSub * kStride * 2;            // a warp's K/V buffers
  static constexpr int SMEM = kQv * kStride * 2 + kQv * 4 + kWarps * kQv * 8 + kWarps * WARP;
  static_assert(kQv * kAcc * 4 <= WARP, "the partials lie over the warp's buffers");
};

__device__ __forceinline__ uint32_t word(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }
__device__ __forceinline__ void copy16(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void load_transposed(uint32_t addr, uint32_t& r0, uint32_t& r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr) : "memory");
}
__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

template <int BUF>
__global__ void __launch_bounds__(kThreads, BUF <= 3 ? 2 : 1) attn_few_kernel(const AttnArgs a) {
  constexpr int kBuf = BUF, kWarpBytes = FewCfg<BUF>::WARP;
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char smem[];
  bf16* sQ = reinterpret_cast<bf16*>(smem);
  int* sPos = reinterpret_cast<int*>(sQ + kQv * kStride);
  float2* sML = reinterpret_cast<float2*>(sPos + kQv);                 // [warp][query vector]: max, sum
  unsigned char* sKV = reinterpret_cast<unsigned char*>(sML + kWarps * kQv);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g8 = lane >> 2, t4 = lane & 3;
  const int kvh = blockIdx.x, g = blockIdx.y, Hkv = a.kv.Hkv, G = a.H / Hkv;
  unsigned char* wkv = sKV + warp * kWarpBytes;

  // Before the wait: the plan tables, the block table and the pre-step length. Rows below `stable` were
  // written before the step, every row of the step lies below ctx_hi; the warps share [0, ctx_hi) in whole
  // sub-tiles.
  const int r0 = a.grp_row0[g], seq = a.grp_seq[g], nqv = min(a.grp_nrows[g] * G, kQv), len = a.pre_len[seq];
  const int row_end = static_cast<int>(min(static_cast<long>(a.kv.bt_stride) * 16, static_cast<long>(a.n_splits) * a.chunk));
  const int stable = min(max(0, len + a.pre_stable), row_end);
  const int ctx_hi = min(max(stable, len + a.pre_stable + a.pre_fresh), row_end);
  const int per = (ctx_hi + kWarps * kSub - 1) / (kWarps * kSub) * kSub;
  const int w_lo = warp * per, w_hi = min(w_lo + per, ctx_hi);
  const int* table = a.kv.table + static_cast<size_t>(seq) * a.kv.bt_stride;
  const bf16* base = static_cast<const bf16*>(a.kv.pool) +
                     (static_cast<size_t>(a.layer) * a.kv.n_blocks * 2 * Hkv + kvh) * 16 * kHd;
  int ids = 0;                             // lane l: the block of sub-tile l of the current 32
  auto load_ids = [&](int j) { ids = table[min((w_lo >> 4) + j + lane, a.kv.bt_stride - 1)]; };
  // rows [from, to) of sub-tile j into its slot: those below `valid` loaded, the others zero
  auto issue = [&](int j, int from, int to, int valid) {
    bf16* dk = reinterpret_cast<bf16*>(wkv + (j % kBuf) * 2 * kSub * kStride * 2);
    bf16* dv = dk + kSub * kStride;
    const bf16* src0 = base + static_cast<size_t>(__shfl_sync(0xffffffffu, ids, j & 31)) * 2 * Hkv * 16 * kHd;
#pragma unroll
    for (int u = 0; u < kSub * kHd / 8 / 32; ++u) {
      const int e = lane + 32 * u, t = e >> 3, c = e & 7, p = w_lo + j * kSub + t;
      if (p < from || p >= to) continue;
      const bool ok = p < valid;
      const bf16* src = ok ? src0 + t * kHd + c * 8 : base;
      copy16(smem_u32(dk + t * kStride + c * 8), src, ok);
      copy16(smem_u32(dv + t * kStride + c * 8), ok ? src + static_cast<size_t>(Hkv) * 16 * kHd : base, ok);
    }
  };
  const int n_all = w_hi > w_lo ? (w_hi - w_lo + kSub - 1) / kSub : 0;
  const int pre_hi = max(w_lo, min(stable, w_hi));
  load_ids(0);
  for (int j = 0; j < kBuf && j < n_all; ++j) issue(j, w_lo, pre_hi, pre_hi);
  pdl_wait();
  for (int j = 0; j < kBuf; ++j) {         // the step's own rows; a group of copies per sub-tile
    if (j < n_all) issue(j, pre_hi, INT_MAX, w_hi);
    copies_commit();
  }
  {
    const int qv = tid >> 4, c4 = tid & 15, m = r0 + qv / G;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (qv < nqv) v = *(reinterpret_cast<const float4*>(a.q + (static_cast<size_t>(m) * a.H + kvh * G + qv % G) * kHd) + c4);
    *reinterpret_cast<uint2*>(sQ + qv * kStride + c4 * 4) = make_uint2(bf16_pair(v.x, v.y), bf16_pair(v.z, v.w));
    if (tid < kQv) sPos[tid] = tid < nqv ? a.row_pos[r0 + tid / G] : -1;
  }
  __syncthreads();
  int pmax = -1;
#pragma unroll
  for (int i = 0; i < kQv; ++i) pmax = max(pmax, sPos[i]);
  // A row beyond the planned bound or the block table is reported; what lies past the splits' cover is just not seen.
  if (tid == 0 && min(static_cast<long>(pmax + 1), static_cast<long>(a.n_splits) * a.chunk) > ctx_hi && a.err)
    atomicOr(a.err, static_cast<unsigned>(ERR_RANGE));
  const int hi = min(pmax + 1, w_hi), n = hi > w_lo ? (hi - w_lo + kSub - 1) / kSub : 0;
  const int pa = sPos[g8], pb = sPos[g8 + 8];          // this lane's two query vectors: g8 and g8 + 8
  uint32_t qa[kHd / 16][4];
#pragma unroll
  for (int kk = 0; kk < kHd / 16; ++kk) {
    const bf16* q0 = sQ + g8 * kStride + kk * 16 + 2 * t4;
    qa[kk][0] = word(q0);
    qa[kk][1] = word(q0 + 8 * kStride);
    qa[kk][2] = word(q0 + 8);
    qa[kk][3] = word(q0 + 8 * kStride + 8);
  }
  constexpr float kScale = 0.125f;         // 1 / sqrt(64)
  float m_a = -INFINITY, m_b = -INFINITY, l_a = 0.f, l_b = 0.f;
  float acc[kHd / 8][4];
#pragma unroll
  for (int d = 0; d < kHd / 8; ++d) acc[d][0] = acc[d][1] = acc[d][2] = acc[d][3] = 0.f;
  for (int j = 0; j < n; ++j) {
    copies_wait<kBuf - 1>();
    __syncwarp();
    const bf16* sK = reinterpret_cast<const bf16*>(wkv + (j % kBuf) * 2 * kSub * kStride * 2);
    const bf16* sV = sK + kSub * kStride;
    float s[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {          // 8 positions each
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int kk = 0; kk < kHd / 16; ++kk) {
        const bf16* kp = sK + (h * 8 + g8) * kStride + kk * 16 + 2 * t4;
        mma(c, qa[kk], word(kp), word(kp + 8));
      }
      const int p = w_lo + j * kSub + h * 8 + 2 * t4;
      s[h][0] = p <= pa ? c[0] * kScale : -INFINITY;
      s[h][1] = p + 1 <= pa ? c[1] * kScale : -INFINITY;
      s[h][2] = p <= pb ? c[2] * kScale : -INFINITY;
      s[h][3] = p + 1 <= pb ? c[3] * kScale : -INFINITY;
    }
    const float mn_a = fmaxf(m_a, quad_max(fmaxf(fmaxf(s[0][0], s[0][1]), fmaxf(s[1][0], s[1][1]))));
    const float mn_b = fmaxf(m_b, quad_max(fmaxf(fmaxf(s[0][2], s[0][3]), fmaxf(s[1][2], s[1][3]))));
    const float mu_a = mn_a == -INFINITY ? 0.f : mn_a, mu_b = mn_b == -INFINITY ? 0.f : mn_b;
    const float f_a = __expf(m_a - mu_a), f_b = __expf(m_b - mu_b);
    m_a = mn_a;
    m_b = mn_b;
    uint32_t p[4];
    float sum_a = 0.f, sum_b = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      p[2 * h] = bf16_pair(__expf(s[h][0] - mu_a), __expf(s[h][1] - mu_a));
      p[2 * h + 1] = bf16_pair(__expf(s[h][2] - mu_b), __expf(s[h][3] - mu_b));
      sum_a += bf_lo(p[2 * h]) + bf_hi(p[2 * h]);
      sum_b += bf_lo(p[2 * h + 1]) + bf_hi(p[2 * h + 1]);
    }
    l_a = l_a * f_a + sum_a;
    l_b = l_b * f_b + sum_b;
    const uint32_t v_row = smem_u32(sV + (lane & 15) * kStride);
#pragma unroll
    for (int d = 0; d < kHd / 8; ++d) {
      acc[d][0] *= f_a;
      acc[d][1] *= f_a;
      acc[d][2] *= f_b;
      acc[d][3] *= f_b;
      uint32_t v0, v1;
      load_transposed(v_row + d * 16, v0, v1);
      mma(acc[d], p, v0, v1);
    }
    __syncwarp();                          // every lane is done with this slot
    if (j + kBuf < n) {
      if (((j + kBuf) & 31) == 0) load_ids(j + kBuf);
      issue(j + kBuf, w_lo, INT_MAX, w_hi);
    }
    copies_commit();
  }
  copies_wait<0>();
  __syncwarp();
  l_a = quad_sum(l_a);
  l_b = quad_sum(l_b);
  float* part = reinterpret_cast<float*>(wkv);          // [kQv][kAcc], over the warp's buffers
#pragma unroll
  for (int d = 0; d < kHd / 8; ++d) {
    *reinterpret_cast<float2*>(part + g8 * kAcc + d * 8 + 2 * t4) = make_float2(acc[d][0], acc[d][1]);
    *reinterpret_cast<float2*>(part + (g8 + 8) * kAcc + d * 8 + 2 * t4) = make_float2(acc[d][2], acc[d][3]);
  }
  if (t4 == 0) {
    sML[warp * kQv + g8] = make_float2(m_a, l_a);
    sML[warp * kQv + g8 + 8] = make_float2(m_b, l_b);
  }
  __syncthreads();
  // the warps' partials in warp order, 4 dimensions a thread
  const int qv = tid >> 4, c4 = tid & 15;
  if (qv < nqv) {
    float2 ml[kWarps];
    float M = -INFINITY, L = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      ml[w] = sML[w * kQv + qv];
      M = fmaxf(M, ml[w].x);
    }
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float f = ml[w].x == -INFINITY ? 0.f : __expf(ml[w].x - M);
      const float4 x = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(sKV + w * kWarpBytes) + qv * kAcc + c4 * 4);
      L = fmaf(f, ml[w].y, L);
      o.x = fmaf(f, x.x, o.x);
      o.y = fmaf(f, x.y, o.y);
      o.z = fmaf(f, x.z, o.z);
      o.w = fmaf(f, x.w, o.w);
    }
    const float inv = 1.f / L;
    bf16* out = static_cast<bf16*>(a.out) + (static_cast<size_t>(r0 + qv / G) * a.H + kvh * G + qv % G) * kHd + c4 * 4;
    *reinterpret_cast<uint2*>(out) = make_uint2(bf16_pair(o.x * inv, o.y * inv), bf16_pair(o.z * inv, o.w * inv));
  }
}

}  // namespace

// Which decode launches are this kernel's: few query vectors (heads of 64), and either many CTAs, whose splits
// would only add merges, or short contexts; few CTAs over long contexts need the splits of the other kernels. By
// the positions expected, us here / on the kernel of attention.cu, 1 row, 4 heads per KV head:
//   8 CTAs (one sequence, 8 KV heads)  128: 2.7 / 3.7, 300: 3.6 / 3.8, 700: 5.1 / 4.3
//   32                                 300: 3.6 / 4.9, 700: 5.1 / 5.5, 1300: 7.9 / 7.4
//   64                                 700: 5.2 / 7.4, 1300: 7.9 / 14.3, 2500: 14.0 / 15.2, 5000: 25.6 / 33.0
//   128                                128: 2.9 / 5.3, 700: 5.2 / 9.3, 1300: 8.7 / 15.2, 5000: 27.1 / 47.4
//   256                                700: 7.8 / 13.2, 1300: 12.7 / 23.9, 5000: 53.3 / 88.1
//   flat mode, 64                      137..500: 4.3 / 7.5, 1000..3000: 16.1 / 15.6
//   flat mode, 128 and 256             137..1289: 8.7 / 12.5, 13.0 / 18.5
// (7 heads per KV head, 2 KV heads: the same lines to within 0.3 us.)
bool attention_few_takes(const AttnArgs& a) {
  if (!a.pre_len || a.hd != kHd || a.n_ctx_clusters > 1 || a.max_rows * (a.H / a.kv.Hkv) > kQv) return false;
  const uintptr_t al = reinterpret_cast<uintptr_t>(a.kv.pool) | reinterpret_cast<uintptr_t>(a.q) | reinterpret_cast<uintptr_t>(a.out);
  if ((al & 15) || a.n_groups > 65535) return false;
  const long ctas = static_cast<long>(a.n_groups) * a.kv.Hkv, covered = static_cast<long>(a.n_splits) * a.chunk;
  const long ctx = a.ctx > 0 ? std::min<long>(a.ctx, covered) : covered;
  if (ctas > 2L * sm_count_cached()) return false;       // one wave
  return a.flat > 0 ? ctas >= 128 || (ctas >= 32 && ctx <= 2048) || ctx <= 512
                    : ctas >= 64 || (ctas >= 32 && ctx <= 1024) || ctx <= 320;
}

namespace {
template <int BUF>
cudaError_t launch_few(const AttnArgs& a, cudaStream_t st) {
  static const cudaError_t configured =
      cudaFuncSetAttribute(attn_few_kernel<BUF>, cudaFuncAttributeMaxDynamicSharedMemorySize, FewCfg<BUF>::SMEM);
  if (configured != cudaSuccess) return configured;
  return launch_pdl(attn_few_kernel<BUF>, dim3(a.kv.Hkv, a.n_groups), dim3(kThreads), FewCfg<BUF>::SMEM, st, a);
}
}  // namespace

cudaError_t attention_few(const AttnArgs& a, cudaStream_t st) {
  return a.n_groups * a.kv.Hkv <= sm_count_cached() ? launch_few<6>(a, st) : launch_few<3>(a, st);
}

}  // namespace sd2
