// GEMM over many token rows (prompts, and the verify blocks of larger batches) on the
// 5th-generation tensor cores, with CTA pairs: Y[m, n] = sum_k X[m, k] W[n, k] and the decoder's
// fused epilogues (store, residual add with the RMSNorm producer, steered SwiGLU of Eq. 2, SiLU).
//
// With many token rows the projection is a full contraction, bound by the tensor cores and by what
// feeds them from shared memory, no longer by the weight stream. So the tokens are the M side: a
// cluster of two CTAs computes 256 tokens x 256 weight rows with tcgen05.mma.cta_group::2 (M = 256,
// N = 256). Each CTA stages 128 token rows and 128 weight rows per 64-column k-block (32 KB), half
// of what one CTA alone would have to stage and read per MMA for the same output; TMEM holds two
// 256-column accumulators, so the epilogue of one tile runs under the MMAs of the next. A thread of
// the epilogue owns one token row (TMEM lane): gate and up of a feature, the row's RMSNorm scale,
// its sum of squares and its contiguous output features are all in its own registers, and it
// requests the global operands of 32 columns at once before it needs any.
// It takes over from the weights-as-M kernel of gemm_tc.cu above 128 rows (kWideMinRows): there a
// 128-row gate/up of the 8B width is still as fast (53.0 against 52.4 us), 144 rows are not (64.1
// against 51.7), and its whole-tile epilogue, 16 columns at a time with dependent loads and stores,
// made 256 rows x 14336 -> 4096 231 us (34.9 here). Gate/up of 2000 rows x 4096 -> 2 x 14336: in a
// short burst 394 -> 252 us (1.86 PFLOP/s; cuBLAS 1.94 on 8192^3), in a long run, at the clocks that
// the power limit leaves, 420 -> 290 (1.62; cuBLAS 1.75); bursts of 8000 rows 1507 -> 989; 8000 rows
// x 14336 -> 4096 1009 -> 522; x 4096 -> 6144 280 -> 235. Prefill of 8352 prompt tokens through the
// 8B/1B pair 206 -> 100 ms, of 512 25.6 -> 9.7.
// Between 129 and 192 rows short and very long weight matrices stay there (weights_as_m_rows).
//
// Work split. Tiles are walked in groups of kGroupTiles token tiles, weight tiles slowest, so a
// group's tokens stay in L2 while the weights pass once per group. With fewer tiles than resident
// CTA pairs, the K range of a tile is split over sp <= 4 pairs of one cluster (2 sp CTAs): the
// ranks share the tile's 32-column units out, push each unit's partial to its owner's drained ring
// (distributed shared memory) between two cluster barriers, and the owner sums them in rank order.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "tc.cuh"

namespace sd2 {
namespace {

using namespace tc;

constexpr int kBK = 64;                       // K per stage (128 bytes of bf16)
constexpr int kHalf = 128;                    // token rows, and weight rows, of one CTA of the pair
constexpr int kTileN = 256;                   // weight rows of a tile
constexpr int kTileM = 256;                   // token rows of a tile
constexpr int kStages = 6;
constexpr int kOpBytes = kHalf * kBK * 2;     // one operand of one stage
constexpr int kStageBytes = 2 * kOpBytes;
constexpr int kEpiWarps = 8;                  // two per TMEM lane quarter, taking turns at the units
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kUnits = 8;                     // units of 32 accumulator columns in a tile
constexpr int kMaxSplit = 4;
constexpr int kGroupTiles = 8;                // token tiles walked together
constexpr int kPatchBytes = 32 * 32 * 4;       // a warp's transposing patch of the f32 epilogues
constexpr int kSmem = 1024 + kStages * kStageBytes + kEpiWarps * kPatchBytes + 512;

struct WideArgs {
  CUtensorMap mapX;
  CUtensorMap mapW[3];
  int seg_rows[3];
  int nseg;
  int M, N, KB, n_tt, n_wt, tiles, sp;        // N: output features (SwiGLU: gate features)
  int weights_once;                           // every weight tile is read by one tile only
  float* out;
  int ldo;
  bf16* out_bf;
  int ldh;
  const float* bias;
  int ld_bias;
  const int* row_seq;
  unsigned* err;
  unsigned long long* stamp;
  const bf16* norm_gamma;
  bf16* norm_out;
  float* norm_ssq_out;
  float* tap;
  const int* tap_row;
  int tap_mask;
  const float* norm_ssq_in;
  int norm_parts, norm_d;
  float norm_eps;
  int ld_ssq;
  // EPI_QKV
  float* q_out;
  bf16* kv_pool;
  const int* kv_table;
  int kv_bt_stride, kv_n_blocks, n_heads, n_kv_heads, head_dim, layer;
  const float* rope_cs;
  const int* row_pos;
  const int* row_valid;
};

// ------------------------------------------------------------------------------ cta_group::2 PTX
__device__ __forceinline__ void tmem_alloc2(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void mma2_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
          d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrives on the mbarrier at this shared-memory offset in every CTA of `mask` (cluster ranks)
__device__ __forceinline__ void mma2_commit(uint32_t bar, uint16_t mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"(mask)
      : "memory");
}
// TMA tile load into this CTA's shared memory, completing on `bar` (a shared::cluster address: the
// pair's leader)
__device__ __forceinline__ void tma2_load(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma2_load_hint(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar,
                                               uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
      "[%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// two groups of 16 accumulator columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld_2x16(uint32_t ta, uint32_t tb, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(ta));
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(tb));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Unit u of a tile: 32 accumulator columns of which the first 16 start at column col_a and the
// others at col_b; it yields `out_cols` output features from feature0 on. SwiGLU: 16 gate and the
// matching 16 up columns; QKV: 16 dimensions of a head and their rotate-half partners, hd / 2 = `half` on;
// otherwise 32 consecutive columns.
template <int E>
struct Unit {
  static constexpr int out_cols = E == EPI_SWIGLU ? 16 : 32;
  __device__ static uint32_t col_a(int u, int half) {
    return static_cast<uint32_t>(E == EPI_QKV ? u * 16 / half * 2 * half + u * 16 % half : out_cols * u);
  }
  __device__ static uint32_t col_b(int u, int half) {
    return E == EPI_QKV ? col_a(u, half) + static_cast<uint32_t>(half)
                        : static_cast<uint32_t>(E == EPI_SWIGLU ? 128 + 16 * u : 32 * u + 16);
  }
  __device__ static int feature0(int wt, int u, int half) {
    return E == EPI_QKV ? wt * kTileN + static_cast<int>(col_a(u, half)) : wt * (kUnits * out_cols) + u * out_cols;
  }
};

// Unit u's accumulators: of the accumulator at tbase, or (two) the sum of it and the next one.
template <int E>
__device__ __forceinline__ void read_unit(uint32_t tbase, int u, int half, bool two, float (&v)[32]) {
  tmem_ld_2x16(tbase + Unit<E>::col_a(u, half), tbase + Unit<E>::col_b(u, half), v);
  if (two) {
    float w[32];
    tmem_ld_2x16(tbase + kTileN + Unit<E>::col_a(u, half), tbase + kTileN + Unit<E>::col_b(u, half), w);
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] += w[i];
  }
}

__device__ __forceinline__ unsigned long long wide_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ float silu(float y) { return y / (1.f + __expf(-y)); }
// 8 f32 as 8 bf16
__device__ __forceinline__ uint4 pack8(const float* v) {
  return make_uint4(bf16_pair(v[0], v[1]), bf16_pair(v[2], v[3]), bf16_pair(v[4], v[5]), bf16_pair(v[6], v[7]));
}

// Tile t -> (token tile, weight tile): groups of kGroupTiles token tiles, weight tiles slowest.
__device__ __forceinline__ void tile_of(const WideArgs& a, int t, int& tt, int& wt) {
  const int per = kGroupTiles * a.n_wt, g = t / per, r = t - g * per;
  const int gsz = min(kGroupTiles, a.n_tt - g * kGroupTiles);
  wt = r / gsz;
  tt = g * kGroupTiles + (r - wt * gsz);
}
// Epilogues with f32 outputs (STORE, ADD) leave TMEM with a lane per token row, but a warp's loads
// and stores of `out` take a token row's 128 bytes of a unit by 8 lanes x 16 bytes, 4 rows at a time:
// the unit's 32 x 32 accumulators are turned through a 4 KB patch of shared memory per warp (chunks of
// 16 bytes, xor-ed with the row, so neither side conflicts). With 16-byte stores straight from the
// row lanes (32 rows, half a sector each) the f32 epilogue took longer than the tile's MMAs at
// K = 4096 (8000 x 6144 rows: 294 us).
// The residuals and the RMSNorm gain of one unit, requested before its accumulators are read:
struct Ops {
  float4 r[8];      // rows 4 i + lane / 8, features 4 (lane % 8) ..
  uint2 g;          // gains of those features
};
template <int E>
__device__ __forceinline__ void load_ops(const WideArgs& a, int m0, int n, int lane, Ops& o) {
  if (E != EPI_ADD || n >= a.N) return;
  const float* x = a.out + static_cast<size_t>(m0 + (lane >> 3)) * a.ldo + n + (lane & 7) * 4;
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (m0 + 4 * i + (lane >> 3) < a.M) o.r[i] = *reinterpret_cast<const float4*>(x + static_cast<size_t>(4 * i) * a.ldo);
  if (a.norm_out) o.g = __ldg(reinterpret_cast<const uint2*>(a.norm_gamma + n) + (lane & 7));
}
// Epilogue of one unit of a warp's 32 token rows from m0 on: v holds the lane's row's 32 summed
// accumulators, scaled. ss[i] collects the squares of row 4 i + lane / 8 over the lane's features.
template <int E>
__device__ __forceinline__ void emit_rows(const WideArgs& a, float4* patch, int m0, int n, int lane,
                                          const float (&v)[32], const Ops& o, float (&ss)[8]) {
  __syncwarp();                          // the patch's previous unit has been read
#pragma unroll
  for (int i = 0; i < 8; ++i)
    patch[lane * 8 + (i ^ (lane & 7))] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
  __syncwarp();
  const int c = lane & 7;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = 4 * i + (lane >> 3), m = m0 + r;
    float4 y = patch[r * 8 + (c ^ (r & 7))];
    if (m >= a.M) continue;
    const size_t at = static_cast<size_t>(m) * a.ldo + n + 4 * c;
    if (E == EPI_ADD) {
      if (a.bias) {
        const float4 b = *reinterpret_cast<const float4*>(
            a.bias + static_cast<size_t>(a.row_seq ? a.row_seq[m] : 0) * a.ld_bias + n + 4 * c);
        y.x += b.x; y.y += b.y; y.z += b.z; y.w += b.w;
      }
      y.x = o.r[i].x + y.x; y.y = o.r[i].y + y.y; y.z = o.r[i].z + y.z; y.w = o.r[i].w + y.w;
    }
    *reinterpret_cast<float4*>(a.out + at) = y;
    if (E == EPI_ADD && a.norm_out) {
      ss[i] += (y.x * y.x + y.y * y.y) + (y.z * y.z + y.w * y.w);
      *reinterpret_cast<uint2*>(a.norm_out + at) =
          make_uint2(bf16_pair(y.x * bf_lo(o.g.x), y.y * bf_hi(o.g.x)), bf16_pair(y.z * bf_lo(o.g.y), y.w * bf_hi(o.g.y)));
      if (a.tap_mask) {
        const int tr = a.tap_row ? a.tap_row[m] : m;
        if (tr >= 0)
          for (int s = 0; s < 3; ++s)
            if (a.tap_mask & (1 << s))
              *reinterpret_cast<float4*>(a.tap + (static_cast<size_t>(tr) * 3 + s) * a.ldo + n + 4 * c) = y;
      }
    }
  }
}
// The rows' sums of squares over the warp's units -> slice `part`.
__device__ __forceinline__ void emit_squares(const WideArgs& a, int part, int m0, int lane, const float (&ss)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float s = ss[i];
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    const int m = m0 + 4 * i + (lane >> 3);
    if ((lane & 7) == 0 && m < a.M) a.norm_ssq_out[static_cast<size_t>(part) * a.ld_ssq + m] = s;
  }
}
// bf16 outputs (SwiGLU: 16 features of a unit, SiLU: 32) go straight from the row lanes, 32 or 64
// contiguous bytes a lane.
template <int E>
__device__ __forceinline__ void emit_bf16(const WideArgs& a, int m, int n, float (&v)[32]) {
  if (m >= a.M) return;
  const float* b = a.bias ? a.bias + static_cast<size_t>(a.row_seq ? a.row_seq[m] : 0) * a.ld_bias + n : nullptr;
  constexpr int nb = Unit<E>::out_cols;
  float h[nb];
#pragma unroll
  for (int i = 0; i < nb; i += 4) {
    const float4 b4 = b ? *reinterpret_cast<const float4*>(b + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    const float bi[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (E == EPI_SWIGLU) {               // Eq. 2: v = gate of 16 features, then their up
        const float g = v[i + j], up = v[16 + ((i + j) & 15)] + bi[j];
        h[i + j] = up * (g / (1.f + __expf(-g)));
      } else {
        h[i + j] = silu(v[i + j] + bi[j]);
      }
    }
  }
  uint4* d = reinterpret_cast<uint4*>(a.out_bf + static_cast<size_t>(m) * a.ldh + n);
#pragma unroll
  for (int i = 0; i < nb / 8; ++i) d[i] = pack8(h + 8 * i);
}

// q, k and v: v holds 16 dimensions of one head from feature n on, then their rotate-half partners. q and k
// are rotated to the row's position; q goes out in f32 through the patch (64 contiguous bytes by 4 lanes),
// k and v in bf16 to the row's place in the paged cache, 32 bytes twice a lane.
__device__ __forceinline__ void emit_qkv(const WideArgs& a, float4* patch, int m0, int n, int lane, float (&v)[32]) {
  const int hd = a.head_dim, half = hd >> 1, head = n / hd, i0 = n % hd, m = m0 + lane;
  const bool rotated = head < a.n_heads + a.n_kv_heads;
  const int pos = m < a.M ? a.row_pos[m] : 0;
  if (rotated && m < a.M) {
    const float4* cs = reinterpret_cast<const float4*>(a.rope_cs + (static_cast<size_t>(pos) * half + i0) * 2);
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      const float4 c = cs[i >> 1];           // (cos, sin) of two dimensions
      const float x0 = v[i], x1 = v[16 + i], y0 = v[i + 1], y1 = v[17 + i];
      v[i] = x0 * c.x - x1 * c.y;
      v[16 + i] = x1 * c.x + x0 * c.y;
      v[i + 1] = y0 * c.z - y1 * c.w;
      v[17 + i] = y1 * c.z + y0 * c.w;
    }
  }
  if (head < a.n_heads) {
    __syncwarp();                            // the patch's previous unit has been read
#pragma unroll
    for (int i = 0; i < 8; ++i)
      patch[lane * 8 + (i ^ (lane & 7))] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    __syncwarp();
    const int c = lane & 7, d = i0 + (c < 4 ? 4 * c : half + 4 * (c - 4));
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = 4 * i + (lane >> 3);
      if (m0 + r < a.M)
        *reinterpret_cast<float4*>(a.q_out + (static_cast<size_t>(m0 + r) * a.n_heads + head) * hd + d) = patch[r * 8 + (c ^ (r & 7))];
    }
  } else if (m < a.M && a.row_valid[m]) {
    const int kv = (head - a.n_heads) / a.n_kv_heads, kvh = (head - a.n_heads) % a.n_kv_heads;   // kv 0: K, 1: V
    const int block = a.kv_table[static_cast<size_t>(a.row_seq[m]) * a.kv_bt_stride + (pos >> 4)];
    bf16* dst = a.kv_pool + (((static_cast<size_t>(a.layer) * a.kv_n_blocks + block) * 2 + kv) * a.n_kv_heads + kvh) * 16 * hd +
                (pos & 15) * hd + i0;
    reinterpret_cast<uint4*>(dst)[0] = pack8(v);
    reinterpret_cast<uint4*>(dst)[1] = pack8(v + 8);
    reinterpret_cast<uint4*>(dst + half)[0] = pack8(v + 16);
    reinterpret_cast<uint4*>(dst + half)[1] = pack8(v + 24);
  }
}

template <int E>
__global__ void __launch_bounds__(kThreads, 1) gemm_wide_kernel(const __grid_constant__ WideArgs a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes + kEpiWarps * kPatchBytes);
  // bars: full[S] (leader's), empty[S], tfull[2], tempty[2] (leader's), drain
  volatile int* flags = reinterpret_cast<volatile int*>(bars + 2 * kStages + 5);   // [0] abort, [1] TMEM base, [2] consumed
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kStages, tfull0 = empty0 + 8 * kStages,
                 tempty0 = tfull0 + 16, drain = tempty0 + 16;
  volatile int* abort_flag = flags;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sp = a.sp, crank = static_cast<int>(cluster_rank());
  const int par = crank & 1, p = crank >> 1;            // CTA of the pair, split rank of the pair
  const uint32_t lead = static_cast<uint32_t>(crank & ~1);
  const int cluster = static_cast<int>(blockIdx.x) / (2 * sp), n_clusters = static_cast<int>(gridDim.x) / (2 * sp);
  // A cluster with one tile adds the halves of its K range up in an accumulator each (summed by the
  // epilogue): the tensor core truncates as it accumulates, so the error grows with the length of the
  // chain. With several tiles the second accumulator lets the epilogue run under the next tile's MMAs.
  const bool two_acc = a.tiles <= n_clusters && a.KB >= 2 * sp;
  constexpr uint32_t ncols = 2 * kTileN;
  if (a.stamp && threadIdx.x == 0) atomicMin(&a.stamp[0], wide_ns());
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(tfull0, 1);
    mbar_init(tfull0 + 8, 1);
    mbar_init(tempty0, 2 * kEpiWarps);
    mbar_init(tempty0 + 8, 2 * kEpiWarps);
    mbar_init(drain, 1);
    flags[0] = 0;
    flags[2] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc2(smem_u32(const_cast<int*>(flags) + 1), ncols);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                     // every barrier of the cluster is initialised before any remote signal
  tc_fence_after();
  const uint32_t tmem = static_cast<uint32_t>(flags[1]);
  const int kb_lo = p * a.KB / sp, nkb = (p + 1) * a.KB / sp - kb_lo;
  pdl_trigger();

  const int q = warp & 3, half = (warp - 2) >> 2;        // epilogue: TMEM lane quarter, turn at the units
  const int row = q * 32 + lane;                         // token row within this CTA's 128
  const uint32_t tlane = static_cast<uint32_t>(q * 32) << 16;
  const int hd2 = E == EPI_QKV ? a.head_dim >> 1 : 1;    // rotate-half distance
  bool done = true;                                      // split-K: this CTA's accumulator completed
  float rs = 1.f;

  // Sum of squares slices -> the row scale of the consumer side of a fused RMSNorm.
  auto row_scale = [&](int m) {
    float s = 0.f;
    if (m < a.M) {
      const float* src = a.norm_ssq_in + m;
      for (int p0 = 0; p0 < a.norm_parts; p0 += 32) {
        float v[32];
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] = src[static_cast<size_t>(min(p0 + u, a.norm_parts - 1)) * a.ld_ssq];
#pragma unroll
        for (int u = 0; u < 32; ++u) s = p0 + u < a.norm_parts ? s + v[u] : s;
      }
    }
    return rsqrtf(s / static_cast<float>(a.norm_d) + a.norm_eps);
  };
  // One unit of a tile, from its summed accumulators.
  float4* patch = reinterpret_cast<float4*>(smem + kStages * kStageBytes) + (warp - 2) * (kPatchBytes / 16);
  auto emit = [&](int m0, int n, float (&v)[32], const Ops& o, float (&ss)[8]) {
    if (n >= a.N) return;
    if (a.norm_ssq_in)
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] *= rs;
    if constexpr (E == EPI_STORE || E == EPI_ADD) emit_rows<E>(a, patch, m0, n, lane, v, o, ss);
    else if constexpr (E == EPI_QKV) emit_qkv(a, patch, m0, n, lane, v);
    else emit_bf16<E>(a, m0 + lane, n, v);
  };

  if (warp == 0) {
    if (lane == 0) {
      const uint64_t wpol = l2_evict_first();
      const uint32_t full_lead = dsmem_addr(full0, lead);
      int n_my = 0;
      for (int t = cluster; t < a.tiles; t += n_clusters) ++n_my;
      const int n_units = n_my * nkb;
      struct Cur {
        int t, kb, tt, wt, seg, row0;
      };
      auto locate = [&](Cur& c) {
        tile_of(a, c.t, c.tt, c.wt);
        if (E == EPI_SWIGLU) {               // CTA 0 stages the gate rows, CTA 1 the up rows
          c.seg = par;
          c.row0 = c.wt * kHalf;
        } else {                             // rows past the last segment read as zeros
          c.seg = 0;
          c.row0 = c.wt * kTileN + par * kHalf;
          while (c.seg + 1 < a.nseg && c.row0 >= a.seg_rows[c.seg]) c.row0 -= a.seg_rows[c.seg++];
        }
      };
      auto advance = [&](Cur& c) {
        if (++c.kb == nkb) {
          c.kb = 0;
          c.t += n_clusters;
          if (c.t < a.tiles) locate(c);
        }
      };
      auto load_w = [&](int s, const Cur& c) {
        const uint32_t dst = smem_u32(smem) + s * kStageBytes + kOpBytes;
        if (a.weights_once) tma2_load_hint(dst, &a.mapW[c.seg], (kb_lo + c.kb) * kBK, c.row0, full_lead + 8 * s, wpol);
        else tma2_load(dst, &a.mapW[c.seg], (kb_lo + c.kb) * kBK, c.row0, full_lead + 8 * s);
      };
      auto load_x = [&](int s, const Cur& c) {
        tma2_load(smem_u32(smem) + s * kStageBytes, &a.mapX, (kb_lo + c.kb) * kBK, c.tt * kTileM + par * kHalf,
                  full_lead + 8 * s);
      };
      Cur c{cluster, 0, 0, 0, 0, 0};
      if (c.t < a.tiles) locate(c);
      // the first stages' weights never depend on earlier kernels: requested before the wait
      const int pre = min(n_units, kStages);
      Cur cx = c;
      for (int j = 0; j < pre; ++j, advance(c)) {
        if (par == 0) mbar_expect_tx(full0 + 8 * j, 2 * kStageBytes);
        load_w(j, c);
      }
      pdl_wait();
      if (a.stamp) atomicMin(&a.stamp[1], wide_ns());
      for (int j = 0; j < pre; ++j, advance(cx)) load_x(j, cx);
      int j = pre, s = pre % kStages;
      uint32_t ph = (pre / kStages) & 1;
      bool ok = true;
      for (; j < n_units; ++j, advance(c)) {
        if (!wait_bar(empty0 + 8 * s, ph ^ 1, abort_flag, a.err)) { ok = false; break; }
        if (par == 0) mbar_expect_tx(full0 + 8 * s, 2 * kStageBytes);
        load_w(s, c);
        load_x(s, c);
        if (++s == kStages) { s = 0; ph ^= 1u; }
      }
      if (!ok && par == 0)                   // let the loads already issued land before the pair exits
        for (int jj = flags[2]; jj < j; ++jj)
          wait_bar_budget(full0 + 8 * (jj % kStages), (jj / kStages) & 1, kDrainCycles);
    }
  } else if (warp == 1) {
    if (lane == 0 && par == 0) {
      const uint32_t idesc = idesc_bf16(kTileM, kTileN);
      const uint64_t desc0 = sw128_desc(smem_u32(smem));
      const uint16_t pair = static_cast<uint16_t>(3u << lead);
      int s = 0, j = 0, seg = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = cluster; t < a.tiles && ok; t += n_clusters, ++seg) {
        const int acc = seg & 1;
        if (!wait_bar(tempty0 + 8 * acc, ((seg >> 1) & 1) ^ 1, abort_flag, a.err)) break;
        tc_fence_after();
        const int k_half = two_acc ? (nkb + 1) / 2 : nkb;   // k-blocks of the first accumulator
        for (int i = 0; i < nkb; ++i, ++j) {
          const uint32_t d = tmem + (two_acc ? (i >= k_half ? kTileN : 0) : acc * kTileN);
          if (!wait_bar(full0 + 8 * s, ph, abort_flag, a.err)) { ok = false; break; }
          tc_fence_after();
          const uint64_t ad = desc0 + static_cast<uint64_t>(s * (kStageBytes >> 4)), bd = ad + (kOpBytes >> 4);
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk)
            mma2_bf16(d, ad + 2 * kk, bd + 2 * kk, idesc, ((i > 0 && i != k_half) || kk > 0) ? 1u : 0u);
          mma2_commit(empty0 + 8 * s, pair);
          flags[2] = j + 1;
          if (++s == kStages) { s = 0; ph ^= 1u; }
        }
        if (ok) mma2_commit(tfull0 + 8 * acc, pair);
      }
      mma2_commit(drain, static_cast<uint16_t>(1u << lead));   // every MMA issued here has completed
      wait_bar_budget(drain, 0, kDrainCycles);
    }
  } else {
    pdl_wait();                              // outputs, residuals and biases come from earlier kernels
    if (sp == 1) {
      const uint32_t tempty_lead = dsmem_addr(tempty0, lead);
      int seg = 0, rs_tt = -1;
      for (int t = cluster; t < a.tiles; t += n_clusters, ++seg) {
        const int acc = seg & 1;
        int tt, wt;
        tile_of(a, t, tt, wt);
        const int m0 = tt * kTileM + par * kHalf + q * 32;
        if (a.norm_ssq_in && tt != rs_tt) {  // the row's RMSNorm scale, while the tile's MMAs run
          rs = row_scale(m0 + lane);
          rs_tt = tt;
        }
        Ops o;
        load_ops<E>(a, m0, Unit<E>::feature0(wt, half, hd2), lane, o);
        if (!__all_sync(0xffffffffu, wait_bar(tfull0 + 8 * acc, (seg >> 1) & 1, abort_flag, a.err))) break;
        tc_fence_after();
        float ss[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int u = half; u < kUnits; u += 2) {
          float v[32];
          read_unit<E>(tmem + tlane + (two_acc ? 0 : acc * kTileN), u, hd2, two_acc, v);
          emit(m0, Unit<E>::feature0(wt, u, hd2), v, o, ss);
          if (u + 2 < kUnits) load_ops<E>(a, m0, Unit<E>::feature0(wt, u + 2, hd2), lane, o);
        }
        if (E == EPI_ADD && a.norm_out) emit_squares(a, 2 * wt + half, m0, lane, ss);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(tempty_lead + 8 * acc);
      }
    } else {
      int tt, wt;
      tile_of(a, cluster, tt, wt);
      if (a.norm_ssq_in) rs = row_scale(tt * kTileM + par * kHalf + row);
      done = __all_sync(0xffffffffu, wait_bar(tfull0, 0, abort_flag, a.err));
    }
  }

  __syncwarp();
  if (sp > 1) {
    // Split-K exchange. Every rank's accumulator is complete (its MMAs no longer read any ring of
    // the pair) before partials land in the rings.
    cluster_sync_all();
    int tt, wt;
    tile_of(a, cluster, tt, wt);
    const int m0 = tt * kTileM + par * kHalf + q * 32;
    const int umax = (kUnits + sp - 1) / sp;
    const int u_lo = p * kUnits / sp, u_hi = (p + 1) * kUnits / sp;
    Ops o;
    if (warp >= 2 && done) {
      tc_fence_after();
      load_ops<E>(a, m0, Unit<E>::feature0(wt, u_lo + half, hd2), lane, o);
      for (int u = half; u < kUnits; u += 2) {
        const int own = ((u + 1) * sp - 1) / kUnits;   // the rank with own kUnits / sp <= u < (own + 1) kUnits / sp
        if (own == p) continue;
        float v[32];
        read_unit<E>(tmem + tlane, u, hd2, two_acc, v);
        const int slot = p < own ? p : p - 1, ul = u - own * kUnits / sp;
        const uint32_t dst = smem_u32(smem) + static_cast<uint32_t>((slot * umax + ul) * 8 * kHalf + row) * 16;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          st_dsmem_v4(dst + i * kHalf * 16, static_cast<uint32_t>(2 * own + par), v[4 * i], v[4 * i + 1], v[4 * i + 2],
                      v[4 * i + 3]);
      }
    }
    __syncwarp();
    cluster_sync_all();
    if (warp >= 2 && done) {
      float ss[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int u = u_lo + half; u < u_hi; u += 2) {
        float acc[32], v[32];
        read_unit<E>(tmem + tlane, u, hd2, two_acc, acc);
        const float4* rc = reinterpret_cast<const float4*>(smem) + (u - u_lo) * 8 * kHalf + row;
        for (int r = 0; r < sp; ++r) {       // in rank order
          const float4* src = rc + (r < p ? r : r - 1) * umax * 8 * kHalf;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float4 x = r == p ? make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]) : src[i * kHalf];
            v[4 * i] = r ? v[4 * i] + x.x : x.x;
            v[4 * i + 1] = r ? v[4 * i + 1] + x.y : x.y;
            v[4 * i + 2] = r ? v[4 * i + 2] + x.z : x.z;
            v[4 * i + 3] = r ? v[4 * i + 3] + x.w : x.w;
          }
        }
        emit(m0, Unit<E>::feature0(wt, u, hd2), v, o, ss);
        if (u + 2 < u_hi) load_ops<E>(a, m0, Unit<E>::feature0(wt, u + 2, hd2), lane, o);
      }
      if (E == EPI_ADD && a.norm_out) emit_squares(a, (wt * sp + p) * 2 + half, m0, lane, ss);
    }
    __syncwarp();
  }
  tc_fence_before();
  cluster_sync_all();                        // no CTA leaves while its pair still signals or reads it
  tc_fence_after();
  if (warp == 1) tmem_dealloc2(tmem, ncols);
  if (a.stamp && threadIdx.x == 0) atomicMax(&a.stamp[2], wide_ns());
}

bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

int out_features(const GemmArgs& g) {
  if (g.epi == EPI_SWIGLU) return g.seg[0].rows;
  int n = 0;
  for (int s = 0; s < g.nseg; ++s) n += g.seg[s].rows;
  return n;
}

struct WidePlan {
  int n_tt, n_wt, tiles, sp, clusters;
};
// Split factor: the one with the least estimated time, in cycles of the tensor core: waves of
// clusters x k-blocks of a tile (512 cycles each at 256 x 256 x 64 over a pair) + the exposed
// epilogue, larger with the split-K exchange. A split tile's cluster must be in the first wave.
WidePlan plan_wide(const GemmArgs& g) {
  WidePlan pl;
  const int N = out_features(g), per = g.epi == EPI_SWIGLU ? kHalf : kTileN, KB = g.K / kBK;
  pl.n_tt = (g.M + kTileM - 1) / kTileM;
  pl.n_wt = (N + per - 1) / per;
  pl.tiles = pl.n_tt * pl.n_wt;
  pl.sp = 0;
  pl.clusters = 0;
  long best = 0;
  for (int sp = 1; sp <= kMaxSplit && (sp == 1 || 2 * sp <= KB); ++sp) {
    const int fit = gemm_max_clusters(2 * sp, kSmem);
    if (fit < 1 || (sp > 1 && pl.tiles > fit)) continue;
    const long waves = (pl.tiles + fit - 1) / fit;
    const long cost = waves * ((KB + sp - 1) / sp) * 512 + (sp > 1 ? 6000 : 3000);
    if (!pl.sp || cost < best) {
      best = cost;
      pl.sp = sp;
      pl.clusters = std::min(pl.tiles, fit);
    }
  }
  return pl;
}

template <int E>
cudaError_t launch_wide(const WideArgs& a, const WidePlan& pl, cudaStream_t st) {
  static const cudaError_t configured =
      cudaFuncSetAttribute(gemm_wide_kernel<E>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (configured != cudaSuccess) return configured;
  return launch_pdl_cluster(gemm_wide_kernel<E>, dim3(static_cast<unsigned>(pl.clusters * 2 * pl.sp)), dim3(kThreads),
                            static_cast<size_t>(kSmem), st, 2 * pl.sp, a);
}

}  // namespace

// Rows up to which the weights-as-M kernel keeps a launch. Against a short weight matrix this kernel's few tiles split
// K four ways on at most 136 SMs, where the other one spreads the same weights over more CTAs; a very long one is a
// weight stream of several waves either way, which the other one starts sooner. Both, us (here / there), weights cold:
//   rows                             144            160            168            192
//     896 x 4864, residual add   14.5 / 11.1    14.5 / 12.3    14.5 / 12.9    14.5 / 13.2    (200: 14.5 / 15.9)
//    1024 x 1024, residual add   10.0 / 9.1     10.1 / 9.7     10.1 / 10.4    10.1 / 10.5
//    2048 x 8192, residual add   19.5 / 16.7    19.5 / 18.6    19.5 / 19.5    19.5 / 24.8
//    2816 x 12800, residual add  25.6 / 22.1    25.6 / 24.6
//    3328 x 12800, residual add  26.0 / 24.0    26.1 / 28.2
//    3840 x 6400, residual add   19.6 / 18.3    19.7 / 20.6
//    4096 x 4096, residual add   17.7 / 15.3    17.6 / 17.0    17.7 / 18.1    17.7 / 18.1
//    4096 x 14336, residual add  33.0 / 29.1    33.1 / 33.1    33.1 / 34.3    33.1 / 34.7
//    4608 x 6400, residual add   21.7 / 19.0    21.7 / 21.3
//    4864 x 6400, residual add   21.9 / 22.3    22.0 / 24.9
//    5120 x 27648, residual add  56.3 / 60.0    56.4 / 68.7    56.3 / 70.3    56.6 / 105
//   32768 x 2048, stored         28.7 / 28.6    28.8 / 29.2    28.8 / 29.8    28.9 / 30.2
//   49152 x 2048, stored         40.3 / 38.4    40.1 / 39.3    40.0 / 39.8    40.7 / 41.1
//  128256 x 2048, stored         99.6 / 96.2   102.2 / 98.6   103.3 / 103.4  105.5 / 106.3
//  151936 x 896, stored          65.1 / 58.3    64.6 / 60.5    65.4 / 63.0    67.3 / 65.8
//   SwiGLU: 1024 x 4096          14.4 / 14.4    14.4 / 15.5;  2048 x 2048 13.7 / 14.1;  14336 x 4096 50.3 / 61.3
// (The other kernel's K splits fit the SMs worst from 3072 to 4095 features: 24 to 31 tiles.)
int weights_as_m_rows(const GemmArgs& g) {
  const int N = out_features(g);
  if (g.epi == EPI_SWIGLU) return N <= 1024 ? 144 : 0;
  if (N < 1024) return 192;
  if (N < 3072 || (N >= 4096 && N <= 4608) || N > 40960) return 160;
  return N < 4096 ? 144 : 0;
}

// Whether gemm_tc runs these arguments (already accepted by gemm_tc_supported) on this kernel.
bool gemm_wide_takes(const GemmArgs& g) {
  if (g.M < kWideMinRows || g.attn_q) return false;
  // the epilogue reads and writes 16 bytes at a time
  if (g.epi == EPI_QKV) {
    if (!al16(g.q_out) || !al16(g.kv_pool) || !al16(g.rope_cs) || (g.head_dim != 64 && g.head_dim != 128)) return false;
  } else if (g.epi == EPI_STORE || g.epi == EPI_ADD) {
    if (!al16(g.out) || g.ldo % 4) return false;
  } else if (!al16(g.out_bf) || g.ldh % 8) {
    return false;
  }
  if (g.epi != EPI_STORE && g.epi != EPI_QKV && g.bias && (!al16(g.bias) || g.ld_bias % 4)) return false;
  if (g.norm_out && (!al16(g.norm_out) || !al16(g.norm_gamma) || g.ldo % 8 || (g.tap_mask && !al16(g.tap)))) return false;
  return g.M > weights_as_m_rows(g) && plan_wide(g).sp > 0;
}

int gemm_wide_norm_parts(const GemmArgs& g) {
  const WidePlan pl = plan_wide(g);
  return pl.n_wt * pl.sp * 2;
}

cudaError_t gemm_wide(const GemmArgs& g, unsigned* err, cudaStream_t st) {
  const WidePlan pl = plan_wide(g);
  if (pl.sp < 1) return cudaErrorInvalidValue;
  WideArgs a{};
  a.nseg = g.nseg;
  for (int s = 0; s < g.nseg; ++s) {
    a.seg_rows[s] = g.seg[s].rows;
    if (!gemm_weight_map(&a.mapW[s], g.seg[s].w, g.seg[s].rows, g.K, kHalf)) return cudaErrorInvalidValue;
  }
  if (!gemm_row_map(&a.mapX, g.x, g.M, g.K, g.ldx, kHalf)) return cudaErrorInvalidValue;
  a.M = g.M; a.N = out_features(g); a.KB = g.K / kBK;
  a.n_tt = pl.n_tt; a.n_wt = pl.n_wt; a.tiles = pl.tiles; a.sp = pl.sp;
  a.weights_once = pl.n_tt == 1;
  a.out = g.out; a.ldo = g.ldo; a.out_bf = static_cast<bf16*>(g.out_bf); a.ldh = g.ldh;
  a.bias = g.bias; a.ld_bias = g.ld_bias; a.row_seq = g.row_seq;
  a.err = err; a.stamp = g.stamp;
  a.norm_gamma = static_cast<const bf16*>(g.norm_gamma); a.norm_out = static_cast<bf16*>(g.norm_out);
  a.norm_ssq_out = g.norm_ssq_out; a.tap = g.tap; a.tap_row = g.tap_row; a.tap_mask = g.tap_mask;
  a.norm_ssq_in = g.norm_ssq_in; a.norm_parts = g.norm_parts; a.norm_d = g.norm_d; a.norm_eps = g.norm_eps;
  a.ld_ssq = g.ld_ssq;
  a.q_out = g.q_out; a.kv_pool = static_cast<bf16*>(g.kv_pool); a.kv_table = g.kv_table;
  a.kv_bt_stride = g.kv_bt_stride; a.kv_n_blocks = g.kv_n_blocks; a.n_heads = g.n_heads;
  a.n_kv_heads = g.n_kv_heads; a.head_dim = g.head_dim; a.layer = g.layer; a.rope_cs = g.rope_cs;
  a.row_pos = g.row_pos; a.row_valid = g.row_valid;
  switch (g.epi) {
    case EPI_STORE: return launch_wide<EPI_STORE>(a, pl, st);
    case EPI_ADD: return launch_wide<EPI_ADD>(a, pl, st);
    case EPI_SWIGLU: return launch_wide<EPI_SWIGLU>(a, pl, st);
    case EPI_SILU: return launch_wide<EPI_SILU>(a, pl, st);
    case EPI_QKV: return launch_wide<EPI_QKV>(a, pl, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sd2
