// Fused multi-head attention over the kept heads only (Eq. 2-3 restricted to
// the DN's head set H; heads outside H were removed from W^Q, W^K, W^V at
// pack time, so this kernel never sees them).
//
// Input: qkv [B, n, 3, h_m, 64] bf16 exactly as the QKV GEMM writes it (q | k |
// v blocks, kept heads in packing order), or [B, n, h_m, 3, 64] when the modes
// share one prefix-ordered packed copy (each head's q, k, v adjacent, so a
// prefix of heads is a prefix of columns). Output: [B, n, h_m * 64] bf16, the
// heads concatenated in the same order (the K axis of the packed W^O).
//
// Persistent kernel; a work item is one (image, kept head) and needs at most
// two 128-query tiles (n <= 256); its unit is one query tile. Items run from
// the last image to the first: the QKV GEMM wrote its rows in increasing order,
// so the most recent (still in L2) are read first. Roles:
//   warp 0      TMA producer: K and V of an item into one of `kv_slots`
//               shared-memory slots, its query tiles into one of two Q
//               buffers per tile (3-D maps: rows past n read as zero);
//   warp 1      tcgen05.mma issuer: S = Q K^T (M=128, N=n_pad, K=64) into the
//               256-column TMEM region of the unit's group, then O = P V with P
//               read from TMEM (M=128, N=64, K=n_pad; V MN-major);
//   warps 2-9   two groups of four, which take the units in turn: one query
//               row per thread (TMEM lane = row). Row max and exp2 numerators
//               over the n valid keys in fp32 (softmax_row); P stored back into
//               TMEM as bf16 pairs over the S columns already consumed; then
//               O row * (1 / row sum) -> bf16, staged in shared memory and
//               stored by 32-row TMA boxes (rows past n are clipped). Warps
//               whose 32 rows are all padding skip the TMEM work.
// The issue order is S(0); then per unit u: S(u+1), PV(u), so the tensor pipe
// computes one group's MMAs while the other runs its softmax. An item's K/V
// slot is released after its last PV, its Q buffers after its last S.
// TMEM per group: S in [0, n_pad), P in [0, n_pad / 2), O in [128, 192) (O
// overwrites S columns the softmax has consumed, so a group's next S waits
// until its O is read out).
// What bounds it: each unit is a serial chain S -> softmax -> PV -> read-out and
// TMEM holds two. ViT-B (256 images, 197 tokens, 12 heads), per unit: softmax
// 2300 clocks (1660 of them the exponentials), PV 1000-1400, scaling and staging
// O 900, S 300; 86.4 -> 61.8 us a call, the memory's share being 46. Before, the
// softmax took 3700 (packed arithmetic and pipelined reads since) and storing
// 16 bytes to each of 32 rows per instruction 1500-2000 (TMA boxes since). With
// one query tile per item the second group had no work: 128 tokens 51.5 -> 34.3
// us, 65 tokens x 3 heads 13.7 -> 7.8.
// Scale 1/sqrt(64) (the base model's head width; it does not change with the
// number of kept heads). Every mbarrier wait is bounded.
#include "common.h"
#include "ptx.cuh"

namespace elasto {

namespace {

constexpr int THREADS = 320;
constexpr int HD = 64;                      // head width d_i
constexpr int QT = 128;                     // queries per tile
constexpr int MAXK = 256;                   // max keys
constexpr int Q_BYTES = QT * HD * 2;        // 16 KB
constexpr int QBUF_BYTES = 4 * Q_BYTES;     // two buffers per query tile
constexpr int O_BYTES = 32 * HD * 2;        // output staging of one softmax warp
constexpr int OBUF_BYTES = 8 * O_BYTES;
constexpr int BAR_BYTES = 256;
constexpr int SMEM_LIMIT = 232448;          // dynamic shared memory per block on sm_103
constexpr int TMEM_COLS = 512;
constexpr int O_COL = 128;

// Shared memory: [Q buffers][output staging][KV slots][barriers], 1024-byte aligned.
__host__ __device__ constexpr int kv_slot_bytes(int n_pad) { return 2 * n_pad * HD * 2; }
__host__ __device__ constexpr int kv_slots_for(int n_pad) {
  return 1024 + QBUF_BYTES + OBUF_BYTES + 3 * kv_slot_bytes(n_pad) + BAR_BYTES <= SMEM_LIMIT ? 3 : 2;
}
__host__ __device__ constexpr int smem_bytes_for(int n_pad) {
  return 1024 + QBUF_BYTES + OBUF_BYTES + kv_slots_for(n_pad) * kv_slot_bytes(n_pad) + BAR_BYTES;
}
__host__ __device__ constexpr int max_smem_bytes() {
  int m = 0;
  for (int n_pad = 16; n_pad <= MAXK; n_pad += 16) m = smem_bytes_for(n_pad) > m ? smem_bytes_for(n_pad) : m;
  return m;
}
static_assert(max_smem_bytes() <= SMEM_LIMIT, "attention shared memory");

constexpr float kScale = 0.125f * 1.4426950408889634f;  // 1/sqrt(64) * log2(e)

__device__ __forceinline__ void load64(uint32_t tm, uint32_t (&v)[2][32]) {
  tmem_ld_32x32b_x32(tm, v[0]);
  tmem_ld_32x32b_x32(tm + 32, v[1]);
}

// Softmax of one score row (this thread's TMEM lane, columns tm .. tm + n):
// the numerators exp2((s - max) * kScale) go back as bf16 pairs over the
// columns already consumed, zeros up to the next multiple of 16; returns their
// fp32 sum. NF = n / 64 whole chunks without masks, then the 1 to 63 columns
// left in masked pieces of 16.
//
// The row is bound by instruction issue and by the TMEM round trips (300 to
// 600 clocks while MMAs run). So: packed fp32 multiply-adds and sums and
// three-input maxima (3 issue slots a score instead of 4.5); nothing read past
// the last piece (n = 197: 208 columns instead of 256, most of the last 64
// masked); each chunk in flight while the one before it is worked on.
template <int NF>
__device__ __forceinline__ float softmax_row(uint32_t tm, int n) {
  float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
  uint32_t v[2][2][32];
  if constexpr (NF > 0) load64(tm, v[0]);
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    tmem_ld_wait();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (i + 1 < NF) tmem_ld_32x32b_x32(tm + 64 * (i + 1) + 32 * h, v[(i + 1) & 1][h]);
#pragma unroll
      for (int j = 0; j < 32; j += 2)
        m[(j >> 1) & 3] = max3(m[(j >> 1) & 3], __uint_as_float(v[i & 1][h][j]), __uint_as_float(v[i & 1][h][j + 1]));
    }
  }
  for (int c = 64 * NF; c < n; c += 16) {
    uint32_t w[16];
    tmem_ld_16(tm + c, w);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (c + j < n) m[j & 3] = fmaxf(m[j & 3], __uint_as_float(w[j]));
  }
  const float neg = -fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])) * kScale;
  const float2 scale2 = make_float2(kScale, kScale), neg2 = make_float2(neg, neg);
  // four partial sums, each of the key pairs 4 i + its number: neighbours are
  // added to one another first, which keeps numerators too small to change the
  // partial sum one by one
  float2 s[2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
  if constexpr (NF > 0) load64(tm, v[0]);
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    tmem_ld_wait();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (i + 1 < NF) tmem_ld_32x32b_x32(tm + 64 * (i + 1) + 32 * h, v[(i + 1) & 1][h]);
      uint32_t pk[16];
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        float2 p[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int e = j + 2 * k;
          const float2 x = fma2(make_float2(__uint_as_float(v[i & 1][h][e]), __uint_as_float(v[i & 1][h][e + 1])),
                                scale2, neg2);
          p[k] = make_float2(ex2_approx(x.x), ex2_approx(x.y));
          pk[e >> 1] = pack_bf16x2(p[k].x, p[k].y);
        }
        s[(j >> 2) & 1] = add2(s[(j >> 2) & 1], add2(make_float2(p[0].x, p[1].x), make_float2(p[0].y, p[1].y)));
      }
      tmem_st_16(tm + 32 * i + 16 * h, pk);
    }
  }
  for (int c = 64 * NF; c < n; c += 16) {
    uint32_t w[16], pk[8];
    tmem_ld_16(tm + c, w);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 16; j += 4) {
      float2 p[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int e = j + 2 * k;
        const float2 x = fma2(make_float2(__uint_as_float(w[e]), __uint_as_float(w[e + 1])), scale2, neg2);
        p[k] = make_float2(c + e < n ? ex2_approx(x.x) : 0.0f, c + e + 1 < n ? ex2_approx(x.y) : 0.0f);
        pk[e >> 1] = pack_bf16x2(p[k].x, p[k].y);
      }
      s[(j >> 2) & 1] = add2(s[(j >> 2) & 1], add2(make_float2(p[0].x, p[1].x), make_float2(p[0].y, p[1].y)));
    }
    tmem_st_8(tm + (c >> 1), pk);
  }
  return (s[0].x + s[0].y) + (s[1].x + s[1].y);
}

__global__ void __launch_bounds__(THREADS, 1)
    attn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmKV,
                   const __grid_constant__ CUtensorMap tmO, int n, int n_pad, int heads, int items, int split,
                   int blk_stride, int head_stride, int* status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int ns = kv_slots_for(n_pad);
  const int slot_bytes = kv_slot_bytes(n_pad);
  uint8_t* qbuf = smem;                                    // [tile][parity] Q_BYTES each
  uint8_t* obuf = smem + QBUF_BYTES;                       // [softmax warp] 32 rows of 128 B
  uint8_t* kvbuf = obuf + OBUF_BYTES;                      // [slot] K then V, n_pad rows of 128 B
  uint64_t* bars = reinterpret_cast<uint64_t*>(kvbuf + ns * slot_bytes);
  uint64_t* full = bars + 0;        // [3] item k's Q, K, V landed (slot k % ns)
  uint64_t* kv_empty = bars + 3;    // [3] slot's PV MMAs finished
  uint64_t* q_empty = bars + 6;     // [2] Q buffers of parity k & 1 consumed by S(k, *)
  uint64_t* s_full = bars + 8;      // [2] the group's S in TMEM
  uint64_t* p_full = bars + 10;     // [2] its P in TMEM (128 arrivals)
  uint64_t* o_full = bars + 12;     // [2] its O in TMEM
  uint64_t* o_empty = bars + 14;    // [2] its O read out (128 arrivals)
  uint64_t* drain = bars + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 17);

  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  // split: an item is one query tile of an (image, head), item & 1
  const int tiles = n > QT && !split ? 2 : 1;
  // items of this CTA: blockIdx.x, blockIdx.x + gridDim.x, ...
  const int nk = items > static_cast<int>(blockIdx.x) ? (items - 1 - blockIdx.x) / gridDim.x + 1 : 0;
  // unit u: query tile u % tiles of item u / tiles, worked on by group u & 1
  const int units = nk * tiles;

  if (threadIdx.x == 0) {
    for (int k = 0; k < 3; ++k) {
      mbar_init(&full[k], 1);
      mbar_init(&kv_empty[k], 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(&q_empty[k], 1);
      mbar_init(&s_full[k], 1);
      mbar_init(&p_full[k], 128);
      mbar_init(&o_full[k], 1);
      mbar_init(&o_empty[k], 128);
    }
    mbar_init(drain, 1);
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = warp_uniform(static_cast<int>(*tmem_slot));
  pdl_wait();  // the set-up above overlapped the previous kernel's tail
  pdl_trigger();

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (elect_one()) {
      tma_prefetch_desc(&tmQ);
      tma_prefetch_desc(&tmKV);
      const uint32_t bytes = tiles * Q_BYTES + 2 * n_pad * HD * 2;
      bool ok = true;
      int k = 0;
      for (; k < nk; ++k) {
        const int item = blockIdx.x + k * gridDim.x;
        const int slot = k % ns, r = items - 1 - item, bh = split ? r >> 1 : r, b = bh / heads, jj = bh - b * heads;
        if (!mbar_wait(&kv_empty[slot], ((k / ns) & 1) ^ 1) || !mbar_wait(&q_empty[k & 1], ((k >> 1) & 1) ^ 1)) {
          ok = false;
          break;
        }
        uint8_t* kb = kvbuf + slot * slot_bytes;
        mbar_expect_tx(&full[slot], bytes);
        const int qx = jj * head_stride;
        tma_load_3d(kb, &tmKV, &full[slot], qx + blk_stride, 0, b);
        tma_load_3d(kb + slot_bytes / 2, &tmKV, &full[slot], qx + 2 * blk_stride, 0, b);
        for (int t = 0; t < tiles; ++t)
          tma_load_3d(qbuf + (2 * t + (k & 1)) * Q_BYTES, &tmQ, &full[slot], qx, (split ? r & 1 : t) * QT, b);
      }
      if (!ok) record_status(status, ELASTO_ERR_TIMEOUT);
      // the loads of the last items have landed before the CTA exits
      for (int j = (k > ns ? k - ns : 0); j < k; ++j) mbar_wait(&full[j % ns], (j / ns) & 1);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (nk > 0) {
      const uint32_t idesc_s = idesc_bf16_f32(QT, n_pad);
      const uint32_t idesc_o = idesc_bf16_f32(QT, HD, false, true);
      bool ok = true;
      // S(u): needs its item landed (waited once, at the first tile) and the
      // group's previous O read out (S overwrites the O columns)
      auto issue_s = [&](int u) -> bool {
        const int k = tiles == 2 ? u >> 1 : u, t = tiles == 2 ? u & 1 : 0, g = u & 1, slot = k % ns;
        if (t == 0 && !mbar_wait_warp(&full[slot], (k / ns) & 1)) return false;
        if (!mbar_wait_warp(&o_empty[g], ((u >> 1) & 1) ^ 1)) return false;
        tc_fence_after();
        const uint64_t dq = sdesc_sw128(smem_addr(qbuf + (2 * t + (k & 1)) * Q_BYTES), 16, 1024);
        const uint64_t dk = sdesc_sw128(smem_addr(kvbuf + slot * slot_bytes), 16, 1024);
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk) tc_mma_warp(tmem + g * 256, dq + 2 * kk, dk + 2 * kk, idesc_s, kk != 0);
        tc_commit_warp(&s_full[g]);
        if (t == tiles - 1) tc_commit_warp(&q_empty[k & 1]);
        return true;
      };
      // PV(u): needs P(u) in TMEM
      auto issue_pv = [&](int u) -> bool {
        const int k = tiles == 2 ? u >> 1 : u, t = tiles == 2 ? u & 1 : 0, g = u & 1;
        if (!mbar_wait_warp(&p_full[g], (u >> 1) & 1)) return false;
        tc_fence_after();
        const uint64_t dv = sdesc_sw128(smem_addr(kvbuf + (k % ns) * slot_bytes + slot_bytes / 2), 16384, 1024);
        for (int s = 0; s < n_pad / 16; ++s)  // 16 keys are 16 rows of 128 bytes
          tc_mma_tmem_a_warp(tmem + g * 256 + O_COL, tmem + g * 256 + 8 * s, dv + 128 * s, idesc_o, s != 0);
        tc_commit_warp(&o_full[g]);
        if (t == tiles - 1) tc_commit_warp(&kv_empty[k % ns]);
        return true;
      };
      ok = issue_s(0);
      const bool issued = ok;
      for (int u = 0; u < units && ok; ++u) {
        if (u + 1 < units) ok = issue_s(u + 1);
        if (ok) ok = issue_pv(u);
      }
      if (!ok && lane == 0) record_status(status, ELASTO_ERR_TIMEOUT);
      if (issued) {  // every MMA this thread issued has finished once `drain` completes
        tc_commit_warp(drain);
        mbar_wait_warp(drain, 0);
      }
    }
  } else {
    // ------------------------------------------------------------ softmax + epilogue
    const int g = (warp - 2) >> 2;           // group: units g, g + 2, ...
    const int qq = warp & 3;                 // TMEM lane quarter: rows 32 qq .. 32 qq + 31 of the tile
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(qq * 32) << 16) + g * 256;
    uint8_t* const stage = obuf + (warp - 2) * O_BYTES;
    {
      for (int u = g; u < units; u += 2) {
        const int k = tiles == 2 ? u >> 1 : u;
        const int item = items - 1 - (blockIdx.x + k * gridDim.x);
        const int t = tiles == 2 ? u & 1 : split ? item & 1 : 0;
        const uint32_t ph = (u >> 1) & 1;
        // a warp whose 32 rows are all past n has no softmax or read-out work
        const bool active = t * QT + qq * 32 < n;
        if (!__all_sync(0xffffffffu, mbar_wait(&s_full[g], ph))) {
          if (lane == 0) record_status(status, ELASTO_ERR_TIMEOUT);
          break;
        }
        tc_fence_after();
        float sum = 1.0f;
        if (active) {
          switch (n >> 6) {  // whole 64-key chunks
            case 0: sum = softmax_row<0>(lane_base, n); break;
            case 1: sum = softmax_row<1>(lane_base, n); break;
            case 2: sum = softmax_row<2>(lane_base, n); break;
            case 3: sum = softmax_row<3>(lane_base, n); break;
            default: sum = softmax_row<4>(lane_base, n); break;
          }
          tmem_st_wait();
        }
        tc_fence_before();
        mbar_arrive(&p_full[g]);
        // epilogue
        if (!__all_sync(0xffffffffu, mbar_wait(&o_full[g], ph))) {
          if (lane == 0) record_status(status, ELASTO_ERR_TIMEOUT);
          break;
        }
        tc_fence_after();
        uint32_t o[2][32];
        if (active) {
          load64(lane_base + O_COL, o);
          tmem_ld_wait();
        }
        tc_fence_before();
        mbar_arrive(&o_empty[g]);
        if (active) {
          const float inv = 1.0f / sum;
          const float2 inv2 = make_float2(inv, inv);
          if (elect_one()) bulk_wait_read<0>();  // the staging's previous store has read it
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            uint32_t pk[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int c = 8 * (j & 3) + 2 * i;
              const float2 x = mul2(make_float2(__uint_as_float(o[j >> 2][c]), __uint_as_float(o[j >> 2][c + 1])), inv2);
              pk[i] = pack_bf16x2(x.x, x.y);
            }
            *reinterpret_cast<uint4*>(stage + lane * 128 + ((j ^ (lane & 7)) << 4)) =
                make_uint4(pk[0], pk[1], pk[2], pk[3]);
          }
          fence_async_smem();
          __syncwarp();
          if (elect_one()) {
            const int bh = split ? item >> 1 : item, b = bh / heads;
            tma_store_3d(&tmO, stage, (bh - b * heads) * HD, t * QT + qq * 32, b);
            bulk_commit();
          }
        }
      }
      if (elect_one()) bulk_wait_all();
    }
  }
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

}  // namespace

cudaError_t attn_init_attributes() {
  return cudaFuncSetAttribute(attn_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem_bytes());
}

elasto_status attn_plan(AttnPlan* p, const bf16* qkv, bf16* out, int batch_cap, int n, int heads, int* status,
                        bool interleaved) {
  if (!p || !qkv || !out || batch_cap <= 0 || n <= 0 || heads <= 0) {
    set_error("attention: invalid arguments");
    return ELASTO_ERR_INVALID_ARG;
  }
  if (n > MAXK) {
    set_error("attention: at most 256 tokens are supported");
    return ELASTO_ERR_UNSUPPORTED;
  }
  *p = AttnPlan{};
  p->qkv = qkv;
  p->out = out;
  p->n = n;
  p->n_pad = (n + 15) / 16 * 16;
  p->heads = heads;
  p->blk_stride = interleaved ? HD : heads * HD;
  p->head_stride = interleaved ? 3 * HD : HD;
  p->batch_cap = batch_cap;
  p->status = status;
  const uint64_t cols = static_cast<uint64_t>(3) * heads * HD;
  const uint64_t ocols = static_cast<uint64_t>(heads) * HD;
  if (!encode_tmap_3d(&p->tmQ, qkv, cols, n, batch_cap, cols * 2, cols * 2 * n, HD, QT, 1) ||
      !encode_tmap_3d(&p->tmO, out, ocols, n, batch_cap, ocols * 2, ocols * 2 * n, HD, 32, 1) ||
      !encode_tmap_3d(&p->tmKV, qkv, cols, n, batch_cap, cols * 2, cols * 2 * n, HD, p->n_pad, 1)) {
    set_error("attention: cuTensorMapEncodeTiled failed");
    return ELASTO_ERR_UNSUPPORTED;
  }
  p->valid = true;
  return ELASTO_OK;
}

cudaError_t attn_launch(const AttnPlan& p, int batch, cudaStream_t s) {
  if (batch <= 0) return cudaSuccess;
  // where the chip would be half empty, a CTA takes one query tile instead of
  // both (K and V are then loaded twice)
  const int split = p.n > QT && 2 * batch * p.heads <= num_sms() ? 1 : 0;
  const int items = batch * p.heads * (1 + split);
  const int grid = items < num_sms() ? items : num_sms();
  return launch_pdl(attn_tc_kernel, dim3(grid), dim3(THREADS), smem_bytes_for(p.n_pad), s, p.tmQ, p.tmKV, p.tmO, p.n,
                    p.n_pad, p.heads, items, split, p.blk_stride, p.head_stride, p.status);
}

}  // namespace elasto
