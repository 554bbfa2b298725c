// Tensor-core GEMM with fused epilogues: out = epi(A[M,K] . W[N,K]^T).
//
// This is every dense contraction of the DN forward (Section 4.1): the patch
// projection, the sliced QKV projection of the kept heads (Eq. 2, 4), the
// sliced output projection W^O (Eq. 2, 4) and the sliced MLP W1 / W2
// (Eq. 5, 6). Slicing happened at create time, so here the kept widths are
// just the problem's N or K.
//
// Design (sm_103a):
//  - persistent grid, one CTA per SM (or one CTA pair per two SMs), static
//    round-robin over 128 x bn tiles (N tile index fastest so the CTAs
//    running together share A rows in L2; m_reverse runs the rows backwards);
//  - warp 0, one elected thread: TMA producer, ring of 128x64 (A) and bn x 64
//    (B) bf16 or f16 tiles with the 128-byte swizzle, one mbarrier pair per
//    stage. W may instead be loaded once per CTA and kept (b_resident: one N
//    tile);
//  - warp 1, as a whole: issues tcgen05.mma (M=128, N=bn, K=16) into one of two
//    TMEM accumulators (2 x 256 fp32 columns), commits stages back to the
//    producer and finished accumulators to the epilogue.
//  - CTA pairs (cta_group::2, M = 256, each CTA holds half of B) where
//    tile_cost() puts them ahead, at every K. What bounds a single 128 x 256
//    tile is shared memory: per k-block the MMAs read 48 KB and TMA writes
//    48 KB, 0.38 us at 128 B a clock, more than the 0.27 us the MMAs take, and
//    the epilogue's staging comes on top. A pair's CTA reads 32 KB and writes
//    32 KB. 400 calls back to back, the clock under the power cap: ViT-B QKV at
//    batch 256 (50432 x 2304 x 768) 137 us single, 114 us pairs (a library bf16
//    GEMM 101); FC1 + GELU 194 -> 170 us; 50432 x 3072 x 768 without GELU 188 ->
//    165 us (library 156).
//  - warps 2-13: epilogue, three warps per 32-lane quarter of TMEM (= 32 rows
//    of the tile). A warp works alone: it takes every third 128-byte-wide
//    chunk of its rows from TMEM to registers, writes it to its own 4 KB
//    staging piece (128B-swizzled, bank conflict free) and stores it with its
//    own TMA box. 16 warps on quarter chunks behind a 512-thread barrier per
//    chunk needed 4.9 us a tile, longer than a pair's main loop (3.7 us), most
//    of it in the barrier and in bias loads from the loaded L2 path; eight
//    warps on their own lack the overlap for GELU (FC1 174 us), sixteen the
//    registers. GELU, bias and residual use packed fp32 pairs.
//    * the fp32 residual stream (out-proj, FC2) leaves by TMA reduce-add, from
//      eight warps: X is not read into the SM. FC2 (K = 3072, 50432 rows) 154 ->
//      142 us, K = 1536 92 -> 85. Where memory sets the pace (K <= 700), and in a
//      plan of few tiles, the old rows are read into the staging pieces ahead
//      instead (K = 192 64.5 -> 54.7), as the 16-bit residual + ReLU of the CNN
//      block outputs are.
//    * a split-K plan (k-block range tile / (mt * nt)) stores fp32 partial sums
//      the same way; the transposing epilogue took its CTAs 2.5 us of a 4.9 us
//      one-image launch.
//    * the remaining epilogue (fp32 out, any row stride) transposes through
//      padded shared memory for row-contiguous stores.
//  - implicit-GEMM convolution: A tiles are 4-D TMA boxes of the NHWC input
//    (one tap and channel group per k-block, padding read as zeros), and the
//    output is stored by 4-D boxes of the tile's pixel block.
//  Every mbarrier wait is bounded; a timeout records ELASTO_ERR_TIMEOUT.
//  The two sides of a figure were taken in turn on one GPU. Figures of different
//  steps are from different GPUs and run lengths, between which the power cap
//  moves the clock, and the times of the large GEMMs by up to 12 %.
#include <algorithm>
#include <atomic>

#include "act.cuh"
#include "common.h"
#include "ptx.cuh"

namespace elasto {

namespace {

constexpr int BM = 128, BK = 64, MAX_STAGES = 8, MAX_BN = 256;
// Epilogue warps: three per TMEM lane quarter; two where the residual is added
// by the store, whose arithmetic is light (the staging saved is an operand
// stage: 50432 x 768 x 1536 91.7 -> 85.5 us, K = 3072 147 -> 142); one for the
// transposing fp32 epilogue.
constexpr int MAX_EPI_WARPS = 12;
constexpr int epi_warps(int epi) {
  return epi == EPI_BIAS_F32 ? 4 : epi == EPI_BIAS_ADD_F32 || epi == EPI_PART_F32 ? 8 : MAX_EPI_WARPS;
}
constexpr int epi_threads(int epi) { return 64 + 32 * epi_warps(epi); }
constexpr int THREADS_CONV = 64 + 32 * MAX_EPI_WARPS + 32;  // implicit convolutions: warp 14 is a second TMA producer
constexpr int A_STAGE = BM * BK * 2;        // 16 KB
constexpr int WBUF = 32 * 128;              // 4 KB staging piece of one epilogue warp (32 rows x 128 B)
constexpr int CBUF = MAX_EPI_WARPS * WBUF;  // 48 KB: one staging piece for each of twelve epilogue warps
constexpr int POOL = 224 * 1024;            // operand ring + staging pieces
constexpr int MAX_CBUFS = 3;                // staging pieces per epilogue warp
constexpr int EPI_LD = 33;                  // padded row of the transpose tile
constexpr int EPI_TILE = 32 * EPI_LD;       // floats per epilogue warp
constexpr int TMEM_COLS = 512;
constexpr size_t SMEM_BYTES = 1024 + POOL + 2048;
constexpr int BARS = 2 * MAX_STAGES + 6 + MAX_EPI_WARPS * MAX_CBUFS;  // mbarriers (the bias after them is read as float4)
static_assert(BARS * 8 % 16 == 0 && BARS * 8 + 32 * MAX_EPI_WARPS * 4 + 4 * (1 + MAX_EPI_WARPS / 4) <= 2048, "barriers and bias");

template <int EPI>
struct EpiTraits {
  static constexpr bool half = EPI == EPI_BIAS_RELU_F16 || EPI == EPI_BIAS_F16 || EPI == EPI_BIAS_RESID_RELU_F16;
  // 16-bit residual + ReLU (block outputs of the CNN): the residual chunk is
  // brought into the staging buffer by TMA like the fp32 residual stream
  static constexpr bool resid16 = EPI == EPI_BIAS_RESID_RELU_BF16 || EPI == EPI_BIAS_RESID_RELU_F16;
  static constexpr bool tma = EPI == EPI_BIAS_BF16 || EPI == EPI_BIAS_GELU_BF16 || EPI == EPI_BIAS_RELU_BF16 ||
                              EPI == EPI_BIAS_RESID_F32 || EPI == EPI_BIAS_ADD_F32 || EPI == EPI_PART_F32 ||
                              EPI == EPI_BIAS_RELU_F16 || EPI == EPI_BIAS_F16 || resid16;
  static constexpr bool f32 = EPI == EPI_BIAS_RESID_F32 || EPI == EPI_BIAS_ADD_F32 || EPI == EPI_PART_F32;
  // the old value is read into the staging piece by TMA; EPI_BIAS_ADD_F32
  // reads nothing: the store itself adds to memory
  static constexpr bool resid = EPI == EPI_BIAS_RESID_F32 || resid16;
  static constexpr int cw = f32 ? 32 : 64;  // columns per 128-byte staging chunk
};

// M-tile of the q-th tile row in the schedule: q, or mt - 1 - q when the plan
// runs its rows last to first (m_reverse: the GEMM then reads first the rows
// of its A operand that the previous kernel wrote last, still in L2).
__device__ __forceinline__ int m_tile(const GemmArgs& a, int q, int mt) { return a.m_reverse ? mt - 1 - q : q; }

// Row of the residual source that a tile starting at output row m0 reads: the
// same row, or for a periodic source (resid_row_mod rows per period, stored
// for enough periods that any 128 consecutive rows from a start below the
// period are present) the row m0 mod period.
__device__ __forceinline__ int resid_row(const GemmArgs& a, int m0) {
  return a.resid_row_mod > 0 ? m0 % a.resid_row_mod : m0;
}

template <int EPI>
__device__ __forceinline__ float2 epi_act2(float2 v) {
  if constexpr (EPI == EPI_BIAS_GELU_BF16) return gelu2(v);
  if constexpr (EPI == EPI_BIAS_RELU_BF16 || EPI == EPI_BIAS_RELU_F16 || EpiTraits<EPI>::resid16)
    return make_float2(fmaxf(v.x, 0.0f), fmaxf(v.y, 0.0f));
  return v;
}

// One 32-bit word of the epilogue's 16-bit type -> two fp32 values.
template <int EPI>
__device__ __forceinline__ float2 unpack_in(uint32_t w) {
  if constexpr (EpiTraits<EPI>::half)
    return __half22float2(*reinterpret_cast<const __half2*>(&w));
  else
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// Two fp32 values -> one 32-bit word of the epilogue's 16-bit output type.
template <int EPI>
__device__ __forceinline__ uint32_t pack_out(float lo, float hi) {
  if constexpr (EpiTraits<EPI>::half)
    return pack_f16x2(lo, hi);
  else
    return pack_bf16x2(lo, hi);
}

// Implicit-GEMM convolution: number of M tiles and the pixel block of one.
__host__ __device__ __forceinline__ int conv_mtiles(const GemmArgs& a) {
  return ((a.cv_wo + a.cv_bw - 1) / a.cv_bw) * ((a.cv_ho + a.cv_bh - 1) / a.cv_bh) *
         ((a.cv_batch + a.cv_nb - 1) / a.cv_nb);
}
__device__ __forceinline__ void conv_tile(const GemmArgs& a, int mtile, int& b0, int& oy0, int& ox0) {
  const int tx = (a.cv_wo + a.cv_bw - 1) / a.cv_bw, ty = (a.cv_ho + a.cv_bh - 1) / a.cv_bh;
  const int r = mtile / tx;
  ox0 = (mtile - r * tx) * a.cv_bw;
  oy0 = (r % ty) * a.cv_bh;
  b0 = (r / ty) * a.cv_nb;
}

// Walks the chunks of one epilogue warp group over this CTA's tiles. The
// chunks of all tiles form one sequence (cols(t) of them in tile t); group g
// takes every GROUPS-th one, so that tiles of a single chunk go round.
template <int GROUPS>
__device__ __forceinline__ int first_chunk(int g, int before) {
  return (g + GROUPS - before) % GROUPS;
}
template <int GROUPS>
struct ChunkIter {
  int t, c, before;  // tile, chunk in it, number of chunks before the tile (mod GROUPS)
  bool valid;
  template <class Cols>
  __device__ __forceinline__ void settle(int tiles, int stride, int g, Cols&& cols) {
    while (valid && c >= cols(t)) {
      before = (before + cols(t)) % GROUPS;
      t += stride;
      c = first_chunk<GROUPS>(g, before);
      valid = t < tiles;
    }
  }
  template <class Cols>
  __device__ __forceinline__ void init(int tiles, int start, int stride, int g, Cols&& cols) {
    t = start;
    before = 0;
    c = g;
    valid = t < tiles;
    settle(tiles, stride, g, cols);
  }
  template <class Cols>
  __device__ __forceinline__ void advance(int tiles, int stride, int g, Cols&& cols) {
    c += GROUPS;
    settle(tiles, stride, g, cols);
  }
};

// PAIR: the kernel runs as clusters of two CTAs on neighbouring SMs that
// share 256-row tiles: each CTA loads its 128 rows of A and half of the B
// tile; the even CTA issues tcgen05.mma.cta_group::2 (M = 256) for both and
// signals both CTAs' barriers with multicast commits; each CTA's epilogue
// reads its own half of the accumulator from its own TMEM.
template <int EPI, int NB, bool PAIR>
__global__ void __launch_bounds__(epi_threads(EPI) + 32, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmB2,
                   const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmR,
                   const GemmArgs args) {
  using TR = EpiTraits<EPI>;
  constexpr int EPI_WARPS = epi_warps(EPI), GROUPS = EPI_WARPS / 4;  // a group is one warp of every quarter: 128 rows
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int S = args.stages, E = args.cbufs;
  // NB: 1, or 2 when W is held as a bf16 (hi, lo) pair
  const int BSTG = args.b_stage;  // NB planes of bn rows (bn / 2 rows per CTA of a pair)
  const bool bres = !PAIR && NB == 1 && args.b_resident;
  uint8_t* sA = smem;
  uint8_t* sB = smem + S * A_STAGE;  // the B ring, or (bres) every k-block of B
  const int bke = args.k16 ? 16 : BK;  // K values per k-block
  const int nk = (args.K + bke - 1) / bke;
  uint8_t* sC = sB + (bres ? nk : S) * BSTG;  // E staging chunks, or the transpose tiles
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + POOL);
  uint64_t* full = bars;
  uint64_t* empty = bars + MAX_STAGES;
  uint64_t* tfull = bars + 2 * MAX_STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint64_t* bfull = drain + 1;  // resident B landed
  uint64_t* rfull = bfull + 1;  // residual landed: one per staging piece
  float* sbias = reinterpret_cast<float*>(bars + BARS);  // 32 values per epilogue warp
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sbias + 32 * EPI_WARPS);

  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int M = args.M, N = args.N, bn = args.bn;
  constexpr int TM = PAIR ? 2 * BM : BM;  // rows per tile
  // (a pair takes two consecutive pixel blocks of a convolution)
  const int mt = args.conv ? (conv_mtiles(args) + PAIR) / (1 + PAIR) : (M + TM - 1) / TM, nt = (N + bn - 1) / bn;
  // split-K (fp32 partial outputs only): tile t covers output tile
  // t % (mt * nt) and k-block range t / (mt * nt) of ks. Every other
  // epilogue has ks = 1 at compile time and no division on its tile path.
  constexpr bool kSplit = EPI == EPI_PART_F32;
  const int ks = kSplit && args.ksplit > 1 ? args.ksplit : 1;
  const int mn_tiles = mt * nt;
  const int tiles = mn_tiles * ks;
  const int rank = PAIR ? warp_uniform(static_cast<int>(cluster_ctarank())) : 0;  // this CTA's row half of a pair tile
  const int t_start = PAIR ? warp_uniform(static_cast<int>(cluster_id_x())) : static_cast<int>(blockIdx.x);
  const int t_stride = PAIR ? warp_uniform(static_cast<int>(cluster_count_x())) : static_cast<int>(gridDim.x);
  const bool leader = rank == 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], (PAIR ? 2 : 1) * EPI_WARPS);
    }
    mbar_init(drain, 1);
    if constexpr (TR::resid)
      for (int e = 0; e < EPI_WARPS * MAX_CBUFS; ++e) mbar_init(&rfull[e], 1);
    mbar_init(bfull, 1);
    for (int i = 0; i < GROUPS; ++i) tmem_slot[1 + i] = 0;  // the convolution epilogue groups' fail flags
    fence_barrier_init();
  }
  if (warp == 0) {
    if constexpr (PAIR) {
      tmem_alloc_pair(tmem_slot, TMEM_COLS);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, TMEM_COLS);
      tmem_relinquish();
    }
  }
  if (warp == 1 && elect_one()) {
    if (nk > 0) {
      tma_prefetch_desc(&tmA);
      tma_prefetch_desc(&tmB);
      if constexpr (NB == 2) tma_prefetch_desc(&tmB2);
    }
    if constexpr (TR::tma) tma_prefetch_desc(&tmC);
    if constexpr (TR::resid) tma_prefetch_desc(&tmR);
  }
  tc_fence_before();
  if constexpr (PAIR)
    cluster_sync_all();  // both CTAs' barriers initialised before any remote arrive
  else
    __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(static_cast<int>(*tmem_slot));
  // Everything above overlapped the previous kernel's tail. Every thread
  // waits for that kernel (pdl_wait) before its first access to data it may
  // write; a model's weights are not such data (w_const), so the producer
  // thread starts loading them first and waits after that.
  if (warp != 0 || nk == 0) {
    pdl_wait();
    pdl_trigger();
  }

  // Implicit convolutions run two producer threads (one of warp 0 and one of
  // warp 14) that take alternate k-blocks: with one, the 4-D boxes pace narrow
  // tiles (128 images of 56 x 56 x 16 -> 16 channels: 54 us with one, 48 us
  // with two; the strided 128-channel 3x3 of stage 2: 37.4 and 35.6).
  const int nprod = (args.conv && static_cast<int>(blockDim.x) == THREADS_CONV) ? 2 : 1;
  if (warp == 0 || warp == 2 + EPI_WARPS) {
    // ------------------------------------------------------------ producer
    const int pid = warp == 0 ? 0 : 1;
    if (pid < nprod && nk > 0 && elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      long seq = 0;         // k-block sequence index over this CTA's tiles
      long last_mine = -1;  // the last k-block this thread issued
      bool ok = true;
      // pair: the even CTA's full barrier counts both CTAs' bytes
      const uint32_t a_bytes = args.conv ? args.cv_a_bytes : A_STAGE;
      const uint32_t bytes = PAIR ? 2 * (a_bytes + (bn / 2) * BK * 2) : a_bytes + (bres ? 0 : NB * bn * bke * 2);
      const bool b_loaded = bres && t_start < tiles && pid == 0;
      if (!args.w_const) pdl_wait();
      if (b_loaded) {  // all of W, once: nk k-blocks of the single N tile
        mbar_expect_tx(bfull, static_cast<uint32_t>(nk) * bn * bke * 2);
        for (int kb = 0; kb < nk; ++kb) tma_load_2d(sB + kb * BSTG, &tmB, bfull, kb * bke, 0);
      }
      // the first tile's first S stages: armed and their weights requested
      // before the wait (fresh stages: no empty-slot wait needed); the first
      // producer issues these k-blocks
      int pre = 0;
      if (!PAIR && !bres && t_start < tiles) {
        const int tq = kSplit ? t_start % mn_tiles : t_start;
        const int kb0 = kSplit ? (t_start / mn_tiles) * nk / ks : 0;
        const int kb1 = kSplit ? (t_start / mn_tiles + 1) * nk / ks : nk;
        const int n0 = (tq % nt) * bn;
        pre = kb1 - kb0 < S ? kb1 - kb0 : S;
        if (pid == 0)
          for (int i = 0; i < pre; ++i) {
            mbar_expect_tx(&full[i], bytes);
            tma_load_2d(sB + i * BSTG, &tmB, &full[i], (kb0 + i) * bke, n0);
            if constexpr (NB == 2) tma_load_2d(sB + i * BSTG + BSTG / 2, &tmB2, &full[i], (kb0 + i) * BK, n0);
          }
      }
      auto mine = [&](long q) { return nprod == 1 || (q < pre ? pid == 0 : static_cast<int>(q & 1) == pid); };
      pdl_wait();
      pdl_trigger();
      for (int t = t_start; t < tiles && ok; t += t_stride) {
        const int tq = kSplit ? t % mn_tiles : t;
        const int kb0 = kSplit ? (t / mn_tiles) * nk / ks : 0, kb1 = kSplit ? (t / mn_tiles + 1) * nk / ks : nk;
        const int m0 = m_tile(args, tq / nt, mt) * TM + rank * BM, n0 = (tq % nt) * bn;
        int cb0 = 0, cy0 = 0, cx0 = 0;  // implicit conv: first image, output row and column of the tile
        int cg = 0, kx = 0, ky = 0;     // implicit conv: the k-block's channel group and tap, advanced in step
        if (args.conv) {
          conv_tile(args, m_tile(args, tq / nt, mt) * (1 + PAIR) + rank, cb0, cy0, cx0);
          const int tap = kb0 / args.cv_cgroups;
          cg = kb0 - tap * args.cv_cgroups;
          ky = tap / args.cv_ks;
          kx = tap - ky * args.cv_ks;
        }
        for (int kb = kb0; kb < kb1; ++kb, ++seq) {
          if (mine(seq)) {
            if (!mbar_wait(&empty[stage], phase ^ 1)) {
              ok = false;
              break;
            }
            if constexpr (PAIR) {
              const uint32_t full_lead = cluster_map(smem_addr(&full[stage]), 0);
              if (leader) mbar_expect_tx(&full[stage], bytes);
              if (args.conv)
                tma_load_4d_pair(sA + stage * A_STAGE, &tmA, full_lead, cg * BK,
                                 cx0 * args.cv_stride - args.cv_pad + kx, cy0 * args.cv_stride - args.cv_pad + ky, cb0);
              else
                tma_load_2d_pair(sA + stage * A_STAGE, &tmA, full_lead, kb * BK, m0);
              tma_load_2d_pair(sB + stage * BSTG, &tmB, full_lead, kb * BK, n0 + rank * (bn / 2));
            } else {
              const bool armed = seq < pre;  // this stage's weights were requested before the wait
              if (!armed) mbar_expect_tx(&full[stage], bytes);
              if (args.conv) {
                tma_load_4d(sA + stage * A_STAGE, &tmA, &full[stage], cg * bke,
                            cx0 * args.cv_stride - args.cv_pad + kx, cy0 * args.cv_stride - args.cv_pad + ky, cb0);
              } else {
                tma_load_2d(sA + stage * A_STAGE, &tmA, &full[stage], kb * BK, m0);
              }
              if (!bres && !armed) tma_load_2d(sB + stage * BSTG, &tmB, &full[stage], kb * bke, n0);
              if constexpr (NB == 2)
                if (!armed) tma_load_2d(sB + stage * BSTG + BSTG / 2, &tmB2, &full[stage], kb * BK, n0);
            }
            last_mine = seq;
          }
          if (++stage == S) {
            stage = 0;
            phase ^= 1;
          }
          if (++cg == args.cv_cgroups) {  // (meaningful for convolutions only)
            cg = 0;
            if (++kx == args.cv_ks) {
              kx = 0;
              ++ky;
            }
          }
        }
      }
      if (!ok) record_status(args.status, ELASTO_ERR_TIMEOUT);
      // Drain: no copy this thread issued may still be landing in shared
      // memory when the CTA exits (returns at once on the normal path): the
      // stages of the sequence's last S k-blocks (no later k-block reuses
      // them) that this thread issued. In a pair only the even CTA's
      // barriers see the copies; the cluster barrier before exit orders the
      // odd CTA behind this drain.
      for (long q = seq - 1; leader && q >= 0 && q > seq - 1 - S; --q) {
        if (!mine(q) || q > last_mine) continue;
        const int st = static_cast<int>(q % S);
        const uint32_t ph = static_cast<uint32_t>((q / S) & 1);
        mbar_wait(&full[st], ph);
      }
      if (b_loaded) mbar_wait(bfull, 0);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (leader) {
      const uint32_t idesc = idesc_16_f32(TM, bn, args.f16 != 0);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true, issued = false;
      // resident B: every tile's MMAs read it; wait for it once
      if (bres && t_start < tiles && !mbar_wait_warp(bfull, 0)) ok = false;
      int local = 0;
      for (int t = t_start; t < tiles && ok; t += t_stride, ++local) {
        const int acc = local & 1;
        const uint32_t use = static_cast<uint32_t>(local >> 1);
        if (!mbar_wait_warp(&tempty[acc], (use & 1) ^ 1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t dtm = tmem_base + acc * MAX_BN;
        if (nk == 0) {
          if (lane == 0) {
            mbar_arrive(&tfull[acc]);
            if constexpr (PAIR) mbar_arrive_cluster(cluster_map(smem_addr(&tfull[acc]), 1));
          }
          continue;
        }
        const int kb0 = kSplit ? (t / mn_tiles) * nk / ks : 0, kb1 = kSplit ? (t / mn_tiles + 1) * nk / ks : nk;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait_warp(&full[stage], phase)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a0 = smem_addr(sA + stage * A_STAGE), b0 = smem_addr(sB + (bres ? kb : stage) * BSTG);
          if (args.k16) {
            // one K=16 step per k-block: rows of 32 bytes in the 32-byte swizzle,
            // 8-row groups 256 bytes apart
            if constexpr (!PAIR && NB == 1)
              tc_mma_warp(dtm, sdesc_sw32(a0, 16, 256), sdesc_sw32(b0, 16, 256), idesc, kb != kb0);
          } else {
            // the stage's descriptors once; a K = 16 step is +32 bytes = +2 in
            // the start-address field (the tiles are 1024-byte aligned, so it
            // never carries out of the field)
            const uint64_t da = sdesc_sw128(a0, 16, 1024), db = sdesc_sw128(b0, 16, 1024);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) {
              if constexpr (PAIR) {
                tc_mma_pair_warp(dtm, da + 2 * k, db + 2 * k, idesc, kb != kb0 || k != 0);
              } else {
                tc_mma_warp(dtm, da + 2 * k, db + 2 * k, idesc, kb != kb0 || k != 0);
                if constexpr (NB == 2)  // low half of the weights: acc += A . W_lo^T
                  tc_mma_warp(dtm, da + 2 * k, sdesc_sw128(b0 + BSTG / 2, 16, 1024) + 2 * k, idesc, 1u);
              }
            }
          }
          issued = true;
          if constexpr (PAIR)
            tc_commit_pair_multicast_warp(&empty[stage], 0x3);
          else
            tc_commit_warp(&empty[stage]);
          if (++stage == S) {
            stage = 0;
            phase ^= 1;
          }
        }
        if (ok) {
          if constexpr (PAIR)
            tc_commit_pair_multicast_warp(&tfull[acc], 0x3);
          else
            tc_commit_warp(&tfull[acc]);
        }
      }
      if (!ok && lane == 0) record_status(args.status, ELASTO_ERR_TIMEOUT);
      // All MMAs this thread issued have finished once `drain` completes.
      if (issued) {
        if constexpr (PAIR) {
          if (elect_one()) tc_commit_pair(drain);
        } else {
          tc_commit_warp(drain);
        }
        mbar_wait_warp(drain, 0);
      }
    }
  } else if constexpr (TR::tma) {
    // ------------------------------------------------------------ TMA-store epilogue
    constexpr int CW = TR::cw;
    const int ew = warp - 2;
    const int q = warp & 3;       // TMEM lane quarter: rows 32q .. 32q + 31 of the tile
    const int g = ew >> 2;        // takes every third chunk
    const int cpt = bn / CW;
    const uint32_t row_tm = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
    auto piece = [&](int e) { return sC + ((g * E + e) * 4 + q) * WBUF; };  // a group's four pieces are one 16 KB chunk
    auto cols = [&](int t) {
      const int left = (N - (t % nt) * bn + CW - 1) / CW;  // (nt divides the tiles of a split)
      return left < cpt ? left : cpt;
    };
    auto row0 = [&](int t) { return m_tile(args, (kSplit ? t % mn_tiles : t) / nt, mt) * TM + rank * BM; };
    // Warps work on their own: each reads its 32 rows of its chunks, writes
    // them to its own staging pieces and stores them with its own 32-row TMA
    // boxes; the only hand-offs are the accumulator barriers. (Convolution
    // tiles are pixel blocks whose quarters are no boxes: the four warps of a
    // group meet at a named barrier and one stores the 128-row chunk.)
    // A convolution warp whose wait gave up tells its group, which leaves
    // together after its next barrier.
    volatile uint32_t* fail = tmem_slot + 1 + g;
    uint64_t* rf = rfull + ew * MAX_CBUFS;
    float* sb = sbias + 32 * ew;
    ChunkIter<GROUPS> pf{};  // residual prefetch (the elected thread)
    long loads = 0, consumed = 0;
    auto fetch = [&](int e) {
      mbar_expect_tx(&rf[e], WBUF);
      tma_load_2d(piece(e), &tmR, &rf[e], (pf.t % nt) * bn + pf.c * CW, resid_row(args, row0(pf.t)) + q * 32);
      pf.advance(tiles, t_stride, g, cols);
      ++loads;
    };
    if constexpr (TR::resid) {
      if (elect_one()) {
        pf.init(tiles, t_start, t_stride, g, cols);
        for (int e = 0; e < E && pf.valid; ++e) fetch(e);
      }
    }
    int e = 0, before = 0;
    uint32_t rph = 0;
    bool ok = true;
    int local = 0;
    for (int t = t_start; t < tiles && ok; t += t_stride, ++local) {
      const int acc = local & 1;
      const uint32_t use = static_cast<uint32_t>(local >> 1);
      const int m0 = row0(t), n0 = (t % nt) * bn, nvalid = cols(t);
      int c = first_chunk<GROUPS>(g, before);
      before = (before + nvalid) % GROUPS;
      // Each chunk's bias is requested a chunk ahead (before the accumulator
      // wait for the first), one column per lane, and broadcast from shared
      // memory: reading it where it is used, every thread every column, left
      // the warp waiting on the loaded L2 path for a third of the chunk.
      float nb[CW / 32];
      auto bias_of = [&](int chunk) {
#pragma unroll
        for (int h = 0; h < CW / 32; ++h) {
          const int k = n0 + chunk * CW + 32 * h + lane;
          nb[h] = args.bias && k < N ? __ldg(args.bias + k) : 0.0f;
        }
      };
      bias_of(c);
      ok = __all_sync(0xffffffffu, mbar_wait(&tfull[acc], use & 1));
      if (!ok) {
        if (!args.conv) break;
        *fail = 1;
        ok = true;
      }
      tc_fence_after();
      const uint32_t acc_tm = row_tm + acc * MAX_BN;
      auto release = [&] {  // this warp's last TMEM read of the tile is done
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if constexpr (PAIR)
            mbar_arrive_cluster(cluster_map(smem_addr(&tempty[acc]), 0));  // the even CTA issues the MMAs
          else
            mbar_arrive(&tempty[acc]);
        }
      };
      if (c >= nvalid) release();
      for (; c < nvalid; c += GROUPS) {
        uint8_t* const rowp = piece(e) + lane * 128;
        const int col = n0 + c * CW;
        uint32_t v[CW / 32][32];
        float bl[CW / 32];
        if (nk > 0) tmem_ld_32x32b_x32(acc_tm + c * CW, v[0]);
#pragma unroll
        for (int h = 0; h < CW / 32; ++h) bl[h] = nb[h];
        if (c + GROUPS < nvalid) bias_of(c + GROUPS);
        sb[lane] = bl[0];
        __syncwarp();
        if (nk > 0) {
          tmem_ld_wait();
          if constexpr (CW == 64) tmem_ld_32x32b_x32(acc_tm + c * CW + 32, v[1]);  // in flight while v[0] is worked on
        } else {
#pragma unroll
          for (int j = 0; j < CW; ++j) v[j / 32][j & 31] = 0u;
        }
        if (CW == 32 && c + GROUPS >= nvalid) release();
        if constexpr (TR::resid) {
          ok = __all_sync(0xffffffffu, mbar_wait(&rf[e], rph));
          if (!ok) break;
          ++consumed;
        } else {
          if (elect_one()) bulk_wait_read<0>();  // the one piece is free once its last store has read it
          if (args.conv)
            named_bar_sync(1 + g, 128);  // (one warp issues the group's stores)
          else
            __syncwarp();
        }
        // 16-byte pieces of the 128-byte staging row, swizzled as the TMA box is
        if constexpr (TR::f32) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float4* p = reinterpret_cast<float4*>(rowp + ((j ^ (lane & 7)) << 4));
            const float4 bb = reinterpret_cast<const float4*>(sb)[j];
            float2 lo = add2(make_float2(__uint_as_float(v[0][4 * j]), __uint_as_float(v[0][4 * j + 1])),
                             make_float2(bb.x, bb.y));
            float2 hi = add2(make_float2(__uint_as_float(v[0][4 * j + 2]), __uint_as_float(v[0][4 * j + 3])),
                             make_float2(bb.z, bb.w));
            if constexpr (TR::resid) {  // X_old arrived by TMA into the same place
              const float4 o = *p;
              lo = add2(make_float2(o.x, o.y), lo);
              hi = add2(make_float2(o.z, o.w), hi);
            }
            *p = make_float4(lo.x, lo.y, hi.x, hi.y);
          }
        } else {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (h == 1) {
              __syncwarp();
              sb[lane] = bl[1];
              __syncwarp();
              if (nk > 0) tmem_ld_wait();
              if (c + GROUPS >= nvalid) release();
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              uint4* p = reinterpret_cast<uint4*>(rowp + (((4 * h + j) ^ (lane & 7)) << 4));
              uint32_t rw[4] = {0u, 0u, 0u, 0u}, ow[4];
              if constexpr (TR::resid16) {  // the residual's 8 values arrived by TMA
                const uint4 rv = *p;
                rw[0] = rv.x, rw[1] = rv.y, rw[2] = rv.z, rw[3] = rv.w;
              }
              const float4 b4[2] = {reinterpret_cast<const float4*>(sb)[2 * j],
                                    reinterpret_cast<const float4*>(sb)[2 * j + 1]};
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const int k = 8 * j + 2 * i;
                const float2 bb = i & 1 ? make_float2(b4[i >> 1].z, b4[i >> 1].w)
                                        : make_float2(b4[i >> 1].x, b4[i >> 1].y);
                float2 x = add2(make_float2(__uint_as_float(v[h][k]), __uint_as_float(v[h][k + 1])), bb);
                if constexpr (TR::resid16) x = add2(x, unpack_in<EPI>(rw[i]));
                x = epi_act2<EPI>(x);
                ow[i] = pack_out<EPI>(x.x, x.y);
              }
              *p = make_uint4(ow[0], ow[1], ow[2], ow[3]);
            }
          }
        }
        fence_async_smem();  // (the barriers below also order this chunk's bias reads before the next one's write)
        if (args.conv) {
          named_bar_sync(1 + g, 128);
          if (*fail) {
            ok = false;
            break;
          }
          if (q == 0 && elect_one()) {  // (its piece is the chunk's first)
            int cb0, cy0, cx0;
            conv_tile(args, m_tile(args, t / nt, mt) * (1 + PAIR) + rank, cb0, cy0, cx0);
            if (cb0 < args.cv_batch) tma_store_4d(&tmC, piece(e), col, cx0, cy0, cb0);  // (a pair's last block may be none)
            bulk_commit();
          }
        } else {
          __syncwarp();
          if (elect_one()) {
            if constexpr (TR::resid)
              if (E > 1) bulk_wait_read<0>();  // the previous chunk's store: its piece is refilled below
            if (m0 + q * 32 < M) {
              if constexpr (EPI == EPI_BIAS_ADD_F32)
                tma_add_2d(&tmC, piece(e), col, m0 + q * 32);
              else if constexpr (kSplit)
                tma_store_3d(&tmC, piece(e), col, m0 + q * 32, t / mn_tiles);
              else
                tma_store_2d(&tmC, piece(e), col, m0 + q * 32);
            }
            bulk_commit();
            if constexpr (TR::resid) {
              if (E == 1) bulk_wait_read<0>();
              if ((E == 1 || consumed > 1) && pf.valid) fetch(e == 0 ? E - 1 : e - 1);
            }
          }
        }
        if (++e == E) {
          e = 0;
          rph ^= 1;
        }
      }
    }
    if (elect_one()) {
      if (!ok) record_status(args.status, ELASTO_ERR_TIMEOUT);
      bulk_wait_all();
      // Residual loads issued for chunks never consumed (only on the abort
      // path): let them land before the CTA releases its shared memory.
      if constexpr (TR::resid)
        for (long i = consumed; i < loads; ++i) {
          mbar_wait(&rf[e], rph);
          if (++e == E) {
            e = 0;
            rph ^= 1;
          }
        }
    }
  } else {
    // ------------------------------------------------------------ transpose epilogue
    {
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    float* st = reinterpret_cast<float*>(sC) + (warp - 2) * EPI_TILE;
    int local = 0;
    for (int t = t_start; t < tiles; t += t_stride, ++local) {
      const int acc = local & 1;
      const uint32_t use = static_cast<uint32_t>(local >> 1);
      if (!mbar_wait(&tfull[acc], use & 1)) {
        if (lane == 0) record_status(args.status, ELASTO_ERR_TIMEOUT);
        break;
      }
      tc_fence_after();
      const int m0 = m_tile(args, t / nt, mt) * TM + rank * BM, n0 = (t % nt) * bn;
      const int row0 = m0 + q * 32;
      for (int c = 0; c < bn; c += 32) {
        if (n0 + c >= N) break;
        uint32_t r[32];
        if (nk > 0) {
          tmem_ld_32x32b_x32(tmem_base + (static_cast<uint32_t>(q * 32) << 16) + acc * MAX_BN + c, r);
          tmem_ld_wait();
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) r[j] = 0u;
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) st[lane * EPI_LD + j] = __uint_as_float(r[j]);
        __syncwarp();
        {  // EPI_BIAS_F32
          const int col = n0 + c + lane;
          const bool cok = col < N;
          const float bv = (cok && args.bias) ? args.bias[col] : 0.0f;
          float* out = static_cast<float*>(args.out);
#pragma unroll 8
          for (int i = 0; i < 32; ++i) {
            const int row = row0 + i;
            if (cok && row < M) out[static_cast<size_t>(row) * args.ldo + col] = st[i * EPI_LD + lane] + bv;
          }
        }
        __syncwarp();
      }
      tc_fence_before();
      if (lane == 0) mbar_arrive(&tempty[acc]);
    }
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();  // the peer's TMEM and barriers are no longer in use
  if (warp == 0) {
    __syncwarp();
    tc_fence_after();
    if constexpr (PAIR)
      tmem_dealloc_pair(tmem_base, TMEM_COLS);
    else
      tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// Split-K residual: out[r, c] += (sum over splits of part[s][r, c]) + bias[c],
// the splits added in order, the sum and bias associated as in the one-pass
// RESID_F32 epilogue (x + (acc + b)). One thread per 4 columns of a row.
__global__ void splitk_reduce_kernel(const float* __restrict__ part, int ks, long long stride, int M, int N,
                                     const float* __restrict__ bias, float* __restrict__ out, int ldo) {
  pdl_wait();
  pdl_trigger();
  const int n4 = N / 4;
  const size_t total = static_cast<size_t>(M) * n4;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < total;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t r = i / n4;
    const int c = static_cast<int>(i - r * n4) * 4;
    float4 acc = *reinterpret_cast<const float4*>(part + r * N + c);
    for (int sp = 1; sp < ks; ++sp) {
      const float4 v = *reinterpret_cast<const float4*>(part + sp * stride + r * N + c);
      acc.x += v.x;
      acc.y += v.y;
      acc.z += v.z;
      acc.w += v.w;
    }
    const float4 b = bias ? *reinterpret_cast<const float4*>(bias + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4* o = reinterpret_cast<float4*>(out + r * ldo + c);
    float4 x = *o;
    x.x += acc.x + b.x;
    x.y += acc.y + b.y;
    x.z += acc.z + b.z;
    x.w += acc.w + b.w;
    *o = x;
  }
}

// Sum over the threads of a block of nw warps (nw <= 32); red: nw floats of
// shared memory. Every thread gets the total.
__device__ __forceinline__ float block_sum(float v, float* red, int nw) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  float t = lane < nw ? red[lane] : 0.0f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  __syncthreads();  // red is reused by the next call
  return t;
}

// The same sum, and then the LayerNorm of each finished row: one block of
// N / 2 threads per row, two channels per thread (all the row's partial sums
// in flight at once). Statistics as layernorm_kernel takes them (mean over
// the first d_true channels, centred sum of squares less the zero padding's
// pad * mean^2, eps 1e-6), summed in another order.
__global__ void __launch_bounds__(512) splitk_reduce_ln_kernel(const float* __restrict__ part, int ks,
                                                               long long stride, int N,
                                                               const float* __restrict__ bias,
                                                               float* __restrict__ out, const float* __restrict__ g,
                                                               const float* __restrict__ b, bf16* __restrict__ y,
                                                               float inv_d, float pad) {
  __shared__ float red[32];
  pdl_wait();
  pdl_trigger();
  const size_t e = static_cast<size_t>(blockIdx.x) * N + 2 * threadIdx.x;
  float2 p2[kSplitMax];
#pragma unroll
  for (int sp = 0; sp < kSplitMax; ++sp)
    p2[sp] = sp < ks ? *reinterpret_cast<const float2*>(part + sp * stride + e) : make_float2(0.f, 0.f);
  float2 acc = p2[0];
#pragma unroll
  for (int sp = 1; sp < kSplitMax; ++sp)
    if (sp < ks) {
      acc.x += p2[sp].x;
      acc.y += p2[sp].y;
    }
  const float2 bb = bias ? reinterpret_cast<const float2*>(bias)[threadIdx.x] : make_float2(0.f, 0.f);
  float2* o = reinterpret_cast<float2*>(out + e);
  float2 x = *o;
  x.x += acc.x + bb.x;
  x.y += acc.y + bb.y;
  *o = x;
  const int nw = blockDim.x >> 5;
  const float mean = block_sum(x.x + x.y, red, nw) * inv_d;
  const float a = x.x - mean, c = x.y - mean;
  const float rstd = rsqrtf((block_sum(a * a + c * c, red, nw) - pad * mean * mean) * inv_d + 1e-6f);
  const float2 gg = reinterpret_cast<const float2*>(g)[threadIdx.x];
  const float2 be = reinterpret_cast<const float2*>(b)[threadIdx.x];
  reinterpret_cast<uint32_t*>(y)[e / 2] = pack_bf16x2(a * rstd * gg.x + be.x, c * rstd * gg.y + be.y);
}

template <int EPI, int NB, bool PAIR>
cudaError_t launch_epi(const GemmPlan& p, int M, cudaStream_t s) {
  GemmArgs a = p.args;
  a.M = M;
  a.cv_batch = M;  // implicit convolutions: M counts images
  const int nt = (a.N + a.bn - 1) / a.bn;
  if constexpr (PAIR) {
    const int threads = a.conv ? THREADS_CONV : epi_threads(EPI);
    int pairs = 0;
    const cudaError_t e = max_cta_pairs(reinterpret_cast<const void*>(gemm_tc_kernel<EPI, NB, true>), threads,
                                        SMEM_BYTES, &pairs);
    if (e != cudaSuccess) return e;
    const int tiles = (a.conv ? (conv_mtiles(a) + 1) / 2 : (M + 2 * BM - 1) / (2 * BM)) * nt;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_pdl
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(2 * std::min(tiles, pairs));
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, gemm_tc_kernel<EPI, NB, true>, p.tmA, p.tmB, p.tmB2, p.tmC, p.tmR, a);
  } else {
    const int tiles = (a.conv ? conv_mtiles(a) : (M + BM - 1) / BM) * nt * (a.ksplit > 1 ? a.ksplit : 1);
    const int grid = tiles < num_sms() ? tiles : num_sms();
    return launch_pdl(gemm_tc_kernel<EPI, NB, false>, dim3(grid), dim3(a.conv ? THREADS_CONV : epi_threads(EPI)), SMEM_BYTES, s,
                      p.tmA, p.tmB, p.tmB2,
                      p.tmC, p.tmR, a);
  }
}

}  // namespace

cudaError_t max_cta_pairs(const void* kernel, int threads, size_t smem, int* pairs) {
  static std::atomic<int> known[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  *pairs = known[dev].load(std::memory_order_relaxed);
  if (*pairs > 0) return cudaSuccess;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(2 * (num_sms() / 2));
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaOccupancyMaxActiveClusters(pairs, kernel, &cfg);
  if (e != cudaSuccess) return e;
  if (*pairs <= 0) return cudaErrorInvalidConfiguration;
  known[dev].store(*pairs, std::memory_order_relaxed);
  return cudaSuccess;
}

cudaError_t gemm_init_attributes() {
  const int bytes = static_cast<int>(SMEM_BYTES);
  cudaError_t e;
#define SET_ATTR(E)                                                                                        \
  e = cudaFuncSetAttribute(gemm_tc_kernel<E, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);   \
  if (e != cudaSuccess) return e;                                                                          \
  e = cudaFuncSetAttribute(gemm_tc_kernel<E, 2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);   \
  if (e != cudaSuccess) return e;
#define SET_ATTR_PAIR(E)                                                                                   \
  e = cudaFuncSetAttribute(gemm_tc_kernel<E, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);    \
  if (e != cudaSuccess) return e;
  SET_ATTR(EPI_BIAS_BF16)
  SET_ATTR(EPI_BIAS_GELU_BF16)
  SET_ATTR(EPI_BIAS_RESID_F32)
  SET_ATTR(EPI_BIAS_ADD_F32)
  SET_ATTR(EPI_PART_F32)
  SET_ATTR(EPI_BIAS_F32)
  SET_ATTR(EPI_BIAS_RELU_BF16)
  SET_ATTR(EPI_BIAS_RESID_RELU_BF16)
  SET_ATTR(EPI_BIAS_RELU_F16)
  SET_ATTR(EPI_BIAS_F16)
  SET_ATTR(EPI_BIAS_RESID_RELU_F16)
  SET_ATTR_PAIR(EPI_BIAS_RELU_F16)
  SET_ATTR_PAIR(EPI_BIAS_F16)
  SET_ATTR_PAIR(EPI_BIAS_BF16)
  SET_ATTR_PAIR(EPI_BIAS_GELU_BF16)
  SET_ATTR_PAIR(EPI_BIAS_RESID_F32)
  SET_ATTR_PAIR(EPI_BIAS_ADD_F32)
  SET_ATTR_PAIR(EPI_BIAS_RELU_BF16)
#undef SET_ATTR
#undef SET_ATTR_PAIR
  return cudaSuccess;
}

namespace {

bool is_resid16(int epi) { return epi == EPI_BIAS_RESID_RELU_BF16 || epi == EPI_BIAS_RESID_RELU_F16; }

// Bytes of one ring stage (A tile and the CTA's part of the B tile).
int stage_bytes(int bn, bool pair, int planes) { return A_STAGE + (pair ? bn / 2 : planes * bn) * BK * 2; }

// A GEMM (or implicit convolution, M = 128 rows per pixel block) to choose a
// tiling for.
struct Problem {
  int M, N, K, planes, epi;
  bool conv;
  int sms;
};

// Estimated nanoseconds of one launch with 128-row (pair: 256-row) x bn tiles.
// A k-block costs its MMAs or the delivery of its operands to shared memory,
// whichever is longer; a tile its k-blocks or its epilogue, which overlap; the
// last tile's epilogue is exposed, and clusters take longer to start. The
// constants are fitted to launches of 197 to 50432 rows.
double tile_cost(const Problem& p, int bn, bool pair) {
  const int units = pair ? p.sms / 2 : p.sms, rows = pair ? 2 * BM : BM;
  const long tiles = static_cast<long>((p.M + rows - 1) / rows) * ((p.N + bn - 1) / bn);
  const long waves = (tiles + units - 1) / units;
  double load = stage_bytes(bn, pair, p.planes) / 126.0, mma = p.planes * (130.0 + 0.9 * bn);
  // 4-D boxes. Narrow tiles advance at 230 to 260 ns a k-block (128 images of 56 x
  // 56 x 64 in 64 columns 242); the margin decides for halo tiles up to 6 % too
  // early on calls of 10 us (17 images of 31 x 31 x 32 -> 80 channels: 10.5, 9.8)
  if (p.conv) load = std::max(load, 280.0);
  const double main_loop = ((p.K + BK - 1) / BK) * std::max(load, mma);
  const bool f32 = p.epi == EPI_BIAS_RESID_F32 || p.epi == EPI_BIAS_ADD_F32;
  double epilogue = 400.0 + bn * (f32 ? 8.0 : p.epi == EPI_BIAS_GELU_BF16 ? 9.0 : 6.0);
  if (is_resid16(p.epi)) {
    // a 16-bit residual is read ahead; past the L2 it moves at the memory's pace,
    // and later where one piece per warp is all that fits ahead (CNN block outputs,
    // 256 -> 128 columns: 100352 x 512 x 128 43.3 -> 41.4 us, 25088 x 1024 x 256
    // 28.2 -> 25.6, 100352 x 256 x 64 24.3 -> 22.4; 192: 6272 x 2048 x 512 17.0 -> 15.7)
    epilogue = 550.0 + 9.0 * bn;
    if (4.0 * p.M * p.N > 64e6) epilogue = std::max(epilogue, 200.0 + 13.0 * bn);
    if (bn > 192) epilogue += 600.0;
  }
  return waves * (std::max(main_loop, epilogue) + 100.0) + epilogue + (pair ? 800.0 : 0.0);
}

// The tiling with the least estimated time: N tile (a multiple of step) on
// single CTAs or, where allowed, CTA pairs. Ties prefer single CTAs, then wider tiles.
void choose_tile(const Problem& p, int step, bool pairs_allowed, int* bn, bool* pair) {
  double best = -1.0;
  for (int two = 0; two <= (pairs_allowed ? 1 : 0); ++two)
    for (int b = 256; b >= step; b -= step) {
      const double cost = tile_cost(p, b, two != 0);
      if (best < 0.0 || cost < best) {
        best = cost;
        *bn = b;
        *pair = two != 0;
      }
    }
}

}  // namespace

namespace {

// Splits the pool between the operand ring and the epilogue's staging pieces.
// cbufs counts pieces per epilogue warp: one, or with a residual read through them
// (its fetch depth) as many of two as leave 3 operand stages, 5 under an fp32 residual
// past 8 k-blocks and 4 under a 16-bit one past 4 (one piece, then two and fewer
// stages: 50432 x 576 x 640 51.0 us, 53.6; 6272 x 2048 x 512 in 192 columns 15.7,
// 16.7). A 16-bit residual's one-k-block tiles take three pieces and 2 stages
// (401408 x 256 x 64 in 128 columns: 71.2 us, 74.6 with two pieces).
bool ring_layout(GemmArgs* a, int epi) {
  const int stage = a->b_stage + A_STAGE, piece = epi_warps(epi) * WBUF;
  const bool resid = epi == EPI_BIAS_RESID_F32 || is_resid16(epi);
  const int kb = (a->K + BK - 1) / BK;
  int most = resid ? 2 : 1, least = 3;
  if (is_resid16(epi)) {
    if (kb == 1) {
      most = MAX_CBUFS;
      least = 2;
    } else if (kb > 4) {
      least = 4;
    }
  } else if (resid && kb > 8) {
    least = 5;
  }
  for (int e = most; e >= 1; --e) {
    a->cbufs = e;
    a->stages = std::min((POOL - e * piece) / stage, MAX_STAGES);
    if (a->stages >= least) break;
  }
  return a->stages >= 2 && a->stages * stage + a->cbufs * piece <= POOL;
}

}  // namespace

elasto_status gemm_plan(GemmPlan* p, const bf16* A, int M_cap, const bf16* W, int N, int K, const float* bias,
                        void* out, int ldo, int epi, int* status, const bf16* W_lo, int M_hint, int ldw,
                        int bn_force) {
  if (!p || M_cap <= 0 || N <= 0 || K < 0 || !out || (K > 0 && (!A || !W))) {
    set_error("gemm_plan: invalid arguments");
    return ELASTO_ERR_INVALID_ARG;
  }
  if (ldw <= 0) ldw = K;
  if (K % 8 != 0 || N % 2 != 0 || ldw < K || ldw % 8 != 0) {
    set_error("gemm: K and ldw must be multiples of 8 (ldw >= K) and N even");
    return ELASTO_ERR_UNSUPPORTED;
  }
  *p = GemmPlan{};
  if (epi == EPI_BIAS_RESID_F32) epi = EPI_BIAS_ADD_F32;  // the residual is the output itself
  const bool resid16 = is_resid16(epi);
  const bool f32_out = epi == EPI_BIAS_ADD_F32 || epi == EPI_PART_F32;
  const bool tma_out = epi != EPI_BIAS_F32;
  GemmArgs& a = p->args;
  a.f16 = (epi == EPI_BIAS_RELU_F16 || epi == EPI_BIAS_F16 || epi == EPI_BIAS_RESID_RELU_F16) ? 1 : 0;
  a.M = M_cap;
  a.N = N;
  a.K = K;
  const int Mt = (M_hint > 0 && M_hint < M_cap) ? M_hint : M_cap;  // rows the tiling is chosen for
  const int planes = W_lo ? 2 : 1;
  // 16-bit staging chunks are 64 columns wide: their tiles are multiples of 64
  const int step = (tma_out && !f32_out) ? 64 : 32;
  const int sms = num_sms() > 0 ? num_sms() : 152;
  // CTA pairs (256-row tiles, each CTA loading half of B): the TMA-store
  // epilogues without a 16-bit residual, single-plane weights
  bool pair = false;
  a.bn = bn_force;
  if (bn_force <= 0)
    choose_tile({Mt, N, K, planes, epi, false, sms}, step, tma_out && !resid16 && !W_lo && Mt >= 2 * BM && K > 0, &a.bn,
                &pair);
  a.pair = pair ? 1 : 0;
  // one B stage holds exactly the tile's rows (both planes); the freed bytes
  // become a deeper operand ring for narrow tiles
  a.b_stage = stage_bytes(a.bn, pair, planes) - A_STAGE;
  a.bias = bias;
  a.out = out;
  a.ldo = ldo;
  a.status = status;
  a.b_planes = planes;
  // Reduce-add stores move 5.1 TB/s of X, loads and stores 5.8, so X is read
  // ahead where memory sets the pace: X past the L2 and a short reduction. 50432 x
  // 768: K = 192 64.5 us added, 54.7 read ahead; 576 65.9, 62.3; 768 67.4, 67.6;
  // 1536 85, 90 (X in the L2, 6304 x 768 x 768: 11.5, 14.9). In the forward a tie
  // goes to the added form: ViT-B, 128 images, K = 768 4.06 -> 4.02 ms. Read ahead
  // too on a nearly idle chip, where the read hides behind the main loop and a
  // reduce-add completes later.
  const int rows = pair ? 2 * BM : BM;
  const long tiles = static_cast<long>((Mt + rows - 1) / rows) * ((N + a.bn - 1) / a.bn);
  const bool memory_bound = K <= 700 && 4.0 * Mt * N > 64e6;
  if (epi == EPI_BIAS_ADD_F32 && (memory_bound || 4 * tiles <= (pair ? sms / 2 : sms))) epi = EPI_BIAS_RESID_F32;
  p->epi = epi;
  if (tma_out) {
    if (!ring_layout(&a, epi)) {
      set_error("gemm_plan: shared-memory layout does not fit");
      return ELASTO_ERR_UNSUPPORTED;
    }
    if (ldo % 8 != 0 ||
        !encode_tmap_2d(&p->tmC, out, ldo, M_cap, static_cast<uint64_t>(ldo) * (f32_out ? 4 : 2),
                        f32_out ? 32 : 64, 32, f32_out)) {
      set_error("gemm_plan: output tensor map (alignment or size)");
      return ELASTO_ERR_UNSUPPORTED;
    }
    p->tmR = p->tmC;
  } else {
    a.stages = std::min((POOL - 4 * EPI_TILE * 4) / (A_STAGE + a.b_stage), 4);
    a.cbufs = 0;
    if (a.stages < 2) {
      set_error("gemm_plan: shared-memory layout does not fit");
      return ELASTO_ERR_UNSUPPORTED;
    }
  }
  if (K > 0) {
    if (!encode_tmap_2d(&p->tmA, A, K, M_cap, static_cast<uint64_t>(K) * 2, BK, BM) ||
        !encode_tmap_2d(&p->tmB, W, K, N, static_cast<uint64_t>(ldw) * 2, BK, pair ? a.bn / 2 : a.bn) ||
        (W_lo && !encode_tmap_2d(&p->tmB2, W_lo, K, N, static_cast<uint64_t>(ldw) * 2, BK, a.bn))) {
      set_error("gemm_plan: cuTensorMapEncodeTiled failed (alignment or size)");
      return ELASTO_ERR_UNSUPPORTED;
    }
  }
  p->valid = true;
  return ELASTO_OK;
}

elasto_status gemm_plan_split_resid(GemmPlan* p, const bf16* A, int M_cap, const bf16* W, int N, int K,
                                    const float* bias, float* out, int ldo, int* status, const bf16* W_lo, int M_rows,
                                    int ldw, float* part, size_t part_floats) {
  const int sms = num_sms() > 0 ? num_sms() : 148;
  const int rows = (M_rows > 0 && M_rows < M_cap) ? M_rows : M_cap;
  const int mt = (rows + BM - 1) / BM, nk = (K + BK - 1) / BK;
  // the N tile and split count with the fewest k-blocks per CTA, every
  // split keeping at least 4 k-blocks
  int best_bn = 0, best_ks = 1, best_kb = nk + 1;
  for (int bn : {64, 32}) {
    const int tiles = mt * ((N + bn - 1) / bn);
    const int ks = std::min({kSplitMax, sms / std::max(tiles, 1), nk / 4});
    if (ks < 2 || static_cast<size_t>(ks) * rows * N > part_floats) continue;
    const int kb = (nk + ks - 1) / ks;
    if (kb < best_kb) {
      best_kb = kb;
      best_bn = bn;
      best_ks = ks;
    }
  }
  // past one image's rows the partial sums cost more: worth it from 16 k-blocks
  // (of one weight plane) saved (ViT-B 3 images, FC2 48 -> 24: 572 -> 525 us a
  // forward; ViT-S 4 images, FC2 18 -> 6, lost: 384 -> 396)
  if (rows > 256 && (nk - best_kb) * (W_lo ? 2 : 1) < 16) best_bn = 0;
  if (best_bn == 0 || !part || N % 4 != 0 || ldo % 4 != 0)
    return gemm_plan(p, A, M_cap, W, N, K, bias, out, ldo, EPI_BIAS_RESID_F32, status, W_lo, M_rows, ldw);
  elasto_status st =
      gemm_plan(p, A, M_cap, W, N, K, nullptr, part, N, EPI_PART_F32, status, W_lo, rows, ldw, best_bn);
  if (st != ELASTO_OK) return st;
  // [split][row][N], rows past `rows` of a tile clipped
  const uint64_t pd[3] = {uint64_t(N), uint64_t(rows), uint64_t(best_ks)};
  const uint64_t ps[2] = {uint64_t(N) * 4, uint64_t(rows) * N * 4};
  const uint32_t pb[3] = {32u, 32u, 1u};
  if (!encode_tmap_plain(&p->tmC, part, 3, pd, ps, pb, true, true)) {
    set_error("gemm_plan_split_resid: tensor map (alignment or size)");
    return ELASTO_ERR_UNSUPPORTED;
  }
  p->args.ksplit = best_ks;
  p->args.split_stride = static_cast<long long>(rows) * N;
  p->rbias = bias;
  p->rout = out;
  p->rldo = ldo;
  p->rcap = rows;
  return ELASTO_OK;
}

bool gemm_split_fuse_layernorm(GemmPlan* p, const float* g, const float* b, bf16* y, int d_true) {
  if (!p || p->args.ksplit <= 1 || !g || !b || !y || p->rldo != p->args.N || p->args.N % 64 != 0 ||
      p->args.N > 1024 || d_true <= 0 || d_true > p->args.N)
    return false;
  p->ln_g = g;
  p->ln_b = b;
  p->ln_y = y;
  p->ln_d = d_true;
  return true;
}

namespace {

// The part both convolution plans share. A is read through the 4D map
// {channels, x, y, image} = xd (byte strides xs) in boxes of bke channels by
// the tile's pixel block; k-block kb covers tap kb / cg (ky = tap / taps_x,
// kx = tap % taps_x) and channel group kb % cg.
elasto_status plan_conv_common(GemmPlan* p, const char* who, const void* x, const uint64_t xd[4],
                               const uint64_t xs[3], int B_cap, int Ho, int Wo, int taps, int taps_x, int cg, int bke,
                               int stride, int pad, const void* Wt, int N, const float* bias, void* out, int ldo,
                               int epi, int* status) {
  *p = GemmPlan{};
  GemmArgs& a = p->args;
  const bool k16 = bke == 16;
  a.M = B_cap;
  a.N = N;
  a.K = taps * cg * bke;
  a.k16 = k16 ? 1 : 0;
  a.conv = 1;
  a.cv_ks = taps_x;
  a.cv_stride = stride;
  a.cv_pad = pad;
  a.cv_cgroups = cg;
  a.cv_ho = Ho;
  a.cv_wo = Wo;
  // pixel block of an M tile: the fewest tiles of at most 128 pixels; whole
  // images when several fit (then nb images per tile)
  long best = -1;
  if (Ho * Wo <= BM / 2) {
    a.cv_bw = Wo;
    a.cv_bh = Ho;
    a.cv_nb = BM / (Ho * Wo);
    best = (B_cap + a.cv_nb - 1) / a.cv_nb;
  }
  for (int bw = 1; bw <= Wo && bw <= BM; ++bw)
    for (int bh = 1; bh <= Ho && bw * bh <= BM; ++bh) {
      const long tiles = long((Wo + bw - 1) / bw) * ((Ho + bh - 1) / bh) * B_cap;
      if (best < 0 || tiles < best || (tiles == best && a.cv_nb == 1 && bw > a.cv_bw)) {
        best = tiles;
        a.cv_bw = bw;
        a.cv_bh = bh;
        a.cv_nb = 1;
      }
    }
  const int rows = a.cv_bw * a.cv_bh * a.cv_nb;
  a.cv_a_bytes = rows * bke * 2;
  a.cv_batch = B_cap;
  const int Mt = conv_mtiles(a) * BM;
  const Problem prob{Mt, N, a.K, 1, epi, true, num_sms() > 0 ? num_sms() : 152};
  bool pair = false;
  choose_tile(prob, 64, false, &a.bn, &pair);
  a.bias = bias;
  a.out = out;
  a.ldo = ldo;
  a.status = status;
  a.b_planes = 1;
  a.f16 = 1;
  // one N tile whose whole W fits beside a 4-stage A ring: W is loaded once
  // per CTA and kept, instead of once per tile and k-block from L2
  const int nk = taps * cg;
  const int b_all = nk * a.bn * bke * 2;
  a.b_resident = (N <= a.bn && 4 * A_STAGE + b_all + CBUF <= POOL) ? 1 : 0;
  if (!a.b_resident && !k16) choose_tile(prob, 64, true, &a.bn, &pair);
  a.pair = pair ? 1 : 0;
  // halo tiles where they are estimated faster than a box per tap (a 16-channel
  // box takes as long as a 64-channel one: counted as a k-block per tap); their
  // offsets within an image are 32-bit, in 16-byte units
  double halo = 0.0;
  Problem boxes = prob;
  boxes.K = nk * BK;
  if ((!k16 || (taps_x == 3 && taps == 9)) && stride == 1 && static_cast<int64_t>(Ho) * Wo * ldo < (int64_t(1) << 34) &&
      halo_layout(&p->halo, B_cap, Ho, Wo, taps_x, taps / taps_x, cg, pad, N, prob.sms, &halo) &&
      halo < tile_cost(boxes, a.bn, pair)) {
    p->halo.tap_stride = cg * bke;
    p->halo.bias = bias;
    p->halo.out = out;
    p->halo.ldo = ldo;
    p->halo.status = status;
    // (the output has no map that would refuse its address: it is stored by 16-byte pieces)
    if (reinterpret_cast<uintptr_t>(out) % 16 != 0 || !halo_maps(p, x, xd, xs, Wt)) {
      set_error(std::string(who) + ": cuTensorMapEncodeTiled failed (alignment or size)");
      return ELASTO_ERR_UNSUPPORTED;
    }
    p->use_halo = true;
    p->epi = epi;
    p->valid = true;
    return ELASTO_OK;
  }
  a.b_stage = (a.pair ? a.bn / 2 : a.bn) * (a.b_resident ? bke : BK) * 2;
  const int ring = POOL - (a.b_resident ? b_all : 0), stage = A_STAGE + (a.b_resident ? 0 : a.b_stage);
  a.stages = std::min((ring - CBUF) / stage, MAX_STAGES);
  a.cbufs = 1;
  if (rows > BM || a.stages < 2) {
    set_error(std::string(who) + ": shared-memory layout does not fit");
    return ELASTO_ERR_UNSUPPORTED;
  }
  const uint32_t xb[4] = {uint32_t(bke), uint32_t(a.cv_bw * stride), uint32_t(a.cv_bh * stride), uint32_t(a.cv_nb)};
  const uint32_t xe[4] = {1u, uint32_t(stride), uint32_t(stride), 1u};
  const uint64_t od[4] = {uint64_t(N), uint64_t(Wo), uint64_t(Ho), uint64_t(B_cap)};
  const uint64_t os[3] = {uint64_t(ldo) * 2, uint64_t(Wo) * ldo * 2, uint64_t(Ho) * Wo * ldo * 2};
  const uint32_t ob[4] = {64u, uint32_t(a.cv_bw), uint32_t(a.cv_bh), uint32_t(a.cv_nb)};
  const uint32_t oe[4] = {1u, 1u, 1u, 1u};
  const bool wmap = k16 ? encode_tmap_2d_sw32(&p->tmB, Wt, a.K, N, uint64_t(a.K) * 2, 16, a.bn)
                        : encode_tmap_2d(&p->tmB, Wt, a.K, N, uint64_t(a.K) * 2, BK, a.pair ? a.bn / 2 : a.bn);
  if (xb[1] > 256 || xb[2] > 256 || !encode_tmap_4d(&p->tmA, x, xd, xs, xb, xe, k16) || !wmap ||
      !encode_tmap_4d(&p->tmC, out, od, os, ob, oe)) {
    set_error(std::string(who) + ": cuTensorMapEncodeTiled failed (alignment or size)");
    return ELASTO_ERR_UNSUPPORTED;
  }
  p->tmR = p->tmC;
  p->epi = epi;
  p->valid = true;
  return ELASTO_OK;
}

bool conv_args_ok(const GemmPlan* p, const void* x, const void* Wt, void* out, int B_cap, int N, int ldo, int epi) {
  return p && x && Wt && out && B_cap > 0 && N > 0 && (epi == EPI_BIAS_RELU_F16 || epi == EPI_BIAS_F16);
}

}  // namespace

elasto_status gemm_plan_conv(GemmPlan* p, const void* x, int B_cap, int H, int W, int C, int k, int stride, int pad,
                             const void* Wt, int N, const float* bias, void* out, int ldo, int epi, int* status,
                             int Ho_out, int Wo_out) {
  if (!conv_args_ok(p, x, Wt, out, B_cap, N, ldo, epi) || H <= 0 || W <= 0 || C <= 0 || k <= 0 || stride <= 0 ||
      pad < 0) {
    set_error("gemm_plan_conv: invalid arguments");
    return ELASTO_ERR_INVALID_ARG;
  }
  const int Ho_full = (H + 2 * pad - k) / stride + 1, Wo_full = (W + 2 * pad - k) / stride + 1;
  const int Ho = Ho_out > 0 ? Ho_out : Ho_full, Wo = Wo_out > 0 ? Wo_out : Wo_full;
  if (Ho > Ho_full || Wo > Wo_full) {
    set_error("gemm_plan_conv: the output window exceeds the convolution's output");
    return ELASTO_ERR_INVALID_ARG;
  }
  if (C % 8 != 0 || ldo % 8 != 0 || N % 2 != 0 || N > ldo || Ho <= 0 || Wo <= 0 || stride > 2) {
    set_error("gemm_plan_conv: needs C and ldo multiples of 8, N even, stride 1 or 2");
    return ELASTO_ERR_UNSUPPORTED;
  }
  // up to 16 channels: one 16-wide k-block per tap (32-byte swizzle) instead
  // of a 64-channel group that would be three quarters zeros
  const int bke = conv_tap_stride(C) == 16 ? 16 : BK;
  const uint64_t xd[4] = {uint64_t(C), uint64_t(W), uint64_t(H), uint64_t(B_cap)};
  const uint64_t xs[3] = {uint64_t(C) * 2, uint64_t(W) * C * 2, uint64_t(H) * W * C * 2};
  return plan_conv_common(p, "gemm_plan_conv", x, xd, xs, B_cap, Ho, Wo, k * k, k, conv_tap_stride(C) / bke, bke,
                          stride, pad, Wt, N, bias, out, ldo, epi, status);
}

elasto_status gemm_plan_conv_rows(GemmPlan* p, const void* x, int B_cap, int Hp, int Wp, int C, int kh, int kw,
                                  const void* Wt, int N, const float* bias, void* out, int ldo, int epi, int* status,
                                  int Ho_out, int Wo_out) {
  if (!conv_args_ok(p, x, Wt, out, B_cap, N, ldo, epi) || C <= 0 || kh <= 0 || kw <= 0 || Hp < kh || Wp < kw) {
    set_error("gemm_plan_conv_rows: invalid arguments");
    return ELASTO_ERR_INVALID_ARG;
  }
  const int Ho_full = Hp - kh + 1, Wo_full = Wp - kw + 1;
  const int Ho = Ho_out > 0 ? Ho_out : Ho_full, Wo = Wo_out > 0 ? Wo_out : Wo_full;
  if (Ho > Ho_full || Wo > Wo_full) {
    set_error("gemm_plan_conv_rows: the output window exceeds the convolution's output");
    return ELASTO_ERR_INVALID_ARG;
  }
  if (kw * C != BK || C % 8 != 0 || ldo % 8 != 0 || N % 2 != 0 || N > ldo) {
    set_error("gemm_plan_conv_rows: needs kw * C == 64, C and ldo multiples of 8, N even");
    return ELASTO_ERR_UNSUPPORTED;
  }
  // the map's x axis steps one pixel (C channels) while each box row takes
  // kw * C = 64 values: the kw pixels that kernel row ky meets, overlapping
  // the next row's; x runs over the Wo_full window starts only, so no box row
  // reaches past the end of an input row
  const uint64_t xd[4] = {uint64_t(BK), uint64_t(Wo_full), uint64_t(Hp), uint64_t(B_cap)};
  const uint64_t xs[3] = {uint64_t(C) * 2, uint64_t(Wp) * C * 2, uint64_t(Hp) * Wp * C * 2};
  return plan_conv_common(p, "gemm_plan_conv_rows", x, xd, xs, B_cap, Ho, Wo, kh, 1, 1, BK, 1, 0, Wt, N, bias, out,
                          ldo, epi, status);
}

elasto_status gemm_set_residual_source(GemmPlan* p, const void* src, int M_cap, int row_period) {
  const bool f32 = p && (p->epi == EPI_BIAS_ADD_F32 || p->epi == EPI_BIAS_RESID_F32);
  const bool r16 = p && is_resid16(p->epi);
  if (!p || !p->valid || !(f32 || r16) || !src) {
    set_error("gemm_set_residual_source: needs a residual plan and a source");
    return ELASTO_ERR_INVALID_ARG;
  }
  if (row_period < 0 || (row_period > 0 && (p->args.conv || M_cap < row_period + BM))) {
    set_error("gemm_set_residual_source: a periodic source needs period + 128 rows and a plain GEMM");
    return ELASTO_ERR_INVALID_ARG;
  }
  p->args.resid_row_mod = row_period;
  const int ldo = p->args.ldo;
  if (f32) {  // the residual is read: stores instead of reduce-adds, and the staging depth to fetch it ahead
    p->epi = EPI_BIAS_RESID_F32;
    if (!ring_layout(&p->args, p->epi)) {
      set_error("gemm_set_residual_source: shared-memory layout does not fit");
      return ELASTO_ERR_UNSUPPORTED;
    }
  }
  if (!encode_tmap_2d(&p->tmR, src, ldo, M_cap, static_cast<uint64_t>(ldo) * (f32 ? 4 : 2), f32 ? 32 : 64, 32,
                      f32)) {
    set_error("gemm_set_residual_source: tensor map (alignment or size)");
    return ELASTO_ERR_UNSUPPORTED;
  }
  return ELASTO_OK;
}

namespace {

cudaError_t gemm_launch_main(const GemmPlan& p, int M, cudaStream_t s) {
  const bool two = p.args.b_planes == 2, pair = p.args.pair != 0;
#define CASE(E) \
  case E: return two ? launch_epi<E, 2, false>(p, M, s) : launch_epi<E, 1, false>(p, M, s);
#define CASE_PAIR(E)                                   \
  case E:                                              \
    if (pair) return launch_epi<E, 1, true>(p, M, s);  \
    return two ? launch_epi<E, 2, false>(p, M, s) : launch_epi<E, 1, false>(p, M, s);
  switch (p.epi) {
    CASE_PAIR(EPI_BIAS_BF16)
    CASE_PAIR(EPI_BIAS_GELU_BF16)
    CASE_PAIR(EPI_BIAS_RESID_F32)
    CASE_PAIR(EPI_BIAS_ADD_F32)
    CASE(EPI_BIAS_F32)
    CASE(EPI_PART_F32)
    CASE_PAIR(EPI_BIAS_RELU_BF16)
    CASE(EPI_BIAS_RESID_RELU_BF16)
    CASE_PAIR(EPI_BIAS_RELU_F16)
    CASE_PAIR(EPI_BIAS_F16)
    CASE(EPI_BIAS_RESID_RELU_F16)
#undef CASE
#undef CASE_PAIR
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t gemm_launch(const GemmPlan& p, int M, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  if (p.use_halo) return halo_launch(p, M, s);
  if (p.args.ksplit <= 1) return gemm_launch_main(p, M, s);
  if (M > p.rcap) return cudaErrorInvalidValue;  // the partial buffer holds rcap rows
  cudaError_t e = gemm_launch_main(p, M, s);
  if (e != cudaSuccess) return e;
  if (p.ln_y) {
    const float inv_d = 1.0f / static_cast<float>(p.ln_d), pad = static_cast<float>(p.args.N - p.ln_d);
    return launch_pdl(splitk_reduce_ln_kernel, dim3(M), dim3(p.args.N / 2), 0, s,
                      static_cast<const float*>(p.args.out), p.args.ksplit, p.args.split_stride, p.args.N, p.rbias,
                      p.rout, p.ln_g, p.ln_b, p.ln_y, inv_d, pad);
  }
  const size_t work = static_cast<size_t>(M) * (p.args.N / 4);
  const unsigned grid = static_cast<unsigned>(std::min<size_t>((work + 255) / 256, 4096));
  return launch_pdl(splitk_reduce_kernel, dim3(grid), dim3(256), 0, s, static_cast<const float*>(p.args.out),
                    p.args.ksplit, p.args.split_stride, M, p.args.N, p.rbias, p.rout, p.rldo);
}

}  // namespace elasto
