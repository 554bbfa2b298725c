// Stride-1 convolution whose input tile is loaded once and read by every tap
// (Eq. 7's 3x3 convolutions over the kept channels, and the CNN stem).
//
// The implicit GEMM of gemm.cu loads one 4-D box per (tap, 64-channel group):
// a 3x3 convolution brings each input pixel into shared memory nine times, and
// the boxes, not the tensor cores, set its pace. Here a CTA loads the (bh + taps_y - 1) x
// (bw + taps_x - 1) halo of its bw x bh output pixels once per channel group.
// In shared memory a pixel is one 128-byte row, pixels in row-major order of
// the halo, wp to a row; the accumulator's row r = y * wp + x is output pixel
// (y, x) of the block, so tap (ky, kx) reads the 128 consecutive halo rows that
// start at ky * wp + kx: the same tile, another start address (the 128-byte
// swizzle follows address bits, so a window may start at any row). Rows with
// x >= bw, and those past the block, compute values that are never stored.
//
// Two CTAs on neighbouring SMs work as a pair (tcgen05.mma.cta_group::2,
// M = 256): each has its own block and half of the filter rows, which halves
// the filter traffic; all of the filter stays in shared memory where it fits.
//
// Roles: warp 0 input producer (and the resident filter), warp 1 MMA issuer
// (even CTA), warps 2-9 epilogue (two groups of four, every second 64-column
// chunk each: bias, ReLU, f16, staged through 4 KB of shared memory per warp
// into 16-byte stores of whole pixels), warp 10 filter producer. Every mbarrier
// wait is bounded; a timeout records ELASTO_ERR_TIMEOUT.
//
// What bounds it: the MMAs, and issuing them: the taps are unrolled, with 32-bit
// descriptor sums (tc_mma_pair_warp_lo), for 3 x 3 and the stem's 1 x 4; below 64
// output channels and in the stem the epilogue, whose tile coordinates advance by
// additions (TileWalk; 128 images of 56 x 56 x 32 27.0 -> 24.3 us, the stem 81 ->
// 70). Tried there without gain: a third group of epilogue warps (stem 73), four
// accumulators instead of two (72).
// 400 calls back to back on one GPU, gemm.cu's box per tap on single CTAs -> here,
// 128 images: 56 x 56 x 64 -> 64 channels 52.3 -> 25.9 us (35.9 with the taps in
// a loop), 56 x 56 x 32 -> 32 48.9 -> 24.0, 56 x 56 x 16 -> 16 49.3 -> 19.7, 28 x
// 28 x 128 -> 128 28.6 -> 20.1 (1.47 PFLOP/s), 28 x 28 x 96 -> 96 27.9 -> 16.4, 14
// x 14 x 256 -> 256 28.0 -> 25.1, 14 x 14 x 192 -> 192 17.7 -> 16.9. 7 x 7 images
// (49 of 128 rows) stay with the box per tap. So do strides: the
// four parity tiles of a 3 x 3 of stride 2 hold one to four taps each (100 images
// of 28 x 28 x 192 at stride 2: 23.7 us on such tiles, 19.0 with a box per tap).
#include <algorithm>

#include "common.h"
#include "ptx.cuh"

namespace elasto {

namespace {

constexpr int ROWS = 128;               // accumulator rows of a CTA
constexpr int EPI_WARPS = 8, THREADS = 64 + 32 * EPI_WARPS + 32;
constexpr int WBUF = 32 * 128;          // staging of one epilogue warp
constexpr int POOL = 224 * 1024;        // input stages, filter, staging
constexpr int MAX_A = 8, MAX_B = 8;     // ring depths
constexpr int TMEM_COLS = 512, ACC_COLS = 256;
constexpr size_t SMEM_BYTES = 1024 + POOL + 2048;
constexpr int BARS = 2 * MAX_A + 2 * MAX_B + 6;  // mbarriers: rings, tfull, tempty, drain, one to pad
static_assert(BARS * 8 % 16 == 0 && BARS * 8 + EPI_WARPS * 128 + 4 <= 2048, "barriers and bias");
static_assert(SMEM_BYTES <= 232448, "shared memory");

// The tiles a CTA works on, in order: N tile n and this CTA's pixel block
// (column x, row y of image b) of tile t0, t0 + step, ... Advanced by additions
// with carries: the divisions, one after another, are a large part of a narrow
// tile's time otherwise.
struct TileWalk {
  struct Pos {
    int x, y, b;
  };
  int n;
  Pos k;
  int nt, nbx, nby, dn;
  Pos d, pair;  // blocks between two tiles, and in a pair

  __device__ __forceinline__ Pos split(int i) const {
    const int r = i / nbx;
    return {i - r * nbx, r % nby, r / nby};
  }
  __device__ __forceinline__ void add(const Pos& v) {
    k.x += v.x;
    k.y += v.y;
    k.b += v.b;
    if (k.x >= nbx) {
      k.x -= nbx;
      ++k.y;
    }
    if (k.y >= nby) {
      k.y -= nby;
      ++k.b;
    }
  }
  __device__ __forceinline__ TileWalk(const HaloArgs& a, int nt_, int t0, int step, int rank)
      : nt(nt_), nbx(a.nbx), nby(a.nby) {
    n = t0 % nt;
    dn = step % nt;
    k = split(t0 / nt * 2 + rank);
    d = split(step / nt * 2);
    pair = split(2);
  }
  __device__ __forceinline__ void next() {
    add(d);
    n += dn;
    if (n >= nt) {
      n -= nt;
      add(pair);
    }
  }
};

// TX x TY taps known at compile time (3 x 3, and the stem's 1 x 4), or 0. KS: K =
// 16 steps of a tap; 1 for at most 16 channels, whose filter box runs into the
// next taps past them (never read).
template <bool RELU, int TX, int TY, int KS = 4>
__global__ void __launch_bounds__(THREADS, 1)
    conv_halo_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                     const HaloArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int KSTRIDE = KS == 1 ? 16 : 64;  // filter values between two k-blocks
  const int taps = a.taps_x * a.taps_y, nk = taps * a.cgroups;
  const int half = a.bn / 2;            // filter rows of one CTA's k-block
  const int b_bytes = half * 128;
  uint8_t* sA = smem;
  uint8_t* sB = sA + a.a_stages * a.a_stage;
  uint8_t* sC = smem + POOL - EPI_WARPS * WBUF;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + POOL);
  uint64_t* a_full = bars;
  uint64_t* a_empty = a_full + MAX_A;
  uint64_t* b_full = a_empty + MAX_A;  // (resident filter: b_full[0])
  uint64_t* b_empty = b_full + MAX_B;
  uint64_t* tfull = b_empty + MAX_B;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  float* sbias = reinterpret_cast<float*>(bars + BARS);  // 32 values per epilogue warp, read as float4
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sbias + 32 * EPI_WARPS);

  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int blocks = a.batch * a.nby * a.nbx;
  const int nt = (a.N + a.bn - 1) / a.bn;
  const int tiles = (blocks + 1) / 2 * nt;
  const int rank = warp_uniform(static_cast<int>(cluster_ctarank()));
  const bool leader = rank == 0;
  const int t0 = warp_uniform(static_cast<int>(cluster_id_x()));
  const int step = warp_uniform(static_cast<int>(cluster_count_x()));

  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_A; ++s) {
      mbar_init(&a_full[s], 1);
      mbar_init(&a_empty[s], 1);
    }
    for (int s = 0; s < MAX_B; ++s) {
      mbar_init(&b_full[s], 1);
      mbar_init(&b_empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 2 * EPI_WARPS);
    }
    mbar_init(drain, 1);
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc_pair(tmem_slot, TMEM_COLS);
    tmem_relinquish_pair();
  }
  if (warp == 1 && elect_one()) {
    tma_prefetch_desc(&tmX);
    tma_prefetch_desc(&tmW);
  }
  tc_fence_before();
  cluster_sync_all();  // both CTAs' barriers initialised before any remote arrive
  tc_fence_after();
  const uint32_t tmem = warp_uniform(static_cast<int>(*tmem_slot));
  // A model's filter is not written by an earlier kernel of the stream
  // (w_const): its producers start before the wait for that kernel.
  if (a.b_resident && warp == 0 && t0 < tiles && elect_one()) {
    if (!a.w_const) pdl_wait();
    if (leader) mbar_expect_tx(&b_full[0], 2u * nk * b_bytes);
    const uint32_t bar = cluster_map(smem_addr(&b_full[0]), 0);
    for (int k = 0; k < nk; ++k) tma_load_2d_pair(sB + k * b_bytes, &tmW, bar, k * KSTRIDE, rank * half);
  }
  const bool early = warp == 10 && !a.b_resident && a.w_const;
  if (!early) {
    pdl_wait();
    pdl_trigger();
  }

  if (warp == 0) {
    // ------------------------------------------------------------ input producer
    if (elect_one()) {
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      long issued = 0;
      TileWalk w(a, nt, t0, step, rank);
      for (int t = t0; t < tiles && ok; t += step, w.next()) {
        // (the last pair's second block may not exist: b = batch, all read as zero or never stored)
        for (int g = 0; g < a.cgroups; ++g) {
          if (!mbar_wait(&a_empty[s], ph ^ 1)) {
            ok = false;
            break;
          }
          if (leader) mbar_expect_tx(&a_full[s], 2u * a.a_tx);
          tma_load_4d_pair(sA + s * a.a_stage, &tmX, cluster_map(smem_addr(&a_full[s]), 0), g * 64, w.k.x * a.bw - a.pad,
                           w.k.y * a.bh - a.pad, w.k.b);
          ++issued;
          if (++s == a.a_stages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok) record_status(a.status, ELASTO_ERR_TIMEOUT);
      // no copy may still be landing when the CTAs exit: the even CTA's
      // barriers count both CTAs' bytes, and the cluster barrier below keeps
      // the odd CTA until they are in
      for (long i = issued > a.a_stages ? issued - a.a_stages : 0; leader && i < issued; ++i)
        mbar_wait(&a_full[i % a.a_stages], static_cast<uint32_t>((i / a.a_stages) & 1));
      if (leader && a.b_resident && t0 < tiles) mbar_wait(&b_full[0], 0);
    }
  } else if (warp == 10) {
    // ------------------------------------------------------------ filter producer
    if (!a.b_resident && elect_one()) {
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      long issued = 0;
      int n = t0 % nt;
      const int dn = step % nt;
      for (int t = t0; t < tiles && ok; t += step, n = n + dn >= nt ? n + dn - nt : n + dn) {
        const int row = n * a.bn + rank * half;
        for (int g = 0; g < a.cgroups && ok; ++g)
          for (int tap = 0; tap < taps; ++tap) {
            if (!mbar_wait(&b_empty[s], ph ^ 1)) {
              ok = false;
              break;
            }
            if (leader) mbar_expect_tx(&b_full[s], 2u * b_bytes);
            tma_load_2d_pair(sB + s * b_bytes, &tmW, cluster_map(smem_addr(&b_full[s]), 0),
                             (tap * a.cgroups + g) * KSTRIDE, row);
            ++issued;
            if (++s == a.b_stages) {
              s = 0;
              ph ^= 1;
            }
          }
      }
      if (!ok) record_status(a.status, ELASTO_ERR_TIMEOUT);
      for (long i = issued > a.b_stages ? issued - a.b_stages : 0; leader && i < issued; ++i)
        mbar_wait(&b_full[i % a.b_stages], static_cast<uint32_t>((i / a.b_stages) & 1));
    }
    if (early) {
      pdl_wait();
      pdl_trigger();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (leader) {
      const uint32_t idesc = idesc_16_f32(2 * ROWS, a.bn, true);
      const uint32_t a_base = sdesc_lo(smem_addr(sA), 16), b_base = sdesc_lo(smem_addr(sB), 16);
      const uint32_t hi = sdesc_sw128_hi(1024), b_units = b_bytes >> 4;
      int as = 0, bs = 0, local = 0;
      uint32_t aph = 0, bph = 0;
      bool ok = t0 >= tiles || !a.b_resident || mbar_wait_warp(&b_full[0], 0);
      bool issued = false;
      for (int t = t0; t < tiles && ok; t += step, ++local) {
        const int acc = local & 1;
        if (!mbar_wait_warp(&tempty[acc], static_cast<uint32_t>((local >> 1) & 1) ^ 1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + acc * ACC_COLS;
        for (int g = 0; g < a.cgroups && ok; ++g) {
          if (!mbar_wait_warp(&a_full[as], aph)) {
            ok = false;
            break;
          }
          tc_fence_after();
          // tap (ky, kx) starts 8 * (ky * wp + kx) 16-byte units after the halo
          const uint32_t a_lo = a_base + as * (a.a_stage >> 4), wp8 = 8u * a.wp;
          auto tap_mma = [&](uint32_t lo, uint32_t b_lo, uint32_t accumulate) {
#pragma unroll
            for (uint32_t k = 0; k < KS; ++k)
              tc_mma_pair_warp_lo(d, lo + 2 * k, b_lo + 2 * k, hi, idesc, k > 0 ? 1u : accumulate);
          };
          auto streamed_tap = [&](uint32_t lo, uint32_t accumulate) -> bool {
            if (!mbar_wait_warp(&b_full[bs], bph)) return false;
            tc_fence_after();
            tap_mma(lo, b_base + bs * b_units, accumulate);
            tc_commit_pair_multicast_warp(&b_empty[bs], 0x3);
            if (++bs == a.b_stages) {
              bs = 0;
              bph ^= 1;
            }
            return true;
          };
          if constexpr (TX > 0) {  // unrolled: issuing has to keep up with the MMAs
            if (a.b_resident) {
#pragma unroll
              for (int ky = 0; ky < TY; ++ky)
#pragma unroll
                for (int kx = 0; kx < TX; ++kx)
                  tap_mma(a_lo + ky * wp8 + 8 * kx, b_base + ((ky * TX + kx) * a.cgroups + g) * b_units,
                          ky + kx > 0 ? 1u : g != 0);
            } else {
#pragma unroll
              for (int ky = 0; ky < TY; ++ky)
#pragma unroll
                for (int kx = 0; kx < TX; ++kx)
                  if (ok) ok = streamed_tap(a_lo + ky * wp8 + 8 * kx, ky + kx > 0 ? 1u : g != 0);
            }
          } else {
            for (int ky = 0; ky < a.taps_y && ok; ++ky)
              for (int kx = 0; kx < a.taps_x && ok; ++kx) {
                const uint32_t lo = a_lo + ky * wp8 + 8 * kx;
                if (a.b_resident)
                  tap_mma(lo, b_base + ((ky * a.taps_x + kx) * a.cgroups + g) * b_units, (g | ky | kx) != 0);
                else
                  ok = streamed_tap(lo, (g | ky | kx) != 0);
              }
          }
          issued = true;
          tc_commit_pair_multicast_warp(&a_empty[as], 0x3);
          if (++as == a.a_stages) {
            as = 0;
            aph ^= 1;
          }
        }
        if (ok) tc_commit_pair_multicast_warp(&tfull[acc], 0x3);
      }
      if (!ok && lane == 0) record_status(a.status, ELASTO_ERR_TIMEOUT);
      if (issued) {  // every MMA has finished once `drain` completes
        if (elect_one()) tc_commit_pair(drain);
        mbar_wait_warp(drain, 0);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 2, q = warp & 3, grp = ew >> 2;
    uint8_t* buf = sC + ew * WBUF;
    float* sb = sbias + 32 * ew;
    // this lane's part of the stores: 16 bytes (8 channels) of eight pixels
    const int piece = lane & 7;
    uint32_t off[8], keep = 0;  // 16-byte units from the block's first pixel; bit i: row i is an output pixel
    int pos[8];                 // y << 16 | x
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = q * 32 + i * 4 + (lane >> 3), y = r / a.wp, x = r - y * a.wp;
      off[i] = static_cast<uint32_t>(y * a.Wo + x) * static_cast<uint32_t>(a.ldo / 8);
      pos[i] = y << 16 | x;
      keep |= (y < a.bh && x < a.bw ? 1u : 0u) << i;
    }
    const bool one = nt == 1;  // N <= 256: the whole bias is kept in sbias
    if (one) {
      const int c = static_cast<int>(threadIdx.x) - 64;
      sbias[c] = a.bias && c < a.N ? __ldg(a.bias + c) : 0.0f;
      named_bar_sync(1, 32 * EPI_WARPS);
    }
    const uint32_t row_tm = tmem + (static_cast<uint32_t>(q * 32) << 16);
    int local = 0, before = 0;
    bool ok = true;
    TileWalk w(a, nt, t0, step, rank);
    for (int t = t0; t < tiles; t += step, ++local, w.next()) {
      const int acc = local & 1, n0 = w.n * a.bn;
      const int width = min(a.bn, a.N - n0), chunks = (width + 63) / 64;
      int c = grp ^ before;
      before ^= chunks & 1;
      float nb[2];
      auto bias_of = [&](int chunk) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k = chunk * 64 + 32 * h + lane;
          nb[h] = a.bias && k < width ? __ldg(a.bias + n0 + k) : 0.0f;
        }
      };
      if (!one) bias_of(c);
      const int oy = w.k.y * a.bh, ox = w.k.x * a.bw;
      uint32_t outs = keep;  // of an edge block less
      if (oy + a.bh > a.Ho || ox + a.bw > a.Wo || w.k.b >= a.batch) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (oy + (pos[i] >> 16) >= a.Ho || ox + (pos[i] & 0xffff) >= a.Wo || w.k.b >= a.batch) outs &= ~(1u << i);
      }
      __half* first = static_cast<__half*>(a.out) + ((static_cast<size_t>(w.k.b) * a.Ho + oy) * a.Wo + ox) * a.ldo + n0;
      ok = __all_sync(0xffffffffu, mbar_wait(&tfull[acc], static_cast<uint32_t>((local >> 1) & 1)));
      if (!ok) break;
      tc_fence_after();
      auto release = [&] {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(cluster_map(smem_addr(&tempty[acc]), 0));
      };
      if (c >= chunks) release();
      for (; c < chunks; c += 2) {
        uint32_t v[2][32];
        tmem_ld_32x32b_x32(row_tm + acc * ACC_COLS + c * 64, v[0]);
        tmem_ld_32x32b_x32(row_tm + acc * ACC_COLS + c * 64 + 32, v[1]);
        const float bl[2] = {nb[0], nb[1]};
        if (!one && c + 2 < chunks) bias_of(c + 2);
        tmem_ld_wait();
        if (c + 2 >= chunks) release();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float* bias = sbias + c * 64 + 32 * h;
          if (!one) {
            bias = sb;
            __syncwarp();
            sb[lane] = bl[h];
            __syncwarp();
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint32_t ow[4];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float4 b4 = reinterpret_cast<const float4*>(bias)[2 * j + i];
              float2 lo = add2(make_float2(__uint_as_float(v[h][8 * j + 4 * i]), __uint_as_float(v[h][8 * j + 4 * i + 1])),
                               make_float2(b4.x, b4.y));
              float2 hi =
                  add2(make_float2(__uint_as_float(v[h][8 * j + 4 * i + 2]), __uint_as_float(v[h][8 * j + 4 * i + 3])),
                       make_float2(b4.z, b4.w));
              ow[2 * i] = pack_f16x2(lo.x, lo.y);
              ow[2 * i + 1] = pack_f16x2(hi.x, hi.y);
              if (RELU) {  // rounding keeps the sign, so the maximum can follow it
                ow[2 * i] = relu_f16x2(ow[2 * i]);
                ow[2 * i + 1] = relu_f16x2(ow[2 * i + 1]);
              }
            }
            *reinterpret_cast<uint4*>(buf + lane * 128 + (((4 * h + j) ^ (lane & 7)) << 4)) =
                make_uint4(ow[0], ow[1], ow[2], ow[3]);
          }
        }
        __syncwarp();
        const int col = c * 64 + piece * 8;
        if (col < width) {
          uint4* dst = reinterpret_cast<uint4*>(first + col);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = i * 4 + (lane >> 3);
            if (outs >> i & 1) dst[off[i]] = *reinterpret_cast<const uint4*>(buf + r * 128 + ((piece ^ (r & 7)) << 4));
          }
        }
        __syncwarp();  // the staging rows are read before the next chunk writes them
      }
    }
    if (!ok && lane == 0) record_status(a.status, ELASTO_ERR_TIMEOUT);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the peer's TMEM, barriers and copies are no longer in use
  if (warp == 0) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem, TMEM_COLS);
  }
}

using HaloKernel = void (*)(CUtensorMap, CUtensorMap, HaloArgs);
HaloKernel halo_kernel(bool relu, int taps_x, int taps_y, bool narrow) {
  if (narrow) return relu ? conv_halo_kernel<true, 3, 3, 1> : conv_halo_kernel<false, 3, 3, 1>;
  if (taps_x == 3 && taps_y == 3) return relu ? conv_halo_kernel<true, 3, 3> : conv_halo_kernel<false, 3, 3>;
  if (taps_x == 1 && taps_y == 4) return relu ? conv_halo_kernel<true, 1, 4> : conv_halo_kernel<false, 1, 4>;
  return relu ? conv_halo_kernel<true, 0, 0> : conv_halo_kernel<false, 0, 0>;
}

int round_up(int v, int m) { return (v + m - 1) / m * m; }

}  // namespace

cudaError_t halo_init_attributes() {
  const int bytes = static_cast<int>(SMEM_BYTES);
  cudaError_t e = cudaSuccess;
  for (int relu = 0; relu < 2; ++relu)
    for (int t = 0; t < 4; ++t) {
      const HaloKernel k = halo_kernel(relu != 0, t == 2 ? 1 : t == 0 ? 0 : 3, t == 2 ? 4 : t == 0 ? 0 : 3, t == 3);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(reinterpret_cast<const void*>(k), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    }
  return e;
}

bool halo_layout(HaloArgs* a, int batch, int Ho, int Wo, int taps_x, int taps_y, int cgroups, int pad, int N, int sms,
                 double* cost) {
  if (taps_x * taps_y < 2 || N % 8 != 0) return false;
  *a = HaloArgs{};
  a->batch = batch;
  a->Ho = Ho;
  a->Wo = Wo;
  a->N = N;
  a->taps_x = taps_x;
  a->taps_y = taps_y;
  a->cgroups = cgroups;
  a->pad = pad;
  // output block: the fewest blocks per image whose last pixel's row still
  // fits the 128 accumulator rows, then the smallest halo
  long best_blocks = -1;
  int best_rows = 0;
  for (int bw = 1; bw <= Wo && bw <= ROWS; ++bw) {
    const int wp = bw + taps_x - 1, bh = std::min(Ho, (ROWS - bw) / wp + 1);
    const int nbx = (Wo + bw - 1) / bw, nby = (Ho + bh - 1) / bh;
    const int bh_even = (Ho + nby - 1) / nby;  // the same number of blocks, evenly high
    const int rows = wp * (bh_even + taps_y - 1);
    if (wp > 256 || bh_even + taps_y - 1 > 256) continue;
    const long n = static_cast<long>(nbx) * nby;
    if (best_blocks < 0 || n < best_blocks || (n == best_blocks && rows < best_rows)) {
      best_blocks = n;
      best_rows = rows;
      a->bw = bw;
      a->bh = bh_even;
      a->nbx = nbx;
      a->nby = nby;
      a->wp = wp;
    }
  }
  if (best_blocks < 0) return false;
  a->a_tx = best_rows * 128;
  a->a_stage = round_up(a->a_tx, 1024);
  // the last tap's window ends this many rows past the halo's end: the rows
  // read there (never used) have to be shared memory too
  const int over = (ROWS + (taps_y - 1) * a->wp + taps_x - 1 - best_rows) * 128;
  const int pool = POOL - EPI_WARPS * WBUF, nk = taps_x * taps_y * cgroups;
  if (over > EPI_WARPS * WBUF) return false;
  const int units = sms / 2;
  *cost = -1.0;
  HaloArgs pick = *a;
  for (int n_tiles = (N + 255) / 256; n_tiles <= (N + 15) / 16; n_tiles *= 2) {
    HaloArgs b = *a;
    b.bn = round_up((N + n_tiles - 1) / n_tiles, 16);
    const int nt = (N + b.bn - 1) / b.bn, b_bytes = b.bn / 2 * 128;
    b.b_resident = nt == 1 && 2 * b.a_stage + nk * b_bytes <= pool ? 1 : 0;
    if (b.b_resident) {
      b.a_stages = std::min((pool - nk * b_bytes) / b.a_stage, MAX_A);
      b.b_stages = 1;
    } else {
      // two input stages (three where that leaves the filter ring full), the rest filter
      b.a_stages = cgroups > 1 && pool - 3 * b.a_stage >= MAX_B * b_bytes ? 3 : 2;
      b.b_stages = std::min((pool - b.a_stages * b.a_stage) / b_bytes, MAX_B);
      if (pool < b.a_stages * b.a_stage || b.b_stages < 3) continue;
    }
    // a 128-row K = 16 step takes bn / 2 clocks, 45 at least; a filter wait per k-block adds ~130
    const double mma = (4 * std::max(0.5 * b.bn, 45.0) + (b.b_resident ? 0 : 130)) / 1.9;
    const double load = (b.a_tx / (taps_x * taps_y) + (b.b_resident ? 0 : b_bytes)) / 126.0;
    const long tiles = (best_blocks * batch + 1) / 2 * nt, waves = (tiles + units - 1) / units;
    const double epilogue = 500.0 + 6.0 * b.bn;
    const double c = waves * (std::max(nk * std::max(mma, load), epilogue) + 150.0) + epilogue + 1000.0;
    if (*cost < 0 || c < *cost) {
      *cost = c;
      pick = b;
    }
    if (b.bn <= 64) break;
  }
  if (*cost < 0) return false;
  *a = pick;
  return true;
}

bool halo_maps(GemmPlan* p, const void* x, const uint64_t xd[4], const uint64_t xs[3], const void* Wt) {
  const HaloArgs& a = p->halo;
  const uint32_t box[4] = {64u, static_cast<uint32_t>(a.wp), static_cast<uint32_t>(a.bh + a.taps_y - 1), 1u};
  const uint32_t es[4] = {1u, 1u, 1u, 1u};
  const uint64_t K = static_cast<uint64_t>(a.taps_x) * a.taps_y * a.tap_stride;
  return encode_tmap_4d(&p->tmA, x, xd, xs, box, es, false) &&
         encode_tmap_2d(&p->tmB, Wt, K, a.N, K * 2, 64, a.bn / 2);
}

cudaError_t halo_launch(const GemmPlan& p, int batch, cudaStream_t s) {
  HaloArgs a = p.halo;
  a.batch = batch;
  const int nt = (a.N + a.bn - 1) / a.bn, blocks = batch * a.nby * a.nbx;
  const HaloKernel kernel = halo_kernel(p.epi == EPI_BIAS_RELU_F16, a.taps_x, a.taps_y, a.tap_stride < 64);
  int pairs = 0;
  const cudaError_t e = max_cta_pairs(reinterpret_cast<const void*>(kernel), THREADS, SMEM_BYTES, &pairs);
  if (e != cudaSuccess) return e;
  const int clusters = std::min((blocks + 1) / 2 * nt, pairs);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(2 * clusters);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, p.tmA, p.tmB, a);
}

}  // namespace elasto
