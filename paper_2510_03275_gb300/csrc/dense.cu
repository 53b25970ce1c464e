// K6 / K7: large-batch forward by rebuilding the layer's weights once per
// call, then one dense GEMM ("decimate, then dense").
//
//   W'[r, bB + k] = 2 sum_j c[r, b n_b + j] G[j, k]      (K6, per block b)
//   y[m, r]       = alpha_r / 2 sum_k W'[r, k] x[m, k]    (K7)
//
// equal to the code-domain forward y = alpha C x_tilde, x_tilde = G x per
// block (section 3.5, eq. 12), by associativity: C (G x) = (C G) x.  The
// code domain costs 2 M N K_eff flops; this route 2 M N K for the GEMM plus
// 4 N K_eff B for the rebuild (hi and lo parts of G), fewer when M exceeds
// about 2 OSR B / (OSR - 1).
//
// K6: the codes are the A operand in tensor memory (as in K5: exact bf16
// +-2 / 0 from one tcgen05.st per 64 codes), G^T the B operand, resident in
// shared memory for the CTA's lifetime (bf16 hi and lo parts, 128 output
// columns k x n_b codes, K-major, 128-byte swizzle, its K order permuted as
// the code expansion orders the codes); one 128 x 128 fp32 accumulator per
// (row tile, block) item, two of them so that an item's epilogue (bf16 W' through
// a swizzled tile and TMA stores) overlaps the next item's MMAs.  Persistent CTAs over the
// items.
//   warp 0     TMEM allocation; G^T once (TMA), then the code slabs
//   warp 1     8 MMAs per 64 codes (4 K steps x hi / lo)
//   warps 2-9  two expander sets (stages of one parity each)
//   warps 10-13 epilogue
// K7: a plain tcgen05 GEMM on CTA pairs, D[r, m] = W' x^T per pair tile of 256
// (or 2 x 256) weight rows x up to 256 batch rows, both operands TMA-loaded
// (128-byte swizzle), 6 (4) stages; epilogue as K5's.
// Every wait on an mbarrier is bounded (about 2 s); a timeout writes the call
// number into the workspace's call record and the CTA waits (again bounded)
// for its own copies and MMAs before it frees TMEM and ends.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "common.cuh"

namespace sdq {

namespace {

constexpr int kBK = 64;                    // codes (K6) or inputs (K7) per stage

// kind::f16 instruction descriptor: D fp32, A and B bf16, both K-major,
// M = 128, N = n.
__host__ __device__ constexpr uint32_t f16_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// ---------------------------------------------------------------- K6 rebuild
constexpr int kRbStages = 6;
constexpr int kRbEpiWarp0 = 10;
constexpr int kRbThreads = 32 * 14;
constexpr int kRbHalf = 128 * 128;          // epilogue buffer: 128 rows x 64 columns of bf16 W'
constexpr int kRbCTile = 128 * 16;          // code slab of a stage: 128 rows x 64 codes, at most 2 KB
constexpr uint32_t kRbAcc = 128;            // accumulator columns (128 outputs k of a block)
constexpr uint32_t kRbAcol = 2 * kRbAcc;    // first A slot column
constexpr uint32_t kRbAslot = kBK / 2;

struct ReconParams {
  const uint32_t* codes;
  uint64_t* rec;
  uint64_t call;
  int nblk, n_b, ngroups, wpg, quantizer, nitems;
  int nstage;           // epilogue buffers (1 or 2)
};

__global__ void __launch_bounds__(kRbThreads, 1)
    recon_kernel(const __grid_constant__ CUtensorMap ghmap, const __grid_constant__ CUtensorMap glmap,
                 const __grid_constant__ CUtensorMap wmap, ReconParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t g_full, full[kRbStages], empty[kRbStages], a_full[kRbStages],
      acc_full[2], acc_empty[2], mma_done;
  __shared__ uint32_t tmem_base;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base = smem_raw + (sbase - smem_u32(smem_raw));
  const int spb = p.n_b / kBK;                        // stages (64-code chunks) per block
  const uint32_t gchunk = 128u * 128u;                // one 64-code chunk of G^T: 128 rows x 128 B
  uint8_t* c_tiles = base + 2 * spb * gchunk;         // after G^T hi, lo
  const uint32_t slab_bytes = (uint32_t)(kTileRows * p.wpg * 4);

  if (tid == 0) {
    mbar_init(&g_full, 1);
    mbar_init(&mma_done, 1);
    for (int s = 0; s < kRbStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&a_full[s], 4);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 4);
    }
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(&tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();
  pdl_launch_dependents();
  prep_record_start(p.rec, p.call, blockIdx.x == 0 && tid == 0);
  const uint32_t tmem = tmem_base;
  bool ok = true;
  // this CTA's items: (row tile, block) = item / nblk, item % nblk
  const int nmine = p.nitems > (int)blockIdx.x ? (p.nitems - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const int nst = nmine * spb;

  if (warp == 0) {
    mbar_expect_tx_warp(&g_full, 2u * spb * gchunk);
    for (int c = 0; c < spb; ++c) {
      tma_load_2d_warp(base + c * gchunk, &ghmap, c * kBK, 0, &g_full);
      tma_load_2d_warp(base + (spb + c) * gchunk, &glmap, c * kBK, 0, &g_full);
    }
    int n = 0;   // slabs copied
    for (; n < nst; ++n) {
      const int i = n, s = i % kRbStages, r = i / kRbStages;
      const int item = (int)blockIdx.x + (i / spb) * (int)gridDim.x, sc = i % spb;
      const int tile = item / p.nblk, b = item - tile * p.nblk;
      if (r > 0) ok = mbar_wait_warp(&empty[s], (r - 1) & 1);
      if (!ok) break;
      mbar_expect_tx_warp(&full[s], slab_bytes);
      const uint32_t* src = p.codes + (size_t)((int64_t)tile * p.ngroups + b * spb + sc) * (slab_bytes / 4);
      bulk_g2s_warp(c_tiles + s * kRbCTile, src, slab_bytes, &full[s]);
    }
    // every copy issued has landed before the CTA ends
    if (!mbar_wait_warp(&g_full, 0)) ok = false;
    for (int j = max(0, n - kRbStages); j < n; ++j)
      if (!mbar_wait_warp(&full[j % kRbStages], (j / kRbStages) & 1)) ok = false;
  } else if (warp == 1) {
    constexpr uint32_t idesc = f16_idesc(128);
    ok = mbar_wait_warp(&g_full, 0);
    for (int i = 0; i < nst && ok; ++i) {
      const int s = i % kRbStages, r = i / kRbStages;
      const int it = i / spb, sc = i % spb, a = it & 1;
      if (sc == 0 && it >= 2) {
        ok = mbar_wait_warp(&acc_empty[a], ((it >> 1) - 1) & 1);
        if (!ok) break;
      }
      ok = mbar_wait_warp(&full[s], r & 1) && mbar_wait_warp(&a_full[s], r & 1);
      if (!ok) break;
      tc_fence_after();
      const uint64_t bh = sw128_desc(sbase + sc * gchunk);
      const uint64_t bl = sw128_desc(sbase + (spb + sc) * gchunk);
      const uint32_t d = tmem + (uint32_t)a * kRbAcc;
#pragma unroll
      for (int kk = 0; kk < kBK / 16; ++kk) {
        const uint32_t at = tmem + kRbAcol + kRbAslot * s + 8 * kk;
        umma_bf16_ts_warp(d, at, bh + 2 * kk, idesc, (sc | kk) != 0);
        umma_bf16_ts_warp(d, at, bl + 2 * kk, idesc, 1u);
      }
      umma_commit_warp(&empty[s]);
      if (sc == spb - 1) umma_commit_warp(&acc_full[a]);
    }
    umma_commit_warp(&mma_done);   // ... and every MMA is done before TMEM is freed
    if (!mbar_wait_warp(&mma_done, 0)) ok = false;
  } else if (warp < kRbEpiWarp0) {
    // Expanders: set x = (warp - 2) / 4 expands stages i = x (mod 2), thread
    // = code row 32 q + lane (q = warp % 4): 64 codes -> 32 TMEM columns.
    const int x = (warp - 2) >> 2, q = warp & 3, rr = 32 * q + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(32 * q) << 16);
    for (int i = x; i < nst && ok; i += 2) {
      const int s = i % kRbStages, r = i / kRbStages;
      ok = mbar_wait(&full[s], r & 1);
      if (ok && r > 0) ok = mbar_wait(&empty[s], (r - 1) & 1);   // the slot's previous MMAs are done
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint8_t* cs = c_tiles + s * kRbCTile;
      uint32_t v[32];
      if (p.quantizer == SDQ_TERNARY) {
        const uint4 w4 = *reinterpret_cast<const uint4*>(cs + rr * 16);
        const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int j = 0; j < 8; ++j) v[8 * k + j] = (w[k] << (2 * j)) & 0xC000C000u;
      } else {   // words hold the inverted bits: 1 = -1
        const uint2 w2 = *reinterpret_cast<const uint2*>(cs + rr * 8);
        const uint32_t w[2] = {~w2.x, ~w2.y};
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int j = 0; j < 16; ++j) v[16 * k + j] = ((w[k] << j) & 0x80008000u) | 0x40004000u;
      }
      tmem_st32(lane_addr + kRbAcol + kRbAslot * s, v);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&a_full[s]);
    }
  } else {
    // Epilogue: item it's accumulator -> W'[row, b B .. b B + 127] as bf16,
    // 64 columns at a time through a shared-memory tile (128-byte rows and
    // swizzle: no bank conflicts) and a TMA store of it (rows past n_out are
    // clipped).  Stored from registers, a lane's row at a time, every 16 bytes
    // were half a sector of their own, as long to issue as the item's MMAs.
    const int q = warp & 3, rr = 32 * q + lane, et = tid - 32 * kRbEpiWarp0;
    const uint32_t lane_addr = tmem + ((uint32_t)(32 * q) << 16);
    uint8_t* stage = c_tiles + kRbStages * kRbCTile;
    int n = 0;   // halves stored
    for (int it = 0; it < nmine && ok; ++it) {
      const int a = it & 1;
      // one outcome for the four warps: one that gave up alone would leave the
      // others in the barriers below for good
      ok = group_and(2, 128, mbar_wait_warp(&acc_full[a], (it >> 1) & 1));
      if (!ok) break;
      tc_fence_after();
      const int item = (int)blockIdx.x + it * (int)gridDim.x;
      const int tile = item / p.nblk, b = item - tile * p.nblk;
#pragma unroll 1
      for (int h = 0; h < 2; ++h, ++n) {
        uint32_t w[32];   // 64 columns as bf16 pairs
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t u[16];
          tmem_ld16(lane_addr + (uint32_t)a * kRbAcc + (uint32_t)(64 * h + 16 * c), u);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 8; ++i) w[8 * c + i] = pack_bf16x2(__uint_as_float(u[2 * i]), __uint_as_float(u[2 * i + 1]));
        }
        if (h == 1) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[a]);
        }
        if (et == 0) {   // the store that last read this buffer is done with it
          if (p.nstage == 2) bulk_store_wait_read<1>();
          else bulk_store_wait_read<0>();
        }
        named_bar_sync(1, 128);
        uint8_t* sb = stage + (p.nstage == 2 ? (n & 1) * kRbHalf : 0) + rr * 128;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          *reinterpret_cast<uint4*>(sb + ((j ^ (rr & 7)) << 4)) =
              make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
        fence_proxy_async_smem();
        named_bar_sync(1, 128);
        if (et == 0)
          tma_store_2d(&wmap, sb - rr * 128, b * 128 + 64 * h, tile * kTileRows);
      }
    }
    if (et == 0) bulk_store_wait_all();   // written before the CTA ends
  }
  if (!ok) prep_record_fail(p.rec, p.call);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------ K7 dense GEMM
// A pair of CTAs (cta_group::2) takes WT = 1 or 2 weight tiles of 256 rows (128
// of each in either CTA) against one tile of `bn` batch rows (a multiple of 32
// up to 256, half of them in either CTA's shared memory).  Each CTA loads its
// rows and signals rank 0's barriers; rank 0 issues the pair's MMAs and
// commits to both CTAs' barriers.  On single CTAs every MMA read all 256 batch
// rows from its own shared memory, and that memory, at 128 bytes a cycle,
// bound the steps: 160 KB per K step of two 128-row tiles against 1024 cycles
// of tensor work, 0.67 us; a pair reads half of that from each.  8192 x 8192 at
// M = 4096: 325 -> 301 us (1.83 PFLOP/s).
constexpr int kDnBN = 256;                  // batch rows at most
constexpr int kDnATile = 128 * kBK * 2;     // 16 KB: 128 weight rows x 64 inputs
constexpr int kDnBTile = kDnBN / 2 * kBK * 2;   // 16 KB: a CTA's half of the batch rows x 64 inputs
constexpr int kDnThreads = 320;
template <int WT> struct DnShape {
  static constexpr int kStages = WT == 1 ? 6 : 4;
  static constexpr int kStage = WT * kDnATile + kDnBTile;
  static constexpr int kSmem = kStages * kStage + 1024;
  static constexpr uint32_t kCols = WT == 1 ? 256u : 512u;
};

struct DenseParams {
  const float* alpha;
  float* y;
  uint64_t* rec;
  uint64_t call;
  int M, N, nks, bn;
  // Pair u < nfull takes unit u (weight-tile group u mod ngroups, batch tile u / ngroups, WT
  // tiles); pairs from nfull on split the remaining units into their WT single tiles
  int ngroups, nfull;
};

template <int WT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kDnThreads, 1)
    dense_kernel(const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap xmap,
                 DenseParams p) {
  constexpr int kStages = DnShape<WT>::kStages, kStage = DnShape<WT>::kStage;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[kStages], empty[kStages], acc_bar;
  __shared__ uint32_t tmem_base;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int rank = (int)cluster_rank();
  int unit = blockIdx.x >> 1, nt = WT, sub = 0;
  if (unit >= p.nfull) {
    sub = (unit - p.nfull) % WT;
    unit = p.nfull + (unit - p.nfull) / WT;
    nt = 1;
  }
  // this CTA's rows of weight tile w: n0 + 256 w ..; the pair's batch rows m0 ..
  const int n0 = (unit % p.ngroups) * 256 * WT + 256 * sub + 128 * rank, m0 = (unit / p.ngroups) * p.bn;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base = smem_raw + (sbase - smem_u32(smem_raw));
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&acc_bar, 1);
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc_pair(&tmem_base, DnShape<WT>::kCols);
  tc_fence_before();
  cluster_sync();   // both CTAs' barriers and tensor memory are set up
  tc_fence_after();
  pdl_wait();
  pdl_launch_dependents();
  call_record_start_prepared(p.rec, p.call, blockIdx.x == 0 && threadIdx.x == 0);
  const uint32_t tmem = tmem_base;
  bool ok = true;
  if (warp == 0) {
    const uint32_t bytes = (uint32_t)(nt * kDnATile + p.bn * kBK);   // of each CTA
    int ks = 0;
    for (; ks < p.nks; ++ks) {
      const int s = ks % kStages, r = ks / kStages;
      if (r > 0) ok = mbar_wait_warp(&empty[s], (r - 1) & 1);
      if (!ok) break;
      if (rank == 0) mbar_expect_tx_warp(&full[s], 2 * bytes);
      const uint32_t bar = cluster_addr(&full[s], 0);
      uint8_t* st = base + s * kStage;
#pragma unroll
      for (int w = 0; w < WT; ++w)
        if (w < nt) tma_load_2d_pair_warp(st + w * kDnATile, &wmap, ks * kBK, n0 + 256 * w, bar);
      tma_load_2d_pair_warp(st + WT * kDnATile, &xmap, ks * kBK, m0 + rank * (p.bn / 2), bar);
    }
    // the pair's copies have landed before either CTA ends
    if (rank == 0)
      for (int j = max(0, ks - kStages); j < ks; ++j)
        if (!mbar_wait_warp(&full[j % kStages], (j / kStages) & 1)) ok = false;
  } else if (warp == 1) {
    if (rank == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.bn >> 3) << 17) |
                             ((uint32_t)(256 >> 4) << 24);   // D fp32, A and B bf16, both K-major, M = 256
      const uint64_t d0 = sw128_desc(sbase);
      for (int ks = 0; ks < p.nks; ++ks) {
        const int s = ks % kStages, r = ks / kStages;
        ok = mbar_wait_warp(&full[s], r & 1);
        if (!ok) break;
        tc_fence_after();
        const uint64_t st = d0 + (uint64_t)(s * (kStage >> 4)), bd = st + (uint64_t)(WT * (kDnATile >> 4));
#pragma unroll
        for (int w = 0; w < WT; ++w) {
          if (w >= nt) break;
          const uint64_t ad = st + (uint64_t)(w * (kDnATile >> 4));
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk)
            umma_bf16_pair_warp(tmem + (uint32_t)(w * kDnBN), ad + 2 * kk, bd + 2 * kk, idesc, (ks | kk) != 0);
        }
        umma_commit_pair_warp(&empty[s]);
      }
      umma_commit_pair_warp(&acc_bar);
    }
    if (!mbar_wait_warp(&acc_bar, 0)) ok = false;   // every MMA of the pair is done
  } else {
    // Epilogue: lane quadrant q holds weight rows n0 + 256 w + 32 q + lane of
    // accumulator w; this warp writes half of its columns (batch rows).
    const int q = warp & 3, h = (warp - 2) >> 2, rr = 32 * q + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(32 * q) << 16);
    ok = mbar_wait_warp(&acc_bar, 0);
    tc_fence_after();
    if (ok) {
#pragma unroll 1
      for (int w = 0; w < nt; ++w) {
        const int row = n0 + 256 * w + rr;
        const float sa = row < p.N ? 0.5f * __ldg(p.alpha + row) : 0.f;
        const int half = p.bn / 2;
        for (int c0 = h ? half : 0; c0 < (h ? p.bn : half); c0 += 16) {
          uint32_t a[16];
          tmem_ld16(lane_addr + (uint32_t)(w * kDnBN + c0), a);
          tmem_ld_wait();
          if (row < p.N) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int m = m0 + c0 + i;
              if (m < p.M) p.y[(size_t)m * p.N + row] = __uint_as_float(a[i]) * sa;
            }
          }
        }
      }
    }
  }
  if (!ok) call_record_fail(p.rec, p.call);
  tc_fence_before();
  cluster_sync();   // both CTAs are done with the pair's tensor memory and barriers
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, DnShape<WT>::kCols);
  }
}

}  // namespace

bool dense_route_applies(const sdq_plan_s* pl, int M) {
  const Geometry& g = pl->geo;
  return M >= kDenseMinM && pl->d_gt_hi && g.block == 128 && g.n_b % kBK == 0 && g.n_b <= kDenseMaxNb &&
         g.k_in % 64 == 0;
}

namespace {
// K7's launch shape: 256-row weight tiles per pair and batch rows per tile
// with the least time over the waves of pairs.  A K step takes the longer of
// its MMAs (2 bn cycles a tile) and its shared-memory traffic in each CTA (tiles
// written once, read by every MMA, at 128 bytes a cycle: 512 + 1.5 bn with
// two tiles, 256 + bn with one); a wave's two ends take about 9000 cycles.  A
// last wave of at most half the pairs runs as single tiles on twice as many.
struct DenseShape {
  int wt, bn, ngroups, nfull, pairs;
};
DenseShape dense_shape(const sdq_plan_s* pl, int M) {
  const Geometry& g = pl->geo;
  const int slots = std::max(1, pl->pf_clusters[2]), tiles = (g.ntiles + 1) / 2;
  const double steps = g.k_in / kBK, ends = 9000.0;
  DenseShape best{};
  double best_t = 0;
  for (int wt = 2; wt >= 1; --wt)
    for (int bn = kDnBN; bn >= 96; bn -= 32) {
      DenseShape s;
      s.wt = wt;
      s.bn = bn;
      s.ngroups = (tiles + wt - 1) / wt;
      const int mt = (M + bn - 1) / bn;
      if (mt > 1 && (M + mt - 1) / mt <= bn - 32) continue;   // smaller equal tiles cover M
      const int units = s.ngroups * mt, full = units / slots, rest = units - full * slots;
      const bool split = wt == 2 && full > 0 && rest > 0 && 2 * rest <= slots;
      s.nfull = split ? full * slots : units;
      s.pairs = s.nfull + wt * (units - s.nfull);
      const double two = std::max(4.0 * bn, 512.0 + 1.5 * bn), one = std::max(2.0 * bn, 256.0 + bn);   // cycles
      const double t = full * ((wt == 2 ? two : one) * steps + ends) +
                       (rest ? (split || wt == 1 ? one : two) * steps + ends : 0.0);
      if (!best.pairs || t < best_t * 0.99) {
        best = s;
        best_t = t;
      }
    }
  return best;
}
}  // namespace

cudaError_t launch_dense_forward(const sdq_plan_s* pl, const uint32_t* codes, const float* alpha,
                                 const uint16_t* x, int M, float* y, void* ws, cudaStream_t st) {
  const Geometry& g = pl->geo;
  if ((reinterpret_cast<uintptr_t>(x) & 15u) || (g.k_in * 2) % 16) return cudaErrorNotSupported;
  auto enc = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(tensor_map_encoder());
  if (!enc) return cudaErrorNotSupported;
  const WsLayout L = workspace_layout(pl, M);
  uint8_t* wbase = static_cast<uint8_t*>(ws);
  uint16_t* wp = reinterpret_cast<uint16_t*>(wbase + L.what);
  const cuuint32_t estr[2] = {1, 1};
  const int spb = g.n_b / kBK;
  const DenseShape sh = dense_shape(pl, M);
  // K6: G^T hi / lo maps (128 rows x n_b), one 64-code chunk per box
  CUtensorMap ghmap, glmap, wmap, xmap;
  {
    const cuuint64_t dims[2] = {(cuuint64_t)g.n_b, 128};
    const cuuint64_t strides[1] = {(cuuint64_t)g.n_b * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, 128};
    if (enc(&ghmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, pl->d_gt_hi, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
        enc(&glmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, pl->d_gt_lo, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  // W' (n_out x k_in; K6 stores it, K7 loads it: rows past n_out clipped, read as zeros) and x (M x k_in)
  {
    const cuuint64_t dims[2] = {(cuuint64_t)g.k_in, (cuuint64_t)g.n_out};
    const cuuint64_t strides[1] = {(cuuint64_t)g.k_in * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, 128};
    if (enc(&wmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, wp, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  {
    const cuuint64_t dims[2] = {(cuuint64_t)g.k_in, (cuuint64_t)M};
    const cuuint64_t strides[1] = {(cuuint64_t)g.k_in * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)(sh.bn / 2)};
    if (enc(&xmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(x), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  ReconParams rp;
  rp.codes = codes;
  rp.rec = reinterpret_cast<uint64_t*>(wbase + L.err);
  rp.call = call_tag(next_call_number());
  rp.nblk = g.nblk; rp.n_b = g.n_b; rp.ngroups = g.ngroups; rp.wpg = g.wpg; rp.quantizer = pl->desc.quantizer;
  rp.nitems = g.ntiles * g.nblk;
  size_t rsmem = 1024 + 2 * (size_t)spb * 128 * 128 + kRbStages * (size_t)kRbCTile + kRbHalf;
  rp.nstage = rsmem + kRbHalf <= 226 * 1024 ? 2 : 1;
  rsmem += (size_t)(rp.nstage - 1) * kRbHalf;
  static std::atomic<int> rb_smem_set[64];
  cudaError_t e = smem_limit_once(recon_kernel, 226 * 1024, pl->device, rb_smem_set);
  if (e != cudaSuccess) return e;
  e = launch_pdl(recon_kernel, dim3(std::min(rp.nitems, std::max(1, pl->sm_count))), dim3(kRbThreads), rsmem, st,
                 ghmap, glmap, wmap, rp);
  if (e != cudaSuccess) return e;
  DenseParams dp;
  dp.alpha = alpha; dp.y = y;
  dp.rec = rp.rec;
  dp.call = call_tag(next_call_number());
  dp.M = M; dp.N = g.n_out; dp.nks = g.k_in / kBK;
  dp.bn = sh.bn;
  dp.ngroups = sh.ngroups;
  dp.nfull = sh.nfull;
  if (sh.wt == 2) {
    e = cudaFuncSetAttribute(dense_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, DnShape<2>::kSmem);
    if (e != cudaSuccess) return e;
    return launch_pdl(dense_kernel<2>, dim3(2 * sh.pairs), dim3(kDnThreads), (size_t)DnShape<2>::kSmem, st, wmap, xmap, dp);
  }
  e = cudaFuncSetAttribute(dense_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, DnShape<1>::kSmem);
  if (e != cudaSuccess) return e;
  return launch_pdl(dense_kernel<1>, dim3(2 * sh.pairs), dim3(kDnThreads), (size_t)DnShape<1>::kSmem, st, wmap, xmap, dp);
}

}  // namespace sdq
