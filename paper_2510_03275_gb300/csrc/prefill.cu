// K5: prefill contraction (M > 64, and the larger decode batches) on the 5th-generation tensor cores.
//
//   y[m, r] = alpha_r * sum_j c[r, j] * x_tilde[m, j]        (section 3.5, eq. 12)
//
// A dense contraction over K_eff = OSR * K, run transposed as a bf16 GEMM
// with fp32 accumulation, D[r, m] = sum_j c[r, j] x_tilde[m, j]: the codes
// are the A operand in tensor memory, expanded from the packed 2-bit / 1-bit
// words to exact bf16 +-2.0 / 0 straight from registers by tcgen05.st (they
// never occupy shared memory: expanded into a shared-memory tile, their
// writes and the MMA's reads of them held the tensor pipe to ~60 %), and
// x_tilde (M x K_eff bf16, written by the prepare kernel in the permuted
// 64-code stage order the expansion yields) is the B operand, loaded by TMA
// in the canonical K-major 128-byte-swizzled layout.
//
// CTA tile 128 code rows (M of the MMA = TMEM lanes) x `bn` batch rows (N, a
// multiple of 16 up to 256: the batch in equal tiles), 64 codes per pipeline
// stage; a cluster of S CTAs splits K, and the sum of its S accumulators goes
// through distributed shared memory in CTA order (the same bits every run):
//   warp 0      TMEM allocation; the TMA loads of the stages' x_tilde tiles
//   warp 1      issues tcgen05.mma (4 x K = 16 per stage, A from the
//               stage's TMEM slot), commits to the stage's "empty" barrier,
//               finally to the accumulator one
//   warps 2..9  two expander sets (set x expands the stages of parity x),
//               thread = code row: its 64 codes become 32 TMEM columns of
//               bf16 pairs (one x32 store); then the epilogue: accumulator
//               column m -> y[m, r] scaled by alpha_r / 2, each warp one lane
//               quadrant and half of the columns
//   warp 10     streams the codes, 4 stages (tiled layout: 4 slabs of
//               128 rows x 64 codes, contiguous) per bulk copy, into a ring
//               of its own that runs ahead of the x_tilde stages: codes come
//               from HBM, x_tilde from the L2
// TMEM: accumulator columns 0 .. bn - 1, A slot s at bn + 32 s; 256 columns
// and two CTAs per SM for bn up to 128 (one CTA's prologue and epilogue then
// run beside the other's MMAs), else 512 and one.
// At M = 201 on the LLaMA-7B linears (4096 x 8192 codes, 32 row tiles): 52 us
// as one 256-row tile per 128 x K, 15 us with S = 4 and 208 columns; 12288
// rows 53 -> 34, 22016 rows 103 -> 64, 4096 x 22016 codes 125 -> 27.  Two
// things bound the stages: an issuing thread needs its operands in uniform
// registers (warp_index, *_warp: 630 -> 360 cycles a stage), and the two
// expander sets take about 350 cycles per stage, so that below 160 batch rows
// per tile the expansion and not the tensor core is the limit.
// Every wait on an mbarrier is bounded (about 2 s); a timeout writes the call
// number into the workspace's call record and the CTA waits (again bounded)
// for its own copies and MMAs before it frees TMEM and ends.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"

namespace sdq {

namespace {

constexpr int kBM = 128, kBK = 64;
constexpr int kCodeStages = 4;            // stages per code copy
constexpr int kCodeSlots = 4;             // code ring
constexpr int kCSlab = kBM * 16;          // packed codes of a stage: 128 rows x 64 codes, at most 2 KB
constexpr int kCSlot = kCodeStages * kCSlab;
constexpr int kMaxStages = 6;             // x_tilde tiles and TMEM A slots
constexpr int kExpWarps = 8;
constexpr int kThreads = 32 * (3 + kExpWarps);   // 2 control warps, 8 expander / epilogue warps, the code stream
constexpr uint32_t kAslot = kBK / 2;      // TMEM columns per A slot (bf16 pairs)
constexpr int kMaxSplit = 8;              // k chunks (portable cluster size)
constexpr int kSmemSm = 227 * 1024;       // shared memory of an SM that blocks can have

struct PrefillParams {
  const uint32_t* codes;
  const float* alpha;
  float* y;
  uint64_t* rec;       // call record
  uint64_t call;
  int M, N, ngroups, wpg, nks, quantizer;
  int bn, stages, split, early, add;   // add: y += the result
};

// 16 bytes of the shared memory of the cluster's CTA `rank`, at this CTA's address `a`.
__device__ __forceinline__ float4 ld_cluster4(uint32_t a, uint32_t rank) {
  uint32_t r;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];\n"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(r) : "memory");
  return v;
}

__global__ void __launch_bounds__(kThreads, 2)
    prefill_kernel(const __grid_constant__ CUtensorMap xmap, PrefillParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t x_full[kMaxStages], empty[kMaxStages], a_full[kMaxStages], c_full[kCodeSlots],
      c_empty[kCodeSlots], acc_bar;
  __shared__ uint32_t tmem_base;

  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int tile = blockIdx.x, n0 = tile * kBM, m0 = blockIdx.y * p.bn, z = blockIdx.z;
  const int kb = (int)((int64_t)p.nks * z / p.split), nst = (int)((int64_t)p.nks * (z + 1) / p.split) - kb;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base = smem_raw + (sbase - smem_u32(smem_raw));
  const uint32_t xtile = (uint32_t)p.bn * 128u;           // bn batch rows x 64 codes of bf16 x_tilde
  uint8_t* c_ring = base + p.stages * xtile;
  const uint32_t slab_bytes = (uint32_t)(kTileRows * p.wpg * 4);
  const uint32_t tcols = p.bn <= 128 ? 256u : 512u;

  if (tid == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(&x_full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&a_full[s], 4);
    }
    for (int s = 0; s < kCodeSlots; ++s) {
      mbar_init(&c_full[s], 1);
      mbar_init(&c_empty[s], kExpWarps);
    }
    mbar_init(&acc_bar, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(&tmem_base, tcols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // with `early` the codes (which the preceding grid does not write) start at once
  if (!(p.early && warp == 2 + kExpWarps)) pdl_wait();
  pdl_launch_dependents();
  call_record_start_prepared(p.rec, p.call, blockIdx.x == 0 && blockIdx.y == 0 && z == 0 && tid == 0);
  const uint32_t tmem = tmem_base;
  const uint32_t acol = tmem + (uint32_t)p.bn;
  bool ok = true;

  if (warp == 0) {
    // x_tilde tile [m0, m0 + bn) x [64 k, 64 k + 64) (rows past M read as zeros)
    int s = 0, r = 0, i = 0;
    for (; i < nst; ++i) {
      if (r > 0) ok = mbar_wait_warp(&empty[s], (r - 1) & 1);
      if (!ok) break;
      mbar_expect_tx_warp(&x_full[s], xtile);
      tma_load_2d_warp(base + s * xtile, &xmap, (kb + i) * kBK, m0, &x_full[s]);
      if (++s == p.stages) { s = 0; ++r; }
    }
    // every copy issued has landed before the CTA ends
    for (int j = max(0, i - p.stages); j < i; ++j)
      if (!mbar_wait_warp(&x_full[j % p.stages], (j / p.stages) & 1)) ok = false;
  } else if (warp == 1) {
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.bn >> 3) << 17) |
                           ((uint32_t)(kBM >> 4) << 24);   // D fp32, A and B bf16, both K-major
    const uint64_t bd0 = sw128_desc(sbase);
    int s = 0, r = 0;
    for (int i = 0; i < nst; ++i) {
      ok = mbar_wait_warp(&x_full[s], r & 1) && mbar_wait_warp(&a_full[s], r & 1);
      if (!ok) break;
      tc_fence_after();
      const uint64_t bd = bd0 + (uint64_t)((uint32_t)s * xtile >> 4);
#pragma unroll
      for (int kk = 0; kk < kBK / 16; ++kk)
        umma_bf16_ts_warp(tmem, acol + kAslot * s + 8 * kk, bd + 2 * kk, idesc, (i | kk) != 0);
      umma_commit_warp(&empty[s]);
      if (++s == p.stages) { s = 0; ++r; }
    }
    umma_commit_warp(&acc_bar);
    if (!mbar_wait_warp(&acc_bar, 0)) ok = false;
  } else if (warp == 2 + kExpWarps) {
    const uint64_t pol = l2_policy_evict_first();
    const uint8_t* src = reinterpret_cast<const uint8_t*>(p.codes) +
                         ((size_t)tile * p.ngroups + kb) * slab_bytes;
    const int ng = (nst + kCodeStages - 1) / kCodeStages;
    int g = 0;
    for (; g < ng; ++g) {
      const int s = g % kCodeSlots, r = g / kCodeSlots;
      if (r > 0) ok = mbar_wait_warp(&c_empty[s], (r - 1) & 1);
      if (!ok) break;
      const uint32_t bytes = (uint32_t)min(kCodeStages, nst - kCodeStages * g) * slab_bytes;
      mbar_expect_tx_warp(&c_full[s], bytes);
      if (p.M <= p.bn) bulk_g2s_hint_warp(c_ring + s * kCSlot, src, bytes, &c_full[s], pol);   // codes read once
      else bulk_g2s_warp(c_ring + s * kCSlot, src, bytes, &c_full[s]);
      src += kCodeStages * slab_bytes;
    }
    if (p.early) pdl_wait();
    for (int j = max(0, g - kCodeSlots); j < g; ++j)
      if (!mbar_wait_warp(&c_full[j % kCodeSlots], (j / kCodeSlots) & 1)) ok = false;
  } else {
    // Expanders: set x = (warp - 2) / 4 expands stages i = x (mod 2); the
    // thread of lane quadrant q = warp % 4 expands code row 32 q + lane.
    const int x = (warp - 2) >> 2, q = warp & 3, rr = 32 * q + lane;
    const uint32_t lane_addr = (uint32_t)(32 * q) << 16;
    int s = x, r = 0;   // stage slot and round (stages is even)
    for (int i = x; i < nst; i += 2) {
      const int g = i / kCodeStages, cs = g % kCodeSlots;
      ok = mbar_wait(&c_full[cs], (g / kCodeSlots) & 1);          // the codes have landed
      if (ok && r > 0) ok = mbar_wait(&empty[s], (r - 1) & 1);   // TMEM slot s: its MMAs are done
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint8_t* slab = c_ring + cs * kCSlot + (i % kCodeStages) * slab_bytes;
      uint32_t v[32];
      if (p.quantizer == SDQ_TERNARY) {
        // 16 codes per word, code 2 bits: (w << 2 j) & 0xC000C000 puts two
        // codes into the sign and exponent-MSB bits of a bf16 pair (+-2 / 0)
        const uint4 w4 = *reinterpret_cast<const uint4*>(slab + rr * 16);
        const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int j = 0; j < 8; ++j) v[8 * k + j] = (w[k] << (2 * j)) & 0xC000C000u;
      } else {   // words hold the inverted bits: 1 = -1
        const uint2 w2 = *reinterpret_cast<const uint2*>(slab + rr * 8);
        const uint32_t w[2] = {~w2.x, ~w2.y};
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int j = 0; j < 16; ++j) v[16 * k + j] = ((w[k] << j) & 0x80008000u) | 0x40004000u;
      }
      // this warp's last stage of the code slot: the slot goes back
      if (i + 2 >= min(nst, kCodeStages * (g + 1))) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&c_empty[cs]);
      }
      tmem_st32(acol + lane_addr + kAslot * s, v);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&a_full[s]);
      s += 2;
      if (s >= p.stages) { s -= p.stages; ++r; }
    }
    // Epilogue: TMEM lane quadrant q holds code rows n0 + 32 q + lane; this
    // warp takes half of the accumulator columns (batch rows).
    if (ok) ok = mbar_wait(&acc_bar, 0);
    ok = __all_sync(0xffffffffu, ok);
    tc_fence_after();
    if (ok) {
      const int row = n0 + rr, half = (p.bn / 16 + 1) / 2 * 16;
      const int mv = min(p.bn, p.M - m0), c1 = x ? mv : min(half, mv);
      const float sa = p.split == 1 && row < p.N ? 0.5f * __ldg(p.alpha + row) : 0.f;
      float* part = reinterpret_cast<float*>(base) + rr;   // [column][code row], over the drained x_tilde tiles
      for (int c0 = x ? half : 0; c0 < c1; c0 += 16) {
        uint32_t a[16];
        tmem_ld16(tmem + lane_addr + (uint32_t)c0, a);
        tmem_ld_wait();
        if (p.split > 1) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (c0 + i < c1) part[(c0 + i) * kBM] = __uint_as_float(a[i]);
        } else if (row < p.N) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (c0 + i < c1) {
              float* o = p.y + (size_t)(m0 + c0 + i) * p.N + row;
              if (p.add) red_add_f32(o, __uint_as_float(a[i]) * sa);
              else *o = __uint_as_float(a[i]) * sa;
            }
        }
      }
    }
  }
  if (!ok) call_record_fail(p.rec, p.call);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, tcols);
  }
  if (p.split == 1) return;
  // The cluster's partial sums, in CTA order: CTA z adds columns z, z + S, ...
  // of all S accumulators, a warp one column (128 code rows) at a time.
  cluster_sync();
  {
    const int mv = min(p.bn, p.M - m0), row = n0 + 4 * lane;
    float al[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) al[i] = row + i < p.N ? 0.5f * __ldg(p.alpha + row + i) : 0.f;
    const bool vec = (p.N & 3) == 0 && row + 3 < p.N;
    for (int c = z + p.split * warp; c < mv; c += p.split * (kThreads / 32)) {
      const uint32_t a = sbase + (uint32_t)(c * kBM + 4 * lane) * 4u;
      float4 v[kMaxSplit];
#pragma unroll
      for (int i = 0; i < kMaxSplit; ++i)
        if (i < p.split) v[i] = ld_cluster4(a, (uint32_t)i);
      float4 t = v[0];
#pragma unroll
      for (int i = 1; i < kMaxSplit; ++i)
        if (i < p.split) { t.x += v[i].x; t.y += v[i].y; t.z += v[i].z; t.w += v[i].w; }
      float* o = p.y + (size_t)(m0 + c) * p.N + row;
      t = make_float4(t.x * al[0], t.y * al[1], t.z * al[2], t.w * al[3]);
      if (vec && !p.add) {
        *reinterpret_cast<float4*>(o) = t;
      } else {
        const float tv[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (row + i < p.N) {
            if (p.add) red_add_f32(o + i, tv[i]);
            else o[i] = tv[i];
          }
      }
    }
  }
  cluster_sync();   // no CTA ends while its accumulator is being read
}

// Launch shape at batch M: the batch in equal tiles of bn rows, S k chunks.
// Time model in ns, fitted to forced splits of LLaMA-7B linears at M = 65 ..
// 500 (within ~10 % of them): a stage takes its MMAs (1.09 bn, one CTA per
// SM) or its code expansion (165 + bn / 4 alone on an SM, 230 + 0.7 bn with
// two CTAs there); a CTA adds a prologue and an epilogue, a split one the
// cluster's sum.  CTAs run in waves of what the device holds of such
// clusters; with two per SM the last wave overlaps the one before.
struct PrefillShape {
  int bn, mt, stages, split, smem;
};
constexpr int kFixedSmem = 1024 + kCodeSlots * kCSlot;
PrefillShape prefill_shape(const sdq_plan_s* pl, int M) {
  const Geometry& g = pl->geo;
  PrefillShape s{};
  s.mt = (M + 255) / 256;
  s.bn = ((M + s.mt - 1) / s.mt + 15) / 16 * 16;
  const int occ = s.bn <= 128 ? 2 : 1;
  const int by_smem = (kSmemSm / occ - 1024 - kFixedSmem) / (s.bn * 128);   // 1 KB a block for the static part
  const int by_tmem = ((occ == 2 ? 256 : 512) - s.bn) / (int)kAslot;
  s.stages = std::min(kMaxStages, std::min(by_smem, by_tmem)) & ~1;
  const int64_t nks = g.k_eff_pad / kBK, tiles = (int64_t)g.ntiles * s.mt;
  double best = 0;
  for (int S = 1; S <= kMaxSplit && S <= nks; ++S) {
    const int64_t held = (int64_t)occ * std::max(1, pl->pf_clusters[S]);
    const double x = (double)tiles / held, up = (double)((tiles + held - 1) / held);
    const double waves = occ == 2 ? std::max(1.0, 0.5 * (x + up)) : up;
    const bool shared = occ == 2 && tiles * S > pl->sm_count;
    const double stage = std::max(1.09 * s.bn, shared ? 230.0 + 0.7 * s.bn : 165.0 + 0.25 * s.bn);
    const double t = waves * ((S == 1 ? 4100.0 : 5900.0 + 400.0 * S) + (double)((nks + S - 1) / S) * stage);
    if (S == 1 || t < best * 0.98) {
      best = t;
      s.split = S;
    }
  }
  s.smem = kFixedSmem + std::max(s.stages * s.bn * 128, s.split > 1 ? s.bn * kBM * 4 - kCodeSlots * kCSlot : 0);
  // a grid that fits one CTA per SM asks for more than half an SM: launched
  // early, CTAs would pair up on the first SMs that the prepare kernel leaves
  // (4096 x 22016 codes at M = 65: 33 us against 22 spread out)
  if (occ == 2 && tiles <= pl->pf_clusters[s.split]) s.smem = std::max(s.smem, kSmemSm / 2 + 4096);
  return s;
}
constexpr int kPfSmemLimit = kSmemSm - 1024;

void prefill_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, dim3 grid, int smem, cudaStream_t st) {
  *cfg = {};
  cfg->gridDim = grid;
  cfg->blockDim = dim3(kThreads);
  cfg->dynamicSmemBytes = (size_t)smem;
  cfg->stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = grid.z;
  cfg->attrs = attr;
  cfg->numAttrs = grid.z > 1 ? 2 : 1;
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  });
  return fn;
}

cudaError_t prefill_smem_limit(int device) {
  static std::atomic<int> smem_set[64];   // per device: limit raised to the largest shape's
  return smem_limit_once(prefill_kernel, kPfSmemLimit, device, smem_set);
}

// ------------------------------------------ prefill prepare, tensor cores
// x_tilde = G x_b for every block b (section 3.5), as one GEMM: x viewed as
// R = M nblk rows of B inputs (row r = block r mod nblk of batch row r /
// nblk), x_tilde rows = x rows . G^T (B x n_b), on tcgen05.mma kind::f16 (M =
// 128 rows, N = ncol, K = 16 per instruction) with G split into bf16 hi and lo
// parts accumulated into the same fp32 accumulator (the pair carries G to
// ~2^-16; x is bf16, exact).  A CTA keeps the hi and lo parts of ncol of
// the n_b columns (grid.y: which) and walks tiles of 128 rows (grid.x):
//   warp 0     TMEM allocation (two accumulators of ncol columns); loads its
//              part of G once, then the x tiles by 64-wide K chunks into a
//              ring (TMA, 128-byte swizzle: the canonical K-major operand)
//   warp 1     issues each tile's B / 8 MMAs into accumulator t mod 2
//   warps 2-9  epilogue, two warps per TMEM lane quadrant (half of the ncol
//              columns each): bf16 x_tilde (round to nearest even) in the
//              prefill operand order (prefill_pos64) with 16-byte stores;
//              the K padding of every batch row set to zero
// Large batches write 2 M K_eff bytes and are bound by that (ncol as large as
// fits); small ones by the chain of one tile, so they take ncol = 64: four
// times the CTAs at OSR 2, each loading a quarter of G (M = 201 on 4096
// inputs: 6.3 -> 4.6 us, M = 65: 6.2 -> 3.3).  Bounded waits as in the contraction kernels.
constexpr int kPtEpiWarps = 8;
constexpr int kPtThreads = 64 + 32 * kPtEpiWarps;
constexpr int kPtRows = 128;
constexpr int kPtChunk = kPtRows * 64 * 2;    // 16 KB: 128 rows x 64 bf16
constexpr int kPtMaxSlots = 6;
constexpr int kPtSmem = 226 * 1024;

struct PrepTcParams {
  uint16_t* xtb;
  float* xt;         // x_tilde in fp32 too, natural order (null: not)
  uint64_t* rec;
  uint64_t call;
  int64_t R, k_eff, kpad;
  int M, nblk, n_b, ntile, ternary;
  int ncol, nch, slots;   // columns per CTA, 64-wide K chunks (B / 64), ring slots
};

__global__ void __launch_bounds__(kPtThreads, 1)
    prep_tc_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap ghmap,
                   const __grid_constant__ CUtensorMap glmap, PrepTcParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t g_full, x_full[kPtMaxSlots], x_empty[kPtMaxSlots], acc_full[2], acc_empty[2],
      mma_done;
  __shared__ uint32_t tmem_base;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31, j0 = (int)blockIdx.y * p.ncol;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base = smem_raw + (sbase - smem_u32(smem_raw));
  const uint32_t gchunk = (uint32_t)p.ncol * 128u;  // one 64-wide K chunk of G^T: ncol rows x 128 B
  uint8_t* gl = base + p.nch * gchunk;              // (hi chunks first)
  const uint32_t xoff = 2u * p.nch * gchunk;        // then the ring
  const uint32_t tcols = p.ncol <= 64 ? 128u : (p.ncol <= 128 ? 256u : 512u);

  if (tid == 0) {
    mbar_init(&g_full, 1);
    mbar_init(&mma_done, 1);
    for (int s = 0; s < kPtMaxSlots; ++s) {
      mbar_init(&x_full[s], 1);
      mbar_init(&x_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&acc_full[s], 1);
      mbar_init(&acc_empty[s], kPtEpiWarps);
    }
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(&tmem_base, tcols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  bool ok = true;

  if (warp == 0) {
    // G (the plan's table, never written by the stream) before the wait
    // for the preceding grid; x and the workspace after it
    mbar_expect_tx_warp(&g_full, 2u * p.nch * gchunk);
    for (int c = 0; c < p.nch; ++c) {
      tma_load_2d_warp(base + c * gchunk, &ghmap, 64 * c, j0, &g_full);
      tma_load_2d_warp(gl + c * gchunk, &glmap, 64 * c, j0, &g_full);
    }
    pdl_wait();
    pdl_launch_dependents();
    int s = 0, r = 0, n = 0;
    for (int t = blockIdx.x; t < p.ntile && ok; t += gridDim.x)
      for (int c = 0; c < p.nch && ok; ++c) {
        if (r > 0) ok = mbar_wait_warp(&x_empty[s], (r - 1) & 1);
        if (!ok) break;
        mbar_expect_tx_warp(&x_full[s], kPtChunk);
        tma_load_2d_warp(base + xoff + s * kPtChunk, &xmap, 64 * c, t * kPtRows, &x_full[s]);
        ++n;
        if (++s == p.slots) { s = 0; ++r; }
      }
    // every copy issued has landed before the CTA ends
    if (!mbar_wait_warp(&g_full, 0)) ok = false;
    for (int i = max(0, n - p.slots); i < n; ++i)
      if (!mbar_wait_warp(&x_full[i % p.slots], (i / p.slots) & 1)) ok = false;
  } else if (warp == 1) {
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.ncol >> 3) << 17) |
                           ((uint32_t)(kPtRows >> 4) << 24);
    ok = mbar_wait_warp(&g_full, 0);
    const uint64_t gd = sw128_desc(sbase), xd = sw128_desc(sbase + xoff);
    const uint32_t gstep = gchunk >> 4;
    int i = 0, s = 0, r = 0;
    for (int t = blockIdx.x; t < p.ntile && ok; t += gridDim.x, ++i) {
      const int a = i & 1, ra = i >> 1;
      if (ra > 0) ok = mbar_wait_warp(&acc_empty[a], (ra - 1) & 1);
      const uint32_t d = tmem + (uint32_t)(a * p.ncol);
      for (int c = 0; c < p.nch && ok; ++c) {
        ok = mbar_wait_warp(&x_full[s], r & 1);
        if (!ok) break;
        tc_fence_after();
        const uint64_t ad = xd + (uint64_t)(s * (kPtChunk >> 4));
        const uint64_t bh = gd + (uint64_t)(c * gstep), bl = gd + (uint64_t)((p.nch + c) * gstep);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          umma_bf16_warp(d, ad + 2 * kk, bh + 2 * kk, idesc, (c | kk) != 0);
          umma_bf16_warp(d, ad + 2 * kk, bl + 2 * kk, idesc, 1);
        }
        umma_commit_warp(&x_empty[s]);
        if (++s == p.slots) { s = 0; ++r; }
      }
      if (ok) umma_commit_warp(&acc_full[a]);
    }
    umma_commit_warp(&mma_done);   // every MMA is done before TMEM is freed
    if (!mbar_wait_warp(&mma_done, 0)) ok = false;
  } else {
    pdl_wait();   // the workspace belongs to the preceding grid until then
    prep_record_start(p.rec, p.call, blockIdx.x == 0 && blockIdx.y == 0 && tid == 64);
    const int et = tid - 64, q = warp & 3, half = (warp - 2) >> 2;
    // the K padding of every batch row (k_eff .. kpad, a multiple of 8; by
    // the CTAs of the first columns)
    if (j0 == 0)
      for (int64_t z = (int64_t)blockIdx.x * (32 * kPtEpiWarps) + et; z < (int64_t)p.M * ((p.kpad - p.k_eff) / 8);
           z += (int64_t)gridDim.x * (32 * kPtEpiWarps)) {
        const int64_t per = (p.kpad - p.k_eff) / 8, m = z / per;
        const int64_t at = m * p.kpad + p.k_eff + 8 * (z - m * per);
        *reinterpret_cast<uint4*>(p.xtb + at) = make_uint4(0, 0, 0, 0);
        if (p.xt) {
          *reinterpret_cast<uint4*>(p.xt + at) = make_uint4(0, 0, 0, 0);
          *reinterpret_cast<uint4*>(p.xt + at + 4) = make_uint4(0, 0, 0, 0);
        }
      }
    const int cw = p.ncol / 2;                                  // this warp's columns
    const uint32_t lq = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(half * cw);
    int i = 0;
    for (int t = blockIdx.x; t < p.ntile && ok; t += gridDim.x, ++i) {
      const int s = i & 1, r = i >> 1;
      ok = mbar_wait_warp(&acc_full[s], r & 1);
      if (!ok) break;
      tc_fence_after();
      const int64_t row = (int64_t)t * kPtRows + 32 * q + lane;
      const bool live = row < p.R;
      const int64_t m = live ? row / p.nblk : 0;
      const int64_t at = m * p.kpad + (live ? (row - m * p.nblk) * p.n_b : 0) + j0 + half * cw;
      uint16_t* out = p.xtb + at;
      const uint32_t acol = (uint32_t)(s * p.ncol);
      // 32 columns at a time: a ternary operand permutes within 16, a binary
      // one within 32 positions (prefill_pos64); physical pair (2k, 2k + 1)
      // of a 16 (32) holds logical 7 - k and 15 - k (15 - k and 31 - k)
      for (int c0 = 0; c0 < cw; c0 += 32) {
        uint32_t a[16], b[16];
        tmem_ld16(lq + acol + (uint32_t)c0, a);
        tmem_ld16(lq + acol + (uint32_t)c0 + 16, b);
        tmem_ld_wait();
        if (c0 + 32 >= cw) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[s]);
        }
        uint32_t w[16];
        if (p.ternary) {
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            w[k] = pack_bf16x2(__uint_as_float(a[7 - k]), __uint_as_float(a[15 - k]));
            w[8 + k] = pack_bf16x2(__uint_as_float(b[7 - k]), __uint_as_float(b[15 - k]));
          }
        } else {
#pragma unroll
          for (int k = 0; k < 16; ++k)
            w[k] = pack_bf16x2(__uint_as_float(a[15 - k]), __uint_as_float(b[15 - k]));
        }
        if (live) {
          // whole 32-byte sectors, every lane has a row of its own (7B layer, M =
          // 64: 112.5 us with 16-byte stores, 109.1 so); the workspace is 256-byte
          // aligned, columns come in multiples of 32
          st_global32(out + c0, w);
          st_global32(out + c0 + 16, w + 8);
          if (p.xt) {
            float* f = p.xt + at + c0;
            st_global32(f, a);
            st_global32(f + 8, a + 8);
            st_global32(f + 16, b);
            st_global32(f + 24, b + 8);
          }
        }
      }
    }
  }
  if (!ok) prep_record_fail(p.rec, p.call);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, tcols);
  }
}

}  // namespace

void* tensor_map_encoder() { return reinterpret_cast<void*>(encode_fn()); }

cudaError_t launch_prefill(const sdq_plan_s* pl, const uint32_t* codes, const float* alpha, int M,
                           float* y, void* ws, cudaStream_t st, int early, int y_mode) {
  const Geometry& g = pl->geo;
  const WsLayout L = workspace_layout(pl, M);
  uint8_t* wbase = static_cast<uint8_t*>(ws);
  auto enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const PrefillShape sh = prefill_shape(pl, M);
  CUtensorMap xmap;
  const cuuint64_t dims[2] = {(cuuint64_t)g.k_eff_pad, (cuuint64_t)M};
  const cuuint64_t strides[1] = {(cuuint64_t)g.k_eff_pad * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)sh.bn};
  const cuuint32_t estr[2] = {1, 1};
  CUresult cr = enc(&xmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, wbase + L.xtb, dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (cr != CUDA_SUCCESS) return cudaErrorInvalidValue;
  PrefillParams p;
  p.codes = codes; p.alpha = alpha; p.y = y;
  p.rec = reinterpret_cast<uint64_t*>(wbase + L.err);
  p.call = call_tag(next_call_number());
  p.M = M; p.N = g.n_out; p.ngroups = g.ngroups; p.wpg = g.wpg;
  p.nks = (int)(g.k_eff_pad / kBK);
  p.quantizer = pl->desc.quantizer;
  p.bn = sh.bn; p.stages = sh.stages; p.split = sh.split; p.early = early; p.add = y_mode == kYAdd;
  cudaError_t e = prefill_smem_limit(pl->device);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  prefill_config(&cfg, attr, dim3(g.ntiles, sh.mt, sh.split), sh.smem, st);
  return cudaLaunchKernelEx(&cfg, prefill_kernel, xmap, p);
}

// Clusters of S CTAs, one CTA per SM, that the device holds at once (GPCs of
// different sizes leave SMs over: asked, not computed).
cudaError_t prefill_occupancy(sdq_plan_s* pl) {
  cudaError_t e = prefill_smem_limit(pl->device);
  pl->pf_clusters[1] = pl->sm_count;
  for (int S = 2; S <= kMaxSplit && e == cudaSuccess; ++S) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    prefill_config(&cfg, attr, dim3(1, 1, S), kPfSmemLimit - 1024, 0);
    cfg.attrs = attr + 1;   // the cluster alone
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&pl->pf_clusters[S], prefill_kernel, &cfg);
  }
  return e;
}

static bool prep_tc_takes(const Geometry& g) { return g.block >= 64 && g.block <= 512 && g.n_b % 64 == 0; }
// us a forward call at OSR 2, B = 128, ternary (4-bit decode kernel / this one):
//   4096 x 4096    M = 24 11.8 / 13.4   M = 40 13.2 / 13.8   M = 44 14.7 / 13.7
//   22016 x 4096   M = 40 30.9 / 37.3   M = 48 34.4 / 37.6   M = 56 41.8 / 38.3
//   57344 x 8192   M = 48  113 / 120    M = 56  122 / 121    M = 64  125 / 122
// Binary codes, B = 64 and OSR 3/2 and 3 cross within 12 rows of these or stay
// with the decode kernel (57344 x 8192 binary, M = 64: 127 / 133), 1024 x 1024
// crosses at 64; B = 512 crosses lower (4096 x 4096 from M = 16, 22016 x 4096 at
// 32, 57344 x 8192 at 44).  The lines were drawn when the decode kernel took 16.1
// us for the first of these and 42.8 for 22016 x 4096 at M = 40, before its launch
// shapes were fitted anew.  They stay below the crossings because this kernel's
// operand is the closer one, bf16 x_tilde against three e2m1 terms (error against
// 64 bits 1.7e-3 and 2.0e-3): at most 1.5x of a call's time is given for it (binary
// 12288 x 4096, OSR 3, M = 40: 25 / 38 us).  This kernel's time is nearly flat in M:
// the expanded codes' stores into tensor memory (16 KB per 2 KB of codes) bound it,
// about 290 cycles a stage and SM.
int wide_min_batch(const sdq_plan_s* pl) {
  const Geometry& g = pl->geo;
  if (!prep_tc_takes(g) || !encode_fn()) return kMaxDecodeM + 1;
  const int64_t codes = (int64_t)g.n_out * g.k_eff;
  return codes <= 40000000 ? 24 : (codes <= 200000000 ? 40 : 56);
}

// The prefill prepare kernel on the tensor cores where it applies (B = 64 ..
// 512, n_b a multiple of 64, x 16-byte aligned); *used = false otherwise.
cudaError_t launch_prep_tc(const sdq_plan_s* pl, const uint16_t* x, int M, void* ws, cudaStream_t st,
                           bool* used, bool fp32_too) {
  const Geometry& g = pl->geo;
  *used = false;
  if (!prep_tc_takes(g) || (reinterpret_cast<uintptr_t>(x) & 15u)) return cudaSuccess;
  auto enc = encode_fn();
  if (!enc) return cudaSuccess;
  const WsLayout L = workspace_layout(pl, M);
  uint8_t* wbase = static_cast<uint8_t*>(ws);
  const int64_t R = (int64_t)M * g.nblk;
  if (R >= (int64_t(1) << 31) - kPtRows) return cudaSuccess;
  PrepTcParams p;
  p.xtb = reinterpret_cast<uint16_t*>(wbase + L.xtb);
  p.xt = fp32_too ? reinterpret_cast<float*>(wbase + L.xt) : nullptr;
  p.rec = reinterpret_cast<uint64_t*>(wbase + L.err);
  p.call = call_tag(next_call_number());
  p.R = R; p.k_eff = g.k_eff; p.kpad = g.k_eff_pad;
  p.M = M; p.nblk = g.nblk; p.n_b = g.n_b; p.ternary = pl->desc.quantizer == SDQ_TERNARY;
  p.ntile = (int)((R + kPtRows - 1) / kPtRows);
  p.nch = g.block / 64;
  // the most columns per CTA (64 .. 256, dividing n_b, with two ring slots
  // beside them) that still give every SM a CTA, else 64
  const int64_t sms = std::max(1, pl->sm_count);
  p.ncol = 64;
  for (int c = 128; c <= 256; c += 64)
    if (g.n_b % c == 0 && 1024 + 256 * p.nch * c + 2 * kPtChunk <= kPtSmem && p.ntile * (int64_t)(g.n_b / c) >= sms)
      p.ncol = c;
  const int gbytes = 256 * p.nch * p.ncol;
  // two CTAs per SM where their parts of G leave room
  const bool two = 2 * (2048 + gbytes + 4 * kPtChunk) <= kPtSmem;
  p.slots = two ? 4 : std::min(kPtMaxSlots, (kPtSmem - 1024 - gbytes) / kPtChunk);
  const int parts = g.n_b / p.ncol;
  CUtensorMap xmap, ghmap, glmap;
  const cuuint32_t estr[2] = {1, 1};
  const cuuint64_t strides[1] = {(cuuint64_t)g.block * 2};
  auto map = [&](CUtensorMap* m, const uint16_t* ptr, int64_t rows, int box_rows) {
    const cuuint64_t dims[2] = {(cuuint64_t)g.block, (cuuint64_t)rows};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  if (!map(&xmap, x, R, kPtRows) || !map(&ghmap, pl->d_g_hi, g.n_b, p.ncol) || !map(&glmap, pl->d_g_lo, g.n_b, p.ncol))
    return cudaSuccess;
  static std::atomic<int> smem_set[64];
  cudaError_t e = smem_limit_once(prep_tc_kernel, kPtSmem, pl->device, smem_set);
  if (e != cudaSuccess) return e;
  *used = true;
  const int64_t ctas = sms * (two ? 2 : 1);
  const int gx = (int)std::min<int64_t>(p.ntile, std::max<int64_t>(1, (ctas + parts - 1) / parts));
  return launch_pdl(prep_tc_kernel, dim3(gx, parts), dim3(kPtThreads),
                    (size_t)(1024 + gbytes + p.slots * kPtChunk), st, xmap, ghmap, glmap, p);
}
}  // namespace sdq
