// Base-3 storage of ternary codes: 5 trits per byte (1.6 bits per code, the
// closest byte-aligned rate to eq. (14)'s log2(3) = 1.58 bits).
//
// Row r of the base-3 layout starts at byte r * bpr, bpr = ceil(K_eff / 5)
// rounded up to a multiple of 16; code j is trit t = code mod 3 (0, +1 -> 1,
// -1 -> 2) at digit j mod 5 of byte j / 5 (byte = sum_d t_d 3^d <= 242).
// Both kernels move 80 codes per thread: 16 base-3 bytes <-> 5 plain-layout
// words (16 two-bit fields each), one table look-up per byte.  The issue of
// the instructions around the look-ups bounds them, so the table (256 words)
// is kept once per lane: word i of lane l at 32 i + l, every lane in a bank
// of its own (a single copy had about 3.5 lanes per bank), its address one
// shift and one or two masks away from the data; computing the digits on two
// bytes at a time in 16-bit halves took twice as many instructions.  A warp
// takes 32 consecutive groups of 80 codes of one row, so that its plain words
// are 640 consecutive bytes, moved in 16-byte pieces through shared memory (5
// words a lane: an odd stride, no bank conflicts), and its base-3 bytes 512.
// Persistent blocks: the table is filled once, and a warp's next loads are in
// flight while it converts.  28672 x 16384 codes (211 MB in and out, 31 us at
// the copy rate): 45 us either way, from 82 us with one table per block and a
// word or byte group per thread.
#include <algorithm>

#include "common.cuh"

namespace sdq {

namespace {

constexpr int kCodesPerThread = 80;   // 16 bytes x 5 trits = 5 words x 16 fields
constexpr int kB3Threads = 256;
constexpr int kB3Warps = kB3Threads / 32;
constexpr int kB3Runs = 2;            // runs of 32 groups per warp and step
constexpr int kB3Words = 160;         // plain words of a run
constexpr int kB3Table = 256 * 32;    // table words: 256 per lane
constexpr int kB3Smem = 4 * (kB3Table + kB3Warps * kB3Runs * kB3Words);
constexpr int kB3BlocksPerSm = 4;     // 42 KB of shared memory each, 64 registers a thread

struct Base3Params {
  int n_out, wpr, bpr, gpr, rpr;   // plain words / base-3 bytes / groups / runs per row
  int srow, sseg;                  // a step in rows and runs: all warps' runs
  int64_t k_eff, total;            // total = n_out * rpr runs
};

// Five 2-bit fields -> their base-3 byte (the invalid field 10 reads as trit
// 0), and a byte -> its five fields (0 for the invalid bytes above 242).
__host__ __device__ __forceinline__ uint32_t fields_byte(uint32_t v) {
  uint32_t b = 0;
  for (int d = 4; d >= 0; --d) {
    const uint32_t f = (v >> (2 * d)) & 3u;
    b = 3u * b + ((f & 1u) ? (f >> 1) + 1u : 0u);
  }
  return b;
}
__host__ __device__ __forceinline__ uint32_t byte_fields(uint32_t x) {
  uint32_t f = 0;
  if (x < 243)
    for (int d = 0; d < 5; ++d) {
      const uint32_t t = x % 3u;
      f |= (t == 2 ? 3u : t) << (2 * d);
      x /= 3u;
    }
  return f;
}
// Bytes of 243 .. 255 in a word: bit 7 of each (set, and the low seven bits
// at least 115).
__host__ __device__ __forceinline__ uint32_t invalid_bytes(uint32_t x) {
  return x & ((x & 0x7F7F7F7Fu) + 0x0D0D0D0Du) & 0x80808080u;
}

// Word `threadIdx.x` of the table to all 32 lanes' copies (16-byte stores,
// the 8 of a thread in rotated order: no bank conflicts).
__device__ __forceinline__ void fill_table(uint32_t* table, uint32_t word) {
  uint4* row = reinterpret_cast<uint4*>(table + 32 * threadIdx.x);
#pragma unroll
  for (int j = 0; j < 8; ++j) row[(j + threadIdx.x) & 7] = make_uint4(word, word, word, word);
  __syncthreads();
}

// The fields of the word's codes first .. first + 15 that lie below K_eff.
__device__ __forceinline__ uint32_t below_k_eff(uint32_t w, int64_t first, int64_t k_eff) {
  const int64_t keep = k_eff - first;
  return keep >= 16 ? w : (keep <= 0 ? 0u : w & ((1u << (2 * keep)) - 1u));
}

// A warp's next kB3Runs runs: row and run within the row (past the last row:
// row 0, run rpr, which has nothing to read or write).  Stepped without a
// division: a 64-bit one per run was 50 of the 254 instructions a thread
// issued per 80 codes, which bound both kernels (52 us for the layer above, 45
// so).
struct RunPlace {
  uint32_t row;
  int seg;
  __device__ __forceinline__ RunPlace(const Base3Params& p, int64_t run0)
      : row((uint32_t)(run0 / p.rpr)), seg((int)(run0 - (int64_t)row * p.rpr)) {}
  __device__ __forceinline__ void place(const Base3Params& p, int u, uint32_t& r, int& sg) const {
    const bool wrap = seg + u >= p.rpr;   // u <= 1
    r = row + (wrap ? 1u : 0u);
    sg = seg + u - (wrap ? p.rpr : 0);
    if (r >= (uint32_t)p.n_out) {
      r = 0u;
      sg = p.rpr;
    }
  }
  __device__ __forceinline__ void next(const Base3Params& p) {
    row += (uint32_t)p.srow;
    seg += p.sseg;
    if (seg >= p.rpr) {
      seg -= p.rpr;
      ++row;
    }
  }
};
static_assert(kB3Runs == 2, "RunPlace wraps once");

// A warp's step is kB3Runs runs: a run is 32 groups (160 plain words, 512
// base-3 bytes) of one row, lane = group.  gpr = bpr / 16.
__global__ void __launch_bounds__(kB3Threads) pack_base3_kernel(const uint32_t* __restrict__ plain,
                                                                uint8_t* __restrict__ out, Base3Params p) {
  extern __shared__ __align__(16) uint32_t b3_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t(*stage)[kB3Words] = reinterpret_cast<uint32_t(*)[kB3Words]>(b3_smem + kB3Table) + kB3Runs * warp;
  const uint8_t* mine = reinterpret_cast<const uint8_t*>(b3_smem + lane);   // this lane's copy, 128 bytes a word
  const int64_t step = (int64_t)gridDim.x * kB3Warps * kB3Runs;
  int64_t run0 = ((int64_t)blockIdx.x * kB3Warps + warp) * kB3Runs;
  RunPlace at(p, run0);
  const int n4 = p.wpr / 4;
  uint32_t row[kB3Runs];
  int seg[kB3Runs];
  uint4 a[kB3Runs], b[kB3Runs];
  auto load = [&]() {
#pragma unroll
    for (int u = 0; u < kB3Runs; ++u) {
      at.place(p, u, row[u], seg[u]);
      const uint4* src = reinterpret_cast<const uint4*>(plain + (int64_t)row[u] * p.wpr);
      const int i = seg[u] * (kB3Words / 4) + lane;
      a[u] = b[u] = make_uint4(0u, 0u, 0u, 0u);
      if (seg[u] < p.rpr && i < n4) a[u] = __ldcs(src + i);
      if (seg[u] < p.rpr && lane < 8 && i + 32 < n4) b[u] = __ldcs(src + i + 32);
    }
    at.next(p);
  };
  load();
  {
    uint32_t w = 0;   // table word i: the bytes of the field patterns 4 i .. 4 i + 3
#pragma unroll
    for (int k = 0; k < 4; ++k) w |= fields_byte(4 * threadIdx.x + k) << (8 * k);
    fill_table(b3_smem, w);
  }
  for (; run0 < p.total; run0 += step) {
    uint32_t r[kB3Runs];
    int sg[kB3Runs];
#pragma unroll
    for (int u = 0; u < kB3Runs; ++u) {
      uint4* st = reinterpret_cast<uint4*>(stage[u]);
      st[lane] = a[u];
      if (lane < 8) st[lane + 32] = b[u];
      r[u] = row[u];
      sg[u] = seg[u];
    }
    __syncwarp();
    load();
#pragma unroll
    for (int u = 0; u < kB3Runs; ++u) {
      const int g = sg[u] * 32 + lane;
      if (g >= p.gpr) continue;
      uint32_t w[6];
#pragma unroll
      for (int q = 0; q < 5; ++q) w[q] = stage[u][5 * lane + q];
      w[5] = 0u;
      const int64_t c0 = (int64_t)kCodesPerThread * g;
      if (c0 + kCodesPerThread > p.k_eff) {
#pragma unroll
        for (int q = 0; q < 5; ++q) w[q] = below_k_eff(w[q], c0 + 16 * q, p.k_eff);
      }
      uint32_t o[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint32_t y[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // byte b's fields, bits s .. s + 9 of word q: table word (their upper
          // eight bits) 128 bytes apart, byte (their lower two)
          const int bit = 10 * (4 * k + j), q = bit >> 5, s = bit & 31;
          const uint32_t x = s <= 22 ? w[q] : __funnelshift_r(w[q], w[q + 1], s);
          const int h = s <= 22 ? s : 0;
          const uint32_t hi = (h >= 5 ? x >> (h - 5) : x << (5 - h)) & 0x7F80u;
          y[j] = mine[hi | ((x >> h) & 3u)];
        }
        o[k] = __byte_perm(__byte_perm(y[0], y[1], 0x0040), __byte_perm(y[2], y[3], 0x0040), 0x5410);
      }
      *reinterpret_cast<uint4*>(out + (int64_t)r[u] * p.bpr + 16 * g) = make_uint4(o[0], o[1], o[2], o[3]);
    }
    __syncwarp();
  }
}

// The same runs the other way (gpr = ceil(wpr / 5)): base-3 bytes past bpr
// read as 0, plain words past wpr are not written.  Bytes above 242 are
// counted into *bad and read as five 0 codes; codes past K_eff are written as
// 0 (the plain layout's padding).
__global__ void __launch_bounds__(kB3Threads) unpack_base3_kernel(const uint8_t* __restrict__ in,
                                                                  uint32_t* __restrict__ plain, uint32_t* bad,
                                                                  Base3Params p) {
  extern __shared__ __align__(16) uint32_t b3_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t(*stage)[kB3Words] = reinterpret_cast<uint32_t(*)[kB3Words]>(b3_smem + kB3Table) + kB3Runs * warp;
  const uint8_t* table = reinterpret_cast<const uint8_t*>(b3_smem);
  const uint32_t lane4 = 4u * lane;
  const int64_t step = (int64_t)gridDim.x * kB3Warps * kB3Runs;
  int64_t run0 = ((int64_t)blockIdx.x * kB3Warps + warp) * kB3Runs;
  RunPlace at(p, run0);
  const int n4 = p.wpr / 4;
  uint32_t row[kB3Runs];
  int seg[kB3Runs];
  uint4 raw[kB3Runs];
  auto load = [&]() {
#pragma unroll
    for (int u = 0; u < kB3Runs; ++u) {
      at.place(p, u, row[u], seg[u]);
      const int g = seg[u] * 32 + lane;
      raw[u] = make_uint4(0u, 0u, 0u, 0u);
      if (seg[u] < p.rpr && 16 * g < p.bpr)
        raw[u] = __ldcs(reinterpret_cast<const uint4*>(in + (int64_t)row[u] * p.bpr + 16 * g));
    }
    at.next(p);
  };
  load();
  fill_table(b3_smem, byte_fields(threadIdx.x));
  int nbad = 0;
  for (; run0 < p.total; run0 += step) {
    uint32_t r[kB3Runs];
    int sg[kB3Runs];
    uint4 x4[kB3Runs];
#pragma unroll
    for (int u = 0; u < kB3Runs; ++u) {
      x4[u] = raw[u];
      r[u] = row[u];
      sg[u] = seg[u];
    }
    load();
#pragma unroll
    for (int u = 0; u < kB3Runs; ++u) {
      const uint32_t xw[4] = {x4[u].x, x4[u].y, x4[u].z, x4[u].w};
      const uint32_t inv[4] = {invalid_bytes(xw[0]), invalid_bytes(xw[1]), invalid_bytes(xw[2]), invalid_bytes(xw[3])};
      if (inv[0] | inv[1] | inv[2] | inv[3])
        nbad += __popc(inv[0]) + __popc(inv[1]) + __popc(inv[2]) + __popc(inv[3]);
      uint32_t w[5] = {0u, 0u, 0u, 0u, 0u};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t x = xw[k];
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
          // table words of bytes j, j + 1: 128 bytes apart, this lane's copy
          const uint32_t i0 = ((j == 0 ? x << 7 : x >> 9) & 0x7F80u) | lane4;
          const uint32_t i1 = ((j == 0 ? x >> 1 : x >> 17) & 0x7F80u) | lane4;
          const uint32_t v = *reinterpret_cast<const uint32_t*>(table + i0) +
                             1024u * *reinterpret_cast<const uint32_t*>(table + i1);
          const int bit = 10 * (4 * k + j), q = bit >> 5, s = bit & 31;
          w[q] += v << s;
          if (s > 12) w[q + 1] += v >> (32 - s);
        }
      }
      const int64_t c0 = (int64_t)kCodesPerThread * (sg[u] * 32 + lane);
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        if (c0 + kCodesPerThread > p.k_eff) w[q] = below_k_eff(w[q], c0 + 16 * q, p.k_eff);
        stage[u][5 * lane + q] = w[q];
      }
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < kB3Runs; ++u) {
      if (sg[u] >= p.rpr) continue;
      uint4* dst = reinterpret_cast<uint4*>(plain + (int64_t)r[u] * p.wpr);
      const uint4* st = reinterpret_cast<const uint4*>(stage[u]);
      const int i = sg[u] * (kB3Words / 4) + lane;
      if (i < n4) dst[i] = st[lane];
      if (lane < 8 && i + 32 < n4) dst[i + 32] = st[lane + 32];
    }
    __syncwarp();
  }
  if (nbad && bad) atomicAdd(bad, (uint32_t)nbad);
}

// Parameters of a plan's conversion with `gpr` groups per row, and its blocks.
Base3Params base3_params(const sdq_plan_s* pl, int bpr, int gpr, int64_t* blocks) {
  const Geometry& g = pl->geo;
  Base3Params bp;
  bp.n_out = g.n_out; bp.wpr = g.words_per_row; bp.bpr = bpr; bp.gpr = gpr;
  bp.rpr = (gpr + 31) / 32;
  bp.k_eff = g.k_eff; bp.total = (int64_t)g.n_out * bp.rpr;
  *blocks = std::min((bp.total + kB3Warps * kB3Runs - 1) / (kB3Warps * kB3Runs),
                     (int64_t)kB3BlocksPerSm * std::max(1, pl->sm_count));
  const int64_t step = *blocks * kB3Warps * kB3Runs;
  bp.srow = (int)(step / bp.rpr);
  bp.sseg = (int)(step - (int64_t)bp.srow * bp.rpr);
  return bp;
}

int base3_bytes_per_row(int64_t k_eff) { return (int)(16 * (((k_eff + 4) / 5 + 15) / 16)); }

}  // namespace

}  // namespace sdq

using namespace sdq;

extern "C" size_t sdq_base3_bytes(const sdq_layer_desc* desc) {
  Geometry g;
  if (validate(desc, &g) != SDQ_OK || desc->quantizer != SDQ_TERNARY) return 0;
  return (size_t)g.n_out * base3_bytes_per_row(g.k_eff);
}

extern "C" int sdq_pack_base3(sdq_plan p, const uint32_t* codes_plain, uint8_t* codes_base3, void* stream) {
  if (!p || !codes_plain || !codes_base3) return SDQ_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(codes_plain) | reinterpret_cast<uintptr_t>(codes_base3)) & 15u)
    return SDQ_ERR_INVALID_ARG;
  if (p->desc.quantizer != SDQ_TERNARY) return SDQ_ERR_UNSUPPORTED;
  const int dv = sdq_check_device(p);
  if (dv != SDQ_OK) return dv;
  const Geometry& g = p->geo;
  const int bpr = base3_bytes_per_row(g.k_eff);
  int64_t blocks;
  const Base3Params bp = base3_params(p, bpr, bpr / 16, &blocks);
  pack_base3_kernel<<<(unsigned)blocks, kB3Threads, kB3Smem, (cudaStream_t)stream>>>(codes_plain, codes_base3, bp);
  return cudaGetLastError() == cudaSuccess ? SDQ_OK : SDQ_ERR_CUDA;
}

extern "C" int sdq_unpack_base3(sdq_plan p, const uint8_t* codes_base3, uint32_t* codes_plain, uint32_t* bad_count,
                                void* stream) {
  if (!p || !codes_plain || !codes_base3) return SDQ_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(codes_plain) | reinterpret_cast<uintptr_t>(codes_base3)) & 15u)
    return SDQ_ERR_INVALID_ARG;
  if (p->desc.quantizer != SDQ_TERNARY) return SDQ_ERR_UNSUPPORTED;
  const int dv = sdq_check_device(p);
  if (dv != SDQ_OK) return dv;
  const Geometry& g = p->geo;
  int64_t blocks;
  const Base3Params bp = base3_params(p, base3_bytes_per_row(g.k_eff), (g.words_per_row + 4) / 5, &blocks);
  unpack_base3_kernel<<<(unsigned)blocks, kB3Threads, kB3Smem, (cudaStream_t)stream>>>(codes_base3, codes_plain,
                                                                                  bad_count, bp);
  return cudaGetLastError() == cudaSuccess ? SDQ_OK : SDQ_ERR_CUDA;
}
