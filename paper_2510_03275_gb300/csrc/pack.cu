// K2: plain <-> tiled code layouts (layout maps in include/sdq.h).
//
// Both layouts keep each row's codes in natural order inside groups of 64
// codes, so the tiled layout is a regrouping of plain-layout runs of wpg
// words (16 bytes ternary, 8 bytes binary): run (row, group G) of the plain
// layout becomes row r = row % 128 of slab (row / 128, G).
//
// Both directions move bytes and nothing else, so HBM bounds them.  A thread
// moves whole runs: one load, one store of the run's 16 (8) bytes.  A warp
// covers 8 rows x 4 groups, so that on the plain side each row's 4 runs are
// 64 (32) contiguous bytes and on the tiled side each slab's 8 rows 128 (64):
// whole 32-byte sectors both ways without staging.  A block takes one row
// tile x 8 groups, every thread 4 runs, all its loads in flight before the
// first store.  One word per thread (a 64-bit division per word, plain-side
// reads of 16 bytes a row apart) took 117 us for the 28672 x 16384 ternary
// codes of a LLaMA-70B gate linear (235 MB in and out); this takes 34 us, the
// rate of a plain copy.
#include "common.cuh"

namespace sdq {

namespace {

constexpr int kPackGroups = 8;    // groups per block
constexpr int kPackThreads = 256;
constexpr int kPackRuns = kTileRows * kPackGroups / kPackThreads;   // runs per thread

struct PackParams {
  int n_out, wpr, ngroups;
};

// The run of thread tid's i-th move: warp w takes row blocks w, w + 8 (8 rows
// each) and for each both group quads.
__device__ __forceinline__ void pack_run(int i, int& r, int& g) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  r = 8 * (warp + 8 * (i >> 1)) + (lane >> 2);
  g = 4 * (i & 1) + (lane & 3);
}

// Vec: the type of a run (uint4 ternary, uint2 binary).  Rows past n_out and
// groups past the plain row are padding (0).  A plain row is a whole number
// of runs (16-byte multiples).
template <typename Vec>
__global__ void __launch_bounds__(kPackThreads) pack_kernel(const Vec* __restrict__ plain, Vec* __restrict__ tiled,
                                                            PackParams p) {
  const int rpr = p.wpr / (int)(sizeof(Vec) / 4);   // runs per plain row
  const int64_t tile = blockIdx.x;
  const int g0 = (int)blockIdx.y * kPackGroups;
  Vec v[kPackRuns];
#pragma unroll
  for (int i = 0; i < kPackRuns; ++i) {
    int r, g;
    pack_run(i, r, g);
    const int64_t row = tile * kTileRows + r;
    v[i] = Vec{};
    if (row < p.n_out && g0 + g < rpr) v[i] = __ldcs(plain + row * rpr + g0 + g);
  }
#pragma unroll
  for (int i = 0; i < kPackRuns; ++i) {
    int r, g;
    pack_run(i, r, g);
    if (g0 + g < p.ngroups) tiled[(tile * p.ngroups + g0 + g) * kTileRows + r] = v[i];
  }
}

// Ternary pattern 10 is counted and decoded as 0.
__device__ __forceinline__ uint32_t valid_fields(uint32_t v, int& nbad) {
  const uint32_t invalid = (v >> 1) & ~v & 0x55555555u;
  nbad += __popc(invalid);
  return v & ~(invalid | (invalid << 1));
}
__device__ __forceinline__ void valid_run(uint4& v, int& nbad) {
  v.x = valid_fields(v.x, nbad);
  v.y = valid_fields(v.y, nbad);
  v.z = valid_fields(v.z, nbad);
  v.w = valid_fields(v.w, nbad);
}
__device__ __forceinline__ void valid_run(uint2&, int&) {}   // every binary pattern is a code

template <typename Vec>
__global__ void __launch_bounds__(kPackThreads) unpack_kernel(const Vec* __restrict__ tiled, Vec* __restrict__ plain,
                                                              uint32_t* bad, PackParams p) {
  const int rpr = p.wpr / (int)(sizeof(Vec) / 4);
  const int64_t tile = blockIdx.x;
  const int g0 = (int)blockIdx.y * kPackGroups;
  Vec v[kPackRuns];
#pragma unroll
  for (int i = 0; i < kPackRuns; ++i) {
    int r, g;
    pack_run(i, r, g);
    v[i] = Vec{};
    if (tile * kTileRows + r < p.n_out && g0 + g < rpr)
      v[i] = __ldcs(tiled + (tile * p.ngroups + g0 + g) * kTileRows + r);
  }
  int nbad = 0;
#pragma unroll
  for (int i = 0; i < kPackRuns; ++i) {
    int r, g;
    pack_run(i, r, g);
    const int64_t row = tile * kTileRows + r;
    valid_run(v[i], nbad);
    if (row < p.n_out && g0 + g < rpr) plain[row * rpr + g0 + g] = v[i];
  }
  if (nbad && bad) atomicAdd(bad, (uint32_t)nbad);
}

// Grid: row tiles (at most 2^17) x group chunks (at most 2^15).
dim3 pack_grid(const Geometry& g) {
  return dim3((unsigned)g.ntiles, (unsigned)((g.ngroups + kPackGroups - 1) / kPackGroups));
}

}  // namespace

cudaError_t launch_pack(const sdq_plan_s* pl, const uint32_t* plain, uint32_t* tiled, cudaStream_t st) {
  const Geometry& g = pl->geo;
  const PackParams p{g.n_out, g.words_per_row, g.ngroups};
  if (g.wpg == 4)
    pack_kernel<uint4><<<pack_grid(g), kPackThreads, 0, st>>>(reinterpret_cast<const uint4*>(plain),
                                                              reinterpret_cast<uint4*>(tiled), p);
  else
    pack_kernel<uint2><<<pack_grid(g), kPackThreads, 0, st>>>(reinterpret_cast<const uint2*>(plain),
                                                              reinterpret_cast<uint2*>(tiled), p);
  return cudaGetLastError();
}

cudaError_t launch_unpack(const sdq_plan_s* pl, const uint32_t* tiled, uint32_t* plain,
                          uint32_t* bad, cudaStream_t st) {
  const Geometry& g = pl->geo;
  const PackParams p{g.n_out, g.words_per_row, g.ngroups};
  if (g.wpg == 4)
    unpack_kernel<uint4><<<pack_grid(g), kPackThreads, 0, st>>>(reinterpret_cast<const uint4*>(tiled),
                                                                reinterpret_cast<uint4*>(plain), bad, p);
  else
    unpack_kernel<uint2><<<pack_grid(g), kPackThreads, 0, st>>>(reinterpret_cast<const uint2*>(tiled),
                                                                reinterpret_cast<uint2*>(plain), bad, p);
  return cudaGetLastError();
}

}  // namespace sdq
