// K1: row-parallel Sigma-Delta encoder (SDQ-LLM Algorithm 1, eqs. (3)-(8)),
// and the per-block half of its GPTQ compensation.
//
// Two kernels, the same codes bit for bit.  encode_tile_kernel (second half of
// this file) takes the layers whose tables and sizes allow it; the row
// encoder takes the others.
//
// The row encoder: one warp owns 4 output rows.  For every block of B input columns it
// rebuilds the upsampled block x_up = A_enc w (A_enc = U Had^T, the
// Hadamard smoothing of eq. (13) fused with the Resample upsampler) with all
// 32 lanes, each lane producing 4 of every 128 samples for the 4 rows, in
// the canonical fp32 order: one rounded product per term, k ascending, no
// FMA.  Pass 1 reduces alpha per row (exact max, or the sequential fp32
// mean); pass 2 recomputes x_up and lanes 0..3 run the first-order
// Sigma-Delta recursion of eq. (8) over their row, reset at every block, and
// write the codes in the plain packed layout.
//
// The kernel covers a range of passes and blocks.  Where the encoder with GPTQ
// block compensation (Algorithm 1's outer loop with the inverse Hessian) has
// no kernel of its own for a layer (csrc/gptq.cu), it runs pass 1 here one
// block at a time on a working copy of W: after the scan, the warp rebuilds the block Q = alpha (c . G), forms E = W_F - Q and the
// normalised error E~ = E U_FF^-1 (forward substitution over the block's
// columns), which gptq_update_kernel then applies to the later columns.
#include <algorithm>

#include "encode.cuh"
#include "encode_tile.cuh"

namespace sdq {

namespace {

constexpr int kRW = 4;     // rows per warp
constexpr int kMaxWarps = 16;
constexpr int kJC = 128;   // upsampled samples per lane pass (4 per lane)

struct EncodeParams {
  const float* W;
  uint32_t* codes;
  float* alpha;       // written by pass 0, read by pass 1 when pass 0 is not run
  const float* at;  // B x n_b, At[k][j] = A_enc[j][k]
  int n_out, k_in, B, n_b, nblk, wpr, quantizer, alpha_mode, warps;
  int64_t k_eff;
  int pass0, pass1, b0, b1;  // passes [pass0, pass1), blocks [b0, b1)
  // GPTQ (et non-null): G in fp32 (n_b x B), the factor U (k_in x k_in,
  // upper), and the normalised block error E~ written per row (n_out x B)
  const float* g32;
  const float* U;
  float* et;
};

// The warp's GPTQ step for block b of its rows, after the scan: xs holds the
// rows' codes (as +-1 / 0 floats), ws the block's current weights.  In the
// order of the oracle's canonical definition: s_k = sum_j c_j G[j][k] from
// +0 in ascending j, E_k = W_k - alpha s_k; then for l ascending E~_l =
// t_l / U_ll and t_k -= E~_l U_lk for k > l (t starts as E).  Lane owns
// columns k = lane (mod 32); t and E~ live in ws in place.
__device__ __noinline__ void gptq_block_error(const EncodeParams p, int b, int row0, int nrows, float* ws,
                                              const float* xs, int xs_stride, float alpha_row) {
  const int lane = threadIdx.x & 31;
  float ar[kRW];
#pragma unroll
  for (int r = 0; r < kRW; ++r) ar[r] = __shfl_sync(0xffffffffu, alpha_row, r);
  __syncwarp();
  // 128 columns at a time (4 per lane), j outermost: every (row, column) sum
  // still runs over j in ascending order, with 16 independent sums per lane
  for (int kc = 0; kc < p.B; kc += 128) {
    float sacc[kRW][4];
#pragma unroll
    for (int r = 0; r < kRW; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) sacc[r][q] = 0.f;
    for (int j = 0; j < p.n_b; ++j) {
      float gv[4], xv[kRW];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = kc + lane + 32 * q;
        gv[q] = k < p.B ? __ldg(p.g32 + (size_t)j * p.B + k) : 0.f;
      }
#pragma unroll
      for (int r = 0; r < kRW; ++r) xv[r] = xs[r * xs_stride + j];
#pragma unroll
      for (int r = 0; r < kRW; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) sacc[r][q] = __fadd_rn(sacc[r][q], __fmul_rn(xv[r], gv[q]));
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = kc + lane + 32 * q;
      if (k >= p.B) continue;
#pragma unroll
      for (int r = 0; r < kRW; ++r) ws[r * p.B + k] = __fsub_rn(ws[r * p.B + k], __fmul_rn(ar[r], sacc[r][q]));
    }
  }
  const size_t ldu = (size_t)p.k_in;
  const float* uff = p.U + (size_t)b * p.B * ldu + (size_t)b * p.B;
  for (int l = 0; l < p.B; ++l) {
    __syncwarp();
    const float d = __ldg(uff + (size_t)l * ldu + l);
    float el[kRW];
#pragma unroll
    for (int r = 0; r < kRW; ++r) el[r] = __fdiv_rn(ws[r * p.B + l], d);
    __syncwarp();
    if ((l & 31) == lane) {
#pragma unroll
      for (int r = 0; r < kRW; ++r) ws[r * p.B + l] = el[r];
    }
    for (int k = lane; k < p.B; k += 32) {
      if (k <= l) continue;
      const float u = __ldg(uff + (size_t)l * ldu + k);
#pragma unroll
      for (int r = 0; r < kRW; ++r) ws[r * p.B + k] = __fsub_rn(ws[r * p.B + k], __fmul_rn(el[r], u));
    }
  }
  __syncwarp();
  for (int i = lane; i < nrows * p.B; i += 32) {
    const int r = i / p.B, k = i - r * p.B;
    p.et[(size_t)(row0 + r) * p.B + k] = ws[i];
  }
  __syncwarp();
}

// kTable: the CTA first copies the table into shared memory (where it fits
// beside the warps' buffers); its reads in the product loop are then
// shared-memory hits instead of L2 round trips, on which the loop waited.
template <bool kTable, bool kGptq>
__global__ void __launch_bounds__(32 * kMaxWarps) encode_kernel(EncodeParams p) {
  extern __shared__ float smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int xs_stride = p.n_b + 1;
  const float* at = p.at;
  float* wbuf = smem;
  if constexpr (kTable) {
    float* ts = smem;
    const int n = p.B * p.n_b;
    for (int i = threadIdx.x; i < n / 4; i += blockDim.x)
      reinterpret_cast<float4*>(ts)[i] = __ldg(reinterpret_cast<const float4*>(p.at) + i);
    __syncthreads();
    at = ts;
    wbuf = smem + n;
  }
  float* ws = wbuf + (size_t)warp * (kRW * p.B + kRW * xs_stride);
  float* xs = ws + kRW * p.B;
  const int row0 = (blockIdx.x * p.warps + warp) * kRW;
  if (row0 >= p.n_out) return;
  const int nrows = min(kRW, p.n_out - row0);
  const bool need_xs_pass0 = p.alpha_mode == SDQ_ALPHA_MEANABS;

  float amax[kRW];
#pragma unroll
  for (int r = 0; r < kRW; ++r) amax[r] = 0.f;
  float mean_acc = 0.f;  // lane r < 8: sequential sum for MEANABS
  bool mean_first = true;
  float alpha_row = 0.f;  // lane r < 8: alpha of row row0 + r
  if (p.pass0 == 1 && lane < nrows) alpha_row = p.alpha[row0 + lane];
  const int per = 32 / p.quantizer;

  for (int pass = p.pass0; pass < p.pass1; ++pass) {
    // pass-2 scan state of lane r (< nrows): the partial code word; a range
    // that starts inside a word continues the word its predecessor wrote
    uint32_t cw = 0;
    if (pass == 1 && lane < nrows && ((int64_t)p.b0 * p.n_b) % per != 0)
      cw = p.codes[(size_t)(row0 + lane) * p.wpr + (int64_t)p.b0 * p.n_b / per];
    for (int b = p.b0; b < p.b1; ++b) {
      __syncwarp();
      const float* wsrc = p.W + (size_t)row0 * p.k_in + (size_t)b * p.B;
      for (int i = lane; i < kRW * p.B; i += 32) {
        const int r = i / p.B, k = i - r * p.B;
        ws[i] = r < nrows ? __ldg(wsrc + (size_t)r * p.k_in + k) : 0.f;
      }
      __syncwarp();
      for (int jc = 0; jc < p.n_b; jc += kJC) {
        float acc[kRW][4];
        int jj[4];
        bool jv[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          jj[s] = jc + lane + 32 * s;
          jv[s] = jj[s] < p.n_b;
        }
        {
          float a[4];
#pragma unroll
          for (int s = 0; s < 4; ++s) a[s] = jv[s] ? at[jj[s]] : 0.f;
#pragma unroll
          for (int r = 0; r < kRW; ++r) {
            const float wk = ws[r * p.B];
#pragma unroll
            for (int s = 0; s < 4; ++s) acc[r][s] = __fmul_rn(a[s], wk);
          }
        }
        for (int k = 1; k < p.B; ++k) {
          float a[4];
#pragma unroll
          for (int s = 0; s < 4; ++s) a[s] = jv[s] ? at[(size_t)k * p.n_b + jj[s]] : 0.f;
#pragma unroll
          for (int r = 0; r < kRW; ++r) {
            const float wk = ws[r * p.B + k];
#pragma unroll
            for (int s = 0; s < 4; ++s) acc[r][s] = __fadd_rn(acc[r][s], __fmul_rn(a[s], wk));
          }
        }
        if (pass == 0 && !need_xs_pass0) {
#pragma unroll
          for (int r = 0; r < kRW; ++r)
#pragma unroll
            for (int s = 0; s < 4; ++s)
              if (jv[s]) amax[r] = fmaxf(amax[r], fabsf(acc[r][s]));
        } else {
#pragma unroll
          for (int r = 0; r < kRW; ++r)
#pragma unroll
            for (int s = 0; s < 4; ++s)
              if (jv[s]) xs[r * xs_stride + jj[s]] = acc[r][s];
        }
      }
      __syncwarp();
      if (pass == 0) {
        if (need_xs_pass0 && lane < nrows) {
          for (int j = 0; j < p.n_b; ++j) {
            const float v = fabsf(xs[lane * xs_stride + j]);
            mean_acc = mean_first ? v : __fadd_rn(mean_acc, v);
            mean_first = false;
          }
        }
      } else if (lane < nrows) {
        // Eq. (8): i = (i + x) - y_prev, reset per block.
        const float a = alpha_row, theta = 0.5f * alpha_row;
        float integ = 0.f, yp = 0.f;
        uint32_t* crow = p.codes + (size_t)(row0 + lane) * p.wpr;
        const bool range_end = b == p.b1 - 1;
        for (int j = 0; j < p.n_b; ++j) {
          integ = __fsub_rn(__fadd_rn(integ, xs[lane * xs_stride + j]), yp);
          uint32_t field;
          float cv;
          if (p.quantizer == SDQ_TERNARY) {
            if (integ > theta) { field = 1u; yp = a; cv = 1.f; }
            else if (integ < -theta) { field = 3u; yp = -a; cv = -1.f; }
            else { field = 0u; yp = 0.f; cv = 0.f; }
          } else {
            if (integ >= 0.f) { field = 1u; yp = a; cv = 1.f; }
            else { field = 0u; yp = -a; cv = -1.f; }
          }
          if (kGptq) xs[lane * xs_stride + j] = cv;
          const int64_t kk = (int64_t)b * p.n_b + j;
          const int pos = (int)(kk % per);
          cw |= field << (p.quantizer * pos);
          if (pos == per - 1 || kk == p.k_eff - 1 || (range_end && j == p.n_b - 1)) {
            crow[kk / per] = cw;
            cw = 0;
          }
        }
      }
      if (kGptq && pass == 1) gptq_block_error(p, b, row0, nrows, ws, xs, xs_stride, alpha_row);
    }
    if (pass == 0) {
      if (p.alpha_mode == SDQ_ALPHA_MAXABS) {
#pragma unroll
        for (int r = 0; r < kRW; ++r) {
          float v = amax[r];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
          if (lane == r) alpha_row = v;
        }
      } else if (lane < nrows) {
        alpha_row = __fdiv_rn(mean_acc, (float)p.k_eff);
      }
      if (lane < nrows) p.alpha[row0 + lane] = alpha_row;
    }
  }
  // Zero the row padding words past the last code.
  if (p.pass1 == 2 && p.b1 == p.nblk && lane < nrows) {
    uint32_t* crow = p.codes + (size_t)(row0 + lane) * p.wpr;
    for (int64_t w = (p.k_eff + per - 1) / per; w < p.wpr; ++w) crow[w] = 0u;
  }
}

// ------------------------------------------------------------ tile encoder
// The encoder for layers whose table has the half-shift symmetry (below) and
// whose codes of a block fill whole words.
//
// A_enc row j + n_b / 2 is row j shifted by half a block, and a shift by B / 2
// of an index below B flips its top bit: in the Hadamard domain
//   A[j + n_b / 2][k] = A[j][k] (k < B / 2),  -A[j][k] (k >= B / 2)
// for every OSR (checked bit for bit at plan creation).  So samples j and j +
// n_b / 2 share their sums over k < B / 2, and above that their products
// p: one adds p, the other subtracts it.  320 rounded operations in place of
// 512 per pair at B = 128, every sum in the canonical order.
//
// fp32 multiply / add issue bounds it, so the rest is arranged around that: a
// warp owns 8 virtual rows (row, block) x all n_b samples, lane l the pairs j =
// l + 32 q (q < PT), 8 PT x 2 sums in registers; per k one shared-memory word of
// the table per pair (conflict-free) and two broadcast 16-byte loads of the 8
// weights serve 8 PT x 2 or 3 operations.  The persistent CTA (one per SM) holds
// half the table and works on groups of whole rows: where a group's virtual
// rows fit in the CTA's tile (8 per warp), alpha and the scan both use the one
// computation of x_up, else pass 0 takes the maxima and pass 1 recomputes.
// The scan (eq. 8) of a tile runs with one lane per virtual row, 32 to a
// warp, beside the other warps' next tile: blocks are independent, so 32
// lanes of a warp scan where 4 did with a lane per row.  Alpha as a mean is one
// chain of rounded sums per row: lane r of the team's first warp adds row r's
// samples, beside the other teams' products (4096 x 4096, B = 128, OSR 2: 3.18
// ms with the row encoder, 1.27 with its pass 0 alone, 0.59 so).
// 11008 x 4096, OSR 2 (46 G rounded operations as two plain passes, 14 G so):
// 6.24 ms with the row encoder, 0.71 ms (0.95 with one
// team per CTA, whose barriers had the other warps wait for the scan).
// warps at most: 16, or 8 where a thread needs more than 128 registers
constexpr int tile_max_warps(int pt) { return pt <= 4 ? 16 : 8; }
constexpr int kTMaxRows = 16;   // rows per group
constexpr int kTMaxTeams = 4;

struct TileParams {
  const float* W;
  uint32_t* codes;
  float* alpha;
  const float* at;   // B x n_b
  int n_out, k_in, B, n_b, nblk, wpr, quantizer, rows, mean, only_alpha;
  float k_eff;
  int gw;            // warps of a team
  uint32_t pad0;     // first padding word of a row
};

// kTable: half the table in shared memory (np at most 32 PT); else it is read
// where it is (every warp of the CTA reads the same rows at about the same
// time: the L1 serves them) and the samples are done 32 PT pairs at a time.
template <int PT, bool kTable>
__global__ void __launch_bounds__(32 * tile_max_warps(PT), 1) encode_tile_kernel(TileParams p) {
  extern __shared__ __align__(16) float smem[];
  __shared__ uint32_t s_amax[kTMaxTeams][2][kTMaxRows];   // bit patterns of the rows' maxima (non-negative floats)
  const int warp = warp_index(), lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  // teams of gw warps work on row groups of their own and meet at their own
  // barriers, so that one team's scan runs beside the others' products
  const int team = warp / p.gw, tw = warp - team * p.gw, nteam = nwarp / p.gw, tt = 32 * tw + lane;
  auto team_sync = [&]() { named_bar_sync(1 + team, 32 * p.gw); };
  const int np = p.n_b / 2, xs_stride = p.n_b + 1;
  const size_t table = kTable ? (size_t)p.B * np : 0;
  float* ts = smem;                                        // B x np
  float* wt = ts + table + (size_t)warp * tile_weight_floats(p.B);
  float* xs0 = ts + table + (size_t)nwarp * tile_weight_floats(p.B) +
               (size_t)team * p.gw * kTv * xs_stride;   // the team's samples
  float* xs = xs0 + (size_t)tw * kTv * xs_stride;
  if constexpr (kTable) tile_load_table(ts, p.at, p.B, p.n_b);
  for (int i = threadIdx.x; i < kTMaxTeams * 2 * kTMaxRows; i += blockDim.x) (&s_amax[0][0][0])[i] = 0u;
  __syncthreads();

  const int tv = kTv * p.gw, ngroups = (p.n_out + p.rows - 1) / p.rows;
  float acc[kTv][PT], acc2[kTv][PT];

  // the 8 x B weights of virtual rows v0 .. v0 + 7 of the group at row0 (nv in
  // all), transposed to [k][8]: lane = (virtual row, float4)
  auto load_weights = [&](int row0, int v0, int nv) {
    const int v = v0 + (lane >> 2), r = min(v, nv - 1) / p.nblk, b = min(v, nv - 1) - r * p.nblk;
    const float4* src = reinterpret_cast<const float4*>(p.W + (size_t)(row0 + r) * p.k_in + (size_t)b * p.B);
    __syncwarp();
    for (int k4 = lane & 3; k4 < p.B / 4; k4 += 4) {
      const float4 w = v < nv ? __ldg(src + k4) : make_float4(0.f, 0.f, 0.f, 0.f);
      float* d = wt + k4 * kWk4 + (lane >> 2);
      d[0] = w.x; d[8] = w.y; d[16] = w.z; d[24] = w.w;
    }
    __syncwarp();
  };
  // their x_up into acc (samples j0 + l + 32 q) and acc2 (the same + n_b / 2)
  auto compute = [&](int j0) {
    if constexpr (kTable) tile_upsample<PT>(ts + lane, np, np - lane, wt, p.B, acc, acc2);
    else tile_upsample<PT>(p.at + j0 + lane, p.n_b, np - j0 - lane, wt, p.B, acc, acc2);
  };
  // row maxima of the warp's 8 virtual rows (pairs past np hold zeros)
  auto maxima = [&](int v0, int nv, uint32_t* am) {
#pragma unroll
    for (int v = 0; v < kTv; ++v) {
      float m = 0.f;
#pragma unroll
      for (int q = 0; q < PT; ++q) m = fmaxf(m, fmaxf(fabsf(acc[v][q]), fabsf(acc2[v][q])));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0 && v0 + v < nv) atomicMax(&am[(v0 + v) / p.nblk], __float_as_uint(m));
    }
  };
  auto store = [&](int j0) {
#pragma unroll
    for (int v = 0; v < kTv; ++v)
#pragma unroll
      for (int q = 0; q < PT; ++q) {
        const int j = j0 + lane + 32 * q;
        if (j < np) {
          xs[v * xs_stride + j] = acc[v][q];
          xs[v * xs_stride + np + j] = acc2[v][q];
        }
      }
  };
  // Eq. (8) over virtual row `lv` of the tile: i = (i + x) - y_prev from 0,
  // the codes packed into whole words.
  auto scan = [&](int row, int b, int lv, float a) {
    const float theta = 0.5f * a;
    const float* x = xs0 + (size_t)lv * xs_stride;
    uint32_t* out = p.codes + (size_t)row * p.wpr + (size_t)b * p.n_b * p.quantizer / 32;
    float integ = 0.f, yp = 0.f;
    if (p.quantizer == SDQ_TERNARY) {
      for (int j = 0; j < p.n_b; j += 16) {
        uint32_t cw = 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) cw |= sd_step<true>(integ, yp, x[j + i], a, theta) << (2 * i);
        out[j / 16] = cw;
      }
    } else {
      for (int j = 0; j < p.n_b; j += 32) {
        uint32_t cw = 0;
#pragma unroll
        for (int i = 0; i < 32; ++i) cw |= sd_step<false>(integ, yp, x[j + i], a, theta) << i;
        out[j / 32] = cw;
      }
    }
    if (b == p.nblk - 1)   // the row's padding words
      for (int w = (int)p.pad0; w < p.wpr; ++w) p.codes[(size_t)row * p.wpr + w] = 0u;
  };

  int turn = 0;   // scanning warps rotate over the team
  int buf = 0;
  for (int g = blockIdx.x + team * gridDim.x; g < ngroups; g += gridDim.x * nteam, buf ^= 1) {
    const int row0 = g * p.rows, nv = min(p.rows, p.n_out - row0) * p.nblk;
    const int tiles = (nv + tv - 1) / tv;
    uint32_t *am = s_amax[team][buf], *am_next = s_amax[team][buf ^ 1];
    const bool single = tiles == 1 && !p.only_alpha;   // one computation for alpha and the scan
    const int n0 = single ? 0 : tiles;                 // steps of pass 0
    const int steps = n0 + (p.only_alpha ? 0 : tiles);
    float mean_acc = 0.f;   // MEANABS: lane r of the team's first warp adds row r's samples
    bool mean_first = true;
    for (int step = 0; step < steps; ++step) {
      const int t = step < n0 ? step : step - n0, v0 = t * tv + tw * kTv;
      const bool pass0 = step < n0, samples = !pass0 || p.mean;
      if (v0 < nv) load_weights(row0, v0, nv);
      for (int j0 = 0; j0 < np; j0 += 32 * PT) {
        if (v0 < nv) {
          compute(j0);
          if (!p.mean && (pass0 || single)) maxima(v0, nv, am);
        }
        if (!samples) continue;
        if (j0 == 0) {
          team_sync();   // the tile before is scanned (summed)
          if (!pass0 && t == 0 && tt < kTMaxRows) am_next[tt] = 0u;
        }
        if (v0 < nv) store(j0);
      }
      if (!samples) continue;
      team_sync();
      if (p.mean && (pass0 || single)) {
        // the canonical mean: one rounded sum in (block, index) order per row
        if (tw == 0 && lane * p.nblk < nv) {
          const int vb = min((lane + 1) * p.nblk, min((t + 1) * tv, nv));
          for (int v = max(lane * p.nblk, t * tv); v < vb; ++v) {
            const float* x = xs0 + (size_t)(v - t * tv) * xs_stride;
#pragma unroll 16
            for (int j = 0; j < p.n_b; ++j) {
              const float a = fabsf(x[j]);
              mean_acc = mean_first ? a : __fadd_rn(mean_acc, a);
              mean_first = false;
            }
          }
          if (t == tiles - 1) am[lane] = __float_as_uint(__fdiv_rn(mean_acc, p.k_eff));
        }
        if (single) team_sync();
      }
      if (pass0) continue;
      // 32 virtual rows per scanning warp
      const int part = (tw - turn + p.gw) % p.gw;
      const int lv = 32 * part + lane, v = t * tv + lv;
      if (lv < tv && v < nv) {
        const int r = v / p.nblk, b = v - r * p.nblk, row = row0 + r;
        const float a = __uint_as_float(am[r]);
        if (b == 0) p.alpha[row] = a;
        scan(row, b, lv, a);
      }
      turn = (turn + (tv + 31) / 32) % p.gw;
    }
    if (p.only_alpha) {
      team_sync();
      if (tt < kTMaxRows) {
        if (tt * p.nblk < nv) p.alpha[row0 + tt] = __uint_as_float(am[tt]);
        am_next[tt] = 0u;
      }
      team_sync();
    }
  }
}

// Warps, warps per team and rows per group of the tile encoder, 0 warps where
// it does not apply: the half-shift table, whole words of codes per block, and
// at least 2 warps' buffers (10 B + 8 (n_b + 1) words each) in shared memory;
// half the table (n_b / 2 x B words) joins them where it has at most 192
// pairs and leaves room for 4 warps, else it is read from global memory (4096 x
// 4096, OSR 2, B = 256 and 512: 0.64 and 1.6 ms, the row encoder 9.0 and 14.4).
struct TileShape {
  bool table;
  int warps, gw, rows, pt;
  size_t smem;
};
TileShape tile_shape(const sdq_plan_s* pl) {
  const Geometry& g = pl->geo;
  TileShape t{};
  const int np = g.n_b / 2;
  if (!pl->half_shift || g.block < 16 || (g.n_b * g.bits) % 32) return t;
  size_t table = sizeof(float) * (size_t)g.block * np;
  const size_t per_warp = sizeof(float) * ((size_t)tile_weight_floats(g.block) + (size_t)kTv * (g.n_b + 1));
  const size_t room = 226 * 1024;
  t.table = np <= 192 && table + 4 * per_warp <= room;
  if (!t.table) {
    table = 0;
    if (2 * per_warp > room) return t;
  }
  t.pt = t.table ? (np + 31) / 32 : 4;
  const int most = (int)std::min<size_t>(tile_max_warps(t.pt), (room - table) / per_warp);
  const int64_t sms = std::max(1, pl->sm_count);
  const bool mean = pl->desc.alpha_mode == SDQ_ALPHA_MEANABS;
  // Teams of 4 warps or of all (most of them in whole teams), and the row
  // count whose groups take the least time on the busiest SM: a tile's
  // products on the warps that have virtual rows in it, twice where alpha
  // and the scan need two computations, and a scan (a fifth of a full
  // tile's products on 12 warps), which other teams' products hide.
  double best = 0;
  const int widths[2] = {4, most & ~1};
  for (int gw : widths) {
    if (gw > most) continue;
    const int nteam = most / gw, tv = kTv * gw;
    for (int r = 1; r <= kTMaxRows; ++r) {
      const int64_t groups = (g.n_out + r - 1) / r;
      const int64_t turns = (groups + sms * nteam - 1) / (sms * nteam);   // groups of the busiest team
      const int64_t tiles = ((int64_t)r * g.nblk + tv - 1) / tv;
      const double live = tiles == 1 ? (double)((r * g.nblk + kTv - 1) / kTv) : (double)gw;   // warps at work
      // the SM's issue slots shared by its teams' warps, at least one warp per quadrant's own pace
      const double products = tiles * std::max(live * nteam / 12.0, 0.35) * (tiles == 1 ? 1.0 : 2.0);
      // MEANABS: a row's sum is one chain of about 5 cycles a sample
      const double chain = mean ? 5.0 * (double)g.k_eff / (1.9 * np * g.block) : 0.0;
      const double c = (double)turns * std::max(products + (nteam > 1 ? 0.08 : 0.3) * tiles,
                                                products / nteam + chain + 0.2 * tiles);
      if (!t.warps || c < best * 0.999) {
        best = c;
        t.warps = gw * nteam;
        t.gw = gw;
        t.rows = r;
      }
    }
  }
  t.smem = table + t.warps * per_warp;
  return t;
}

cudaError_t launch_encode_tile(const sdq_plan_s* pl, const TileShape& t, const float* W, uint32_t* codes, float* alpha,
                               cudaStream_t st, bool only_alpha) {
  const Geometry& g = pl->geo;
  TileParams p;
  p.W = W; p.codes = codes; p.alpha = alpha; p.at = pl->d_at;
  p.n_out = g.n_out; p.k_in = g.k_in; p.B = g.block; p.n_b = g.n_b; p.nblk = g.nblk;
  p.wpr = g.words_per_row; p.quantizer = pl->desc.quantizer; p.rows = t.rows;
  p.mean = pl->desc.alpha_mode == SDQ_ALPHA_MEANABS; p.only_alpha = only_alpha; p.gw = t.gw;
  p.k_eff = (float)g.k_eff;
  p.pad0 = (uint32_t)(g.k_eff * g.bits / 32);
  auto kern = !t.table ? encode_tile_kernel<4, false>
              : t.pt <= 1 ? encode_tile_kernel<1, true> : t.pt == 2 ? encode_tile_kernel<2, true>
              : t.pt == 3 ? encode_tile_kernel<3, true> : t.pt == 4 ? encode_tile_kernel<4, true>
              : t.pt == 5 ? encode_tile_kernel<5, true> : encode_tile_kernel<6, true>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
  if (e != cudaSuccess) return e;
  const int groups = (g.n_out + t.rows - 1) / t.rows;
  kern<<<std::min(groups, std::max(1, pl->sm_count)), 32 * t.warps, t.smem, st>>>(p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_encode(const sdq_plan_s* pl, const float* W, uint32_t* codes, float* alpha,
                          cudaStream_t st) {
  const TileShape t = tile_shape(pl);
  return t.warps ? launch_encode_tile(pl, t, W, codes, alpha, st, false)
                 : launch_encode_range(pl, W, codes, alpha, st, 0, 2, 0, pl->geo.nblk, nullptr, nullptr);
}

cudaError_t launch_encode_alpha(const sdq_plan_s* pl, const float* W, uint32_t* codes, float* alpha, cudaStream_t st) {
  const TileShape t = tile_shape(pl);
  return t.warps ? launch_encode_tile(pl, t, W, codes, alpha, st, true)
                 : launch_encode_range(pl, W, codes, alpha, st, 0, 1, 0, pl->geo.nblk, nullptr, nullptr);
}

cudaError_t launch_encode_range(const sdq_plan_s* pl, const float* W, uint32_t* codes, float* alpha,
                                cudaStream_t st, int pass0, int pass1, int b0, int b1, const float* U,
                                float* et) {
  const Geometry& g = pl->geo;
  EncodeParams p;
  p.W = W; p.codes = codes; p.alpha = alpha; p.at = pl->d_at;
  p.n_out = g.n_out; p.k_in = g.k_in; p.B = g.block; p.n_b = g.n_b; p.nblk = g.nblk;
  p.wpr = g.words_per_row; p.quantizer = pl->desc.quantizer; p.alpha_mode = pl->desc.alpha_mode;
  p.k_eff = g.k_eff;
  p.pass0 = pass0; p.pass1 = pass1; p.b0 = b0; p.b1 = b1;
  p.g32 = pl->d_g32; p.U = U; p.et = et;
  const size_t per_warp = sizeof(float) * ((size_t)kRW * g.block + (size_t)kRW * (g.n_b + 1));
  const size_t table = sizeof(float) * (size_t)g.block * g.n_b;
  if (per_warp > 227 * 1024) return cudaErrorInvalidConfiguration;
  // the table in shared memory when it fits beside at least 4 warps' buffers
  // (a multiple of 4 floats: copied as float4)
  const bool in_smem = (g.block * g.n_b) % 4 == 0 && table + 4 * per_warp <= 224 * 1024;
  int warps = (int)(((in_smem ? 224 * 1024 - table : 200 * 1024)) / per_warp);
  warps = warps < 1 ? 1 : (warps > kMaxWarps ? kMaxWarps : warps);
  p.warps = warps;
  const size_t smem = per_warp * warps + (in_smem ? table : 0);
  const bool gptq = et != nullptr;
  auto kern = in_smem ? (gptq ? encode_kernel<true, true> : encode_kernel<true, false>)
                      : (gptq ? encode_kernel<false, true> : encode_kernel<false, false>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int rows_per_cta = warps * kRW;
  const int grid = (g.n_out + rows_per_cta - 1) / rows_per_cta;
  kern<<<grid, warps * 32, smem, st>>>(p);
  return cudaGetLastError();
}

}  // namespace sdq
