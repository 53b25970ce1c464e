// GPTQ block compensation for the Sigma-Delta encoder (SDQ-LLM Algorithm 1:
// the outer loop over blocks of B columns, with the inverse Hessian H^-1 =
// (2 X X^T + lambda I)^-1 given through its upper Cholesky factor U,
// U^T U = H^-1).
//
// Blocks are encoded in order on a working copy of W: by the row-owner kernel
// (second half of this file) where it applies, else with encode_kernel and
// gptq_update_kernel, a launch of each per block.  After block b is encoded,
// each row's block error E =
// W_F - alpha (c . G) is normalised by the factor's diagonal block, E~ =
// E U_FF^-1, and the later columns take the update W_R -= E~ U_FR: the exact
// block update of GPTQ / optimal brain surgeon (for B = 1 it is GPTQ's
// division by the diagonal), equal to E H_FR H_RR^-1.  Every product and sum
// is a rounded fp32 operation in a fixed order (ascending k, first product
// not added to a zero), so the codes are a deterministic function of W and U.
#include <algorithm>
#include <type_traits>

#include "encode.cuh"
#include "encode_tile.cuh"

namespace sdq {

namespace {

constexpr int kUpT = 128;      // rows and columns of W per CTA
constexpr int kUpK = 32;       // block columns (k) per shared-memory chunk
constexpr int kUpThreads = 256;

// W[r, c] -= sum_k E~[r, k] U[f0 + k, c] for r < n_out, c in [col0, k_in):
// 128 x 128 outputs per CTA, 8 x 8 per thread (rows 4 ty .. 4 ty + 3 and 64 +
// the same, columns likewise in tx), E~ and U staged through shared memory
// 32 k at a time.
__global__ void __launch_bounds__(kUpThreads, 2)
    gptq_update_kernel(float* __restrict__ W, const float* __restrict__ et, const float* __restrict__ U,
                       int n_out, int k_in, int B, int f0, int col0) {
  __shared__ __align__(16) float es[kUpK][kUpT];   // es[k][row] = E~[r0 + row, kc + k]
  __shared__ __align__(16) float us[kUpK][kUpT];   // us[k][col] = U[f0 + kc + k, c0 + col]
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int r0 = blockIdx.y * kUpT, c0 = col0 + blockIdx.x * kUpT;
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = -0.0f;   // -0 + p == p: the first product is taken as is
  for (int kc = 0; kc < B; kc += kUpK) {
    const int kn = min(kUpK, B - kc);
    for (int i = tid; i < kUpT * (kUpK / 4); i += kUpThreads) {
      const int row = i / (kUpK / 4), k4 = i % (kUpK / 4);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r0 + row < n_out && 4 * k4 < kn)
        v = __ldg(reinterpret_cast<const float4*>(et + (size_t)(r0 + row) * B + kc + 4 * k4));
      es[4 * k4 + 0][row] = v.x;
      es[4 * k4 + 1][row] = v.y;
      es[4 * k4 + 2][row] = v.z;
      es[4 * k4 + 3][row] = v.w;
    }
    for (int i = tid; i < kUpK * (kUpT / 4); i += kUpThreads) {
      const int k = i / (kUpT / 4), c4 = i % (kUpT / 4);
      const int col = c0 + 4 * c4;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k < kn && col < k_in)
        v = __ldg(reinterpret_cast<const float4*>(U + (size_t)(f0 + kc + k) * k_in + col));
      *reinterpret_cast<float4*>(&us[k][4 * c4]) = v;
    }
    __syncthreads();
    for (int k = 0; k < kn; ++k) {
      float a[8], b[8];
      *reinterpret_cast<float4*>(&a[0]) = *reinterpret_cast<const float4*>(&es[k][4 * ty]);
      *reinterpret_cast<float4*>(&a[4]) = *reinterpret_cast<const float4*>(&es[k][64 + 4 * ty]);
      *reinterpret_cast<float4*>(&b[0]) = *reinterpret_cast<const float4*>(&us[k][4 * tx]);
      *reinterpret_cast<float4*>(&b[4]) = *reinterpret_cast<const float4*>(&us[k][64 + 4 * tx]);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = __fadd_rn(acc[i][j], __fmul_rn(a[i], b[j]));
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = r0 + (i < 4 ? 4 * ty + i : 64 + 4 * ty + i - 4);
    if (row >= n_out) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int col = c0 + 64 * h + 4 * tx;   // k_in and col are multiples of 4
      if (col >= k_in) continue;
      float4* wp = reinterpret_cast<float4*>(W + (size_t)row * k_in + col);
      float4 w = *wp;
      w.x = __fsub_rn(w.x, acc[i][4 * h + 0]);
      w.y = __fsub_rn(w.y, acc[i][4 * h + 1]);
      w.z = __fsub_rn(w.z, acc[i][4 * h + 2]);
      w.w = __fsub_rn(w.w, acc[i][4 * h + 3]);
      *wp = w;
    }
  }
}

// ------------------------------------------------------------ row-owner kernel
// The whole of the block loop for a group of up to NR rows by one CTA: every
// row's codes depend on that row and U alone, so nothing crosses CTAs and no
// launch separates the blocks.  Per block b of B columns F:
//   upsample   groups of 8 rows x parts of the sample pairs, a warp each
//              (tile_upsample: half of A_enc in shared memory; at B = 256 read
//              through the L1)
//   scan       the last warp, lane = row (eq. 8), the codes left in shared
//              memory as floats in place of the samples, sample-major
//   rebuild    s_k = sum_j c_j G[j][k], E = W_F - alpha s, behind the scan: a
//              warp 4 rows x all columns (lane: l + 32 q), one FMA per term
//              (c_j in {-1, 0, 1}: the product is exact, so fma(c, g, s) =
//              fl(s + fl(c g)))
//   solve      E~ = E U_FF^-1 by forward substitution, 32 columns at a time:
//              within them a lane has 4 columns of one row, so that one shuffle
//              and one quotient serve a warp's 4 rows, then their products come
//              off the later columns (31 -> 23 k cycles a block)
//   update     W_R -= E~ U_FR: thread = 4 columns x half of the rows, U from
//              the L2 with 8 rows' loads in flight (staged by cp.async it was
//              slower, 226 against 178 k cycles a block; so were 4 or 16 rows,
//              157 and 216 against 149: the loop's code grows with them), E~
//              broadcast from shared memory.  A broadcast 16-byte load still
//              returns 512 bytes to its warp, 4 cycles of the SM's one
//              shared-memory pipe: with 2 columns x all rows a thread that pipe
//              was as busy as the multiplies and adds
// The update's multiplies and adds bound it (no FMA: both are rounded), 155 of
// 218 k cycles a block of a 4096 x 4096 layer (100 + 8 at their issue rate, 133
// with every load of U an L1 hit); the steps before it are chains of dependent
// operations.  Two teams of rows per CTA, one's chains beside the other's
// update, took 330 k: single warps a quadrant wait on their own latencies.
// CTAs start at different column chunks: in step they all ask the same few L2
// lines at once (88 -> 72 k cycles a block of updates for 8 rows).  The launch
// per block and per update that this replaces took 12.6 ms for that layer, this
// 3.8; 2560 x 3584, B = 256, OSR 3: 21 and 4.8.
// W_F and W_R come from W itself at block 0 and from the working copy after
// it; the values and their order are those of a launch per block.
constexpr int kGqThreads = 256;
constexpr int kGqRp = 36;        // floats per sample / column of up to 32 rows (16-byte rows, 4-way bank spread)
constexpr int kCols = 2 * kGqThreads;   // columns of an update step
constexpr int kGqChunk = 32;     // rows of U_FF staged at a time

struct GptqParams {
  const float* W;
  float* wc;
  const float* U;
  const float* alpha;
  uint32_t* codes;
  const float* at;    // B x n_b
  const float* g32;   // n_b x B
  int n_out, k_in, B, n_b, nblk, wpr, quantizer;
  uint32_t pad0;
};

// Shared memory in floats: half the table (not for B = 256: read through the
// L1), weights, samples (later U_FF chunks), E~, a U_FF chunk, the diagonal and
// its reciprocals.
__host__ __device__ inline size_t gq_xs_floats(int B, int n_b) {
  const size_t a = (size_t)n_b * kGqRp, b = (size_t)kGqChunk * B;
  return a > b ? a : b;
}
__host__ __device__ inline size_t gq_smem_floats(int B, int n_b) {
  return (size_t)(B < 256 ? B : 0) * (n_b / 2) + 4 * tile_weight_floats(B) + gq_xs_floats(B, n_b) + (size_t)B * kGqRp +
         (size_t)kGqChunk * B + 2 * B;
}

// t / d given r = 1 / d correctly rounded (0 where |d| is outside [2^-30,
// 2^30]): a first quotient and two corrections by its exact remainder
// (Markstein, IBM J. Res. Dev. 34, 1990: the second starts within one unit in
// the last place of the quotient, so it ends correctly rounded).  *ok is
// cleared where something could over- or underflow.
__device__ __forceinline__ float quotient(float t, float d, float r, bool* ok) {
  *ok = *ok && r != 0.f && fabsf(t) >= 0x1p-60f && fabsf(t) <= 0x1p60f;
  float e = __fmul_rn(t, r);
#pragma unroll
  for (int n = 0; n < 2; ++n) e = __fmaf_rn(__fmaf_rn(-e, d, t), r, e);
  return e;
}

template <int NR, int QB, int PT>
__global__ void __launch_bounds__(kGqThreads, 1) gptq_rows_kernel(GptqParams p) {
  constexpr int kB = 32 * QB;              // block columns
  constexpr int kVg = (NR + 7) / 8;        // groups of 8 rows, 8 / kVg (rounded down) warps each for the upsampling
  constexpr int kHw = kVg == 3 ? 2 : 8 / kVg;
  constexpr bool kTable = kB < 256;
  extern __shared__ __align__(16) float smem[];
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int np = p.n_b / 2;
  float* ts = smem;
  float* wt = ts + (kTable ? (size_t)kB * np : 0);                  // 4 groups of 8 rows, transposed
  float* xs = wt + 4 * tile_weight_floats(kB);       // samples / codes [n_b][kGqRp]; then U_FF rows
  float* et = xs + gq_xs_floats(kB, p.n_b);          // E, then E~ [B][kGqRp]
  float* ub = et + kB * kGqRp;                       // U_FF rows
  float* dg = ub + kGqChunk * kB;                    // diagonal, reciprocals
  if constexpr (kTable) tile_load_table(ts, p.at, kB, p.n_b);
  const int ngroups = (p.n_out + NR - 1) / NR;
  const int vw = warp % kVg, hw = warp / kVg;   // (hw >= kHw: none)
  const size_t ldu = (size_t)p.k_in;

  for (int grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
    const int row0 = grp * NR, nr = min(NR, p.n_out - row0);
    for (int b = 0; b < p.nblk; ++b) {
      const float* wsrc = (b == 0 ? p.W : p.wc) + (size_t)row0 * p.k_in + (size_t)b * kB;
      const float* uff = p.U + (size_t)b * kB * ldu + (size_t)b * kB;
      __syncthreads();   // the update before (the working copy, E~) is done
      auto stage_u = [&](float* dst, int c) {   // U_FF rows 32 c .. 32 c + 31
        for (int i = tid; i < kGqChunk * (kB / 4); i += kGqThreads) {
          const int l = i / (kB / 4), k4 = i - l * (kB / 4);
          cp_async16(dst + l * kB + 4 * k4, uff + (size_t)(kGqChunk * c + l) * ldu + 4 * k4, 16);
        }
        cp_async_commit();
      };
      // The last block has no solve: staged for it too, the copies would still be
      // in flight when the next group of rows stages its first into the same rows
      // (asynchronous copies keep no order among them).
      const bool later = b != p.nblk - 1;
      if (later) {
        stage_u(ub, 0);
        if (tid < kB) {   // (kB at most kGqThreads)
          const float d = __ldg(uff + (size_t)tid * ldu + tid);
          dg[tid] = d;
          dg[kB + tid] = fabsf(d) >= 0x1p-30f && fabsf(d) <= 0x1p30f ? __frcp_rn(d) : 0.f;
        }
      }
      // the rows' weights, each warp a part of its 8 rows' columns
      if (hw < kHw) {
        const int r = 8 * vw + (lane >> 2);
        const float4* src = reinterpret_cast<const float4*>(wsrc + (size_t)min(r, nr - 1) * p.k_in);
        for (int k4 = (lane & 3) + 4 * hw; k4 < kB / 4; k4 += 4 * kHw) {
          const float4 w = r < nr ? __ldcg(src + k4) : make_float4(0.f, 0.f, 0.f, 0.f);
          float* d = wt + vw * tile_weight_floats(kB) + k4 * kWk4 + (lane >> 2);
          d[0] = w.x; d[8] = w.y; d[16] = w.z; d[24] = w.w;
        }
      }
      __syncthreads();
      if (hw < kHw && 8 * vw < nr)
        for (int jb = 32 * PT * hw; jb < np; jb += 32 * PT * kHw) {
          const int j0 = jb + lane, left = np - j0;
          const float* w8 = wt + vw * tile_weight_floats(kB);
          float acc[kTv][PT], acc2[kTv][PT];
          if constexpr (kTable) tile_upsample<PT>(ts + j0, np, left, w8, kB, acc, acc2);
          else tile_upsample<PT>(p.at + j0, p.n_b, left, w8, kB, acc, acc2);
#pragma unroll
          for (int q = 0; q < PT; ++q)
            if (32 * q < left) {
              float4* a = reinterpret_cast<float4*>(xs + (size_t)(j0 + 32 * q) * kGqRp + 8 * vw);
              float4* c = reinterpret_cast<float4*>(xs + (size_t)(np + j0 + 32 * q) * kGqRp + 8 * vw);
              a[0] = make_float4(acc[0][q], acc[1][q], acc[2][q], acc[3][q]);
              a[1] = make_float4(acc[4][q], acc[5][q], acc[6][q], acc[7][q]);
              c[0] = make_float4(acc2[0][q], acc2[1][q], acc2[2][q], acc2[3][q]);
              c[1] = make_float4(acc2[4][q], acc2[5][q], acc2[6][q], acc2[7][q]);
            }
        }
      __syncthreads();
      // The last warp scans in up to 4 parts; the other warps rebuild a part
      // while it scans the next ones.
      const int part = (p.n_b + 127) / 128 * 32;
      const int nmine = (nr + 3) / 4, scan_bar = 32 * (min(nmine, kGqThreads / 32 - 1) + 1);
      if (warp == kGqThreads / 32 - 1) {
        // Eq. (8); the codes replace the samples (rows past nr: zeros)
        const bool live = lane < nr;
        const float a = live ? p.alpha[row0 + lane] : 0.f, theta = 0.5f * a;
        float integ = 0.f, yp = 0.f;
        float* x = xs + lane;
        uint32_t* out = p.codes + (size_t)(row0 + lane) * p.wpr + (size_t)b * p.n_b * p.quantizer / 32;
        for (int j0 = 0, bar = 1; j0 < p.n_b; j0 += part, ++bar) {
          const int j1 = min(j0 + part, p.n_b);
          if (p.quantizer == SDQ_TERNARY) {
            for (int j = j0; j < j1; j += 16) {
              uint32_t cw = 0;
              float v[16];
#pragma unroll
              for (int i = 0; i < 16; ++i) v[i] = x[(size_t)(j + i) * kGqRp];
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const uint32_t f = sd_step<true>(integ, yp, v[i], a, theta);
                cw |= f << (2 * i);
                x[(size_t)(j + i) * kGqRp] = live ? (f == 1u ? 1.f : (f ? -1.f : 0.f)) : 0.f;
              }
              if (live) out[j / 16] = cw;
            }
          } else {
            for (int j = j0; j < j1; j += 32) {
              uint32_t cw = 0;
#pragma unroll
              for (int i = 0; i < 32; ++i) {
                const uint32_t f = sd_step<false>(integ, yp, x[(size_t)(j + i) * kGqRp], a, theta);
                cw |= f << i;
                x[(size_t)(j + i) * kGqRp] = live ? (f ? 1.f : -1.f) : 0.f;
              }
              if (live) out[j / 32] = cw;
            }
          }
          __syncwarp();
          if (later) named_bar_arrive(bar, scan_bar);
        }
        if (live && !later)   // the row's padding words
          for (int w = (int)p.pad0; w < p.wpr; ++w) p.codes[(size_t)(row0 + lane) * p.wpr + w] = 0u;
      }
      if (!later) break;
      // warp w's rows 4 w .. 4 w + 3, columns l + 32 q of lane l, in registers
      // from here to E~
      const bool mine = 4 * warp < nr;
      float t[4][QB];
      if (mine) {
        // s_k: one term per sample, in order, the next kGd samples' G in flight
        // (n_b is a multiple of 16)
        constexpr int kGd = QB < 8 ? 16 : 8;
        float gn[kGd][QB];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int q = 0; q < QB; ++q) t[i][q] = 0.f;
        const float* gk = p.g32 + lane;
#pragma unroll
        for (int j = 0; j < kGd; ++j)
#pragma unroll
          for (int q = 0; q < QB; ++q) gn[j][q] = __ldg(gk + j * kB + 32 * q);
        const float* c = xs + 4 * warp;
        int wait = 0, bar = 1;
#pragma unroll 1
        for (int j = 0; j < p.n_b; j += kGd, c += kGd * kGqRp) {
          if (j == wait) {   // the part that starts here is scanned
            if (warp != kGqThreads / 32 - 1) named_bar_sync(bar, scan_bar);
            ++bar;
            wait += part;
          }
          gk += kGd * kB;
          const bool more = j + kGd < p.n_b;
#pragma unroll
          for (int l = 0; l < kGd; ++l) {
            const float4 cv = *reinterpret_cast<const float4*>(c + l * kGqRp);
#pragma unroll
            for (int q = 0; q < QB; ++q) {
              t[0][q] = __fmaf_rn(cv.x, gn[l][q], t[0][q]);
              t[1][q] = __fmaf_rn(cv.y, gn[l][q], t[1][q]);
              t[2][q] = __fmaf_rn(cv.z, gn[l][q], t[2][q]);
              t[3][q] = __fmaf_rn(cv.w, gn[l][q], t[3][q]);
              if (more) gn[l][q] = __ldg(gk + l * kB + 32 * q);
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = 4 * warp + i;
          const float a = r < nr ? p.alpha[row0 + r] : 0.f;
#pragma unroll
          for (int q = 0; q < QB; ++q) {
            const int k = lane + 32 * q;
            const float w = wt[(r >> 3) * tile_weight_floats(kB) + (k >> 2) * kWk4 + (k & 3) * 8 + (r & 7)];
            // (1 in rows past the group's: no division by the slow way there)
            t[i][q] = r < nr ? __fsub_rn(w, __fmul_rn(a, t[i][q])) : 1.f;
          }
        }
      }
      // forward substitution, 32 rows of U_FF at a time, alternating buffers
#pragma unroll
      for (int c = 0; c < QB; ++c) {
        __syncthreads();   // the samples (c = 0) or the chunk before are used up
        if (c + 1 < QB) stage_u((c & 1) ? ub : xs, c + 1);
        if (c + 1 < QB) cp_async_wait_group<1>(); else cp_async_wait_group<0>();
        __syncthreads();
        if (!mine) continue;
        const float* u = (c & 1) ? xs : ub;
        // the chunk's columns by way of E~'s place in shared memory from lane =
        // column to lane = (4 columns, row), so that one shuffle and one quotient
        // serve the 4 rows
        *reinterpret_cast<float4*>(et + (size_t)(32 * c + lane) * kGqRp + 4 * warp) =
            make_float4(t[0][c], t[1][c], t[2][c], t[3][c]);
        __syncwarp();
        const int cg = lane >> 2;
        float* ec = et + (size_t)(32 * c + 4 * cg) * kGqRp + 4 * warp + (lane & 3);
        float tc[4];
        auto substitute = [&](auto fast) {
          bool ok = true;
#pragma unroll
          for (int j = 0; j < 4; ++j) tc[j] = ec[j * kGqRp];
#pragma unroll 2
          for (int l4 = 0; l4 < 8; ++l4) {
            const float4 d4 = *reinterpret_cast<const float4*>(dg + 32 * c + 4 * l4);
            const float4 r4 = *reinterpret_cast<const float4*>(dg + kB + 32 * c + 4 * l4);
            const float d[4] = {d4.x, d4.y, d4.z, d4.w}, r[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              const float4 u4 = *reinterpret_cast<const float4*>(u + (4 * l4 + m) * kB + 32 * c + 4 * cg);
              const float uv[4] = {u4.x, u4.y, u4.z, u4.w};
              const float tl = __shfl_sync(0xffffffffu, tc[m], 4 * l4 + (lane & 3));
              const float e = decltype(fast)::value ? quotient(tl, d[m], r[m], &ok) : __fdiv_rn(tl, d[m]);
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (cg > l4 || (j > m && cg == l4)) tc[j] = __fsub_rn(tc[j], __fmul_rn(e, uv[j]));
              if (cg == l4) tc[m] = e;
            }
          }
          return __all_sync(0xffffffffu, ok);
        };
        if (!substitute(std::true_type())) substitute(std::false_type());
#pragma unroll
        for (int j = 0; j < 4; ++j) ec[j * kGqRp] = tc[j];
        __syncwarp();
        // the later chunks' columns
        if (c + 1 < QB) {
#pragma unroll 8
          for (int l = 0; l < kGqChunk; ++l) {
            const float4 e = *reinterpret_cast<const float4*>(et + (size_t)(32 * c + l) * kGqRp + 4 * warp);
#pragma unroll
            for (int q = c + 1; q < QB; ++q) {
              const float uv = u[l * kB + 32 * q + lane];
              t[0][q] = __fsub_rn(t[0][q], __fmul_rn(e.x, uv));
              t[1][q] = __fsub_rn(t[1][q], __fmul_rn(e.y, uv));
              t[2][q] = __fsub_rn(t[2][q], __fmul_rn(e.z, uv));
              t[3][q] = __fsub_rn(t[3][q], __fmul_rn(e.w, uv));
            }
          }
        }
      }
      __syncthreads();
      // W_R -= E~ U_FR: a thread's 4 adjacent columns from ca, kN rows from r0
      const float* uf = p.U + (size_t)b * kB * ldu;
      auto columns = [&](int ca, auto rows, int r0) {
        constexpr int kN = decltype(rows)::value;
        constexpr int kD = kN > 4 ? 8 : 16;   // rows of U in flight: the L2's round trip under this load is over 1000 cycles
        auto get = [](const float4& v, int c) { return reinterpret_cast<const float*>(&v)[c]; };
        const float* wr = (b == 0 ? p.W : p.wc) + (size_t)(row0 + r0) * p.k_in + ca;
#pragma unroll
        for (int r = 0; r < kN; ++r)   // into the L2 by the time they are read
          if (r0 + r < nr) asm volatile("prefetch.global.L2 [%0];" ::"l"(wr + (size_t)r * p.k_in));
        const float* u0 = uf + ca;
        float acc[4][kN];
        float4 u[kD];
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int r = 0; r < kN; ++r) acc[c][r] = -0.0f;   // -0 + p == p: the first product is taken as is
#pragma unroll
        for (int i = 0; i < kD; ++i) u[i] = __ldg(reinterpret_cast<const float4*>(u0 + (size_t)i * ldu));
#pragma unroll 1
        for (int k = 0; k < kB; k += kD) {
          u0 += kD * ldu;
          // past the last row: its 8 again (a branch on the loads costs the loop 11 %)
          const size_t step = k + kD < kB ? ldu : 0;
          if (!step) u0 -= kD * ldu;
#pragma unroll
          for (int i = 0; i < kD; ++i) {
            const float4* e4 = reinterpret_cast<const float4*>(et + (size_t)(k + i) * kGqRp + r0);
#pragma unroll
            for (int r = 0; r < kN; r += 4) {
              const float4 e = e4[r / 4];
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                acc[c][r] = __fadd_rn(acc[c][r], __fmul_rn(e.x, get(u[i], c)));
                acc[c][r + 1] = __fadd_rn(acc[c][r + 1], __fmul_rn(e.y, get(u[i], c)));
                acc[c][r + 2] = __fadd_rn(acc[c][r + 2], __fmul_rn(e.z, get(u[i], c)));
                acc[c][r + 3] = __fadd_rn(acc[c][r + 3], __fmul_rn(e.w, get(u[i], c)));
              }
            }
            u[i] = __ldg(reinterpret_cast<const float4*>(u0 + (size_t)i * step));
          }
        }
        float* wo = p.wc + (size_t)(row0 + r0) * p.k_in + ca;
        // four rows' loads before their stores: a round trip per four rows, not
        // one per row (8192 x 8192: 29.2 ms, 26.0 so, 25.5 with the prefetch above;
        // all rows' loads first cost the loop above registers: 158 k cycles a block
        // against 149)
#pragma unroll
        for (int r4 = 0; r4 < kN; r4 += 4) {
          float4 w[4];
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (r0 + r4 + r < nr) w[r] = __ldcg(reinterpret_cast<const float4*>(wr + (size_t)(r4 + r) * p.k_in));
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            if (r0 + r4 + r >= nr) break;
            w[r].x = __fsub_rn(w[r].x, acc[0][r4 + r]);
            w[r].y = __fsub_rn(w[r].y, acc[1][r4 + r]);
            w[r].z = __fsub_rn(w[r].z, acc[2][r4 + r]);
            w[r].w = __fsub_rn(w[r].w, acc[3][r4 + r]);
            *reinterpret_cast<float4*>(wo + (size_t)(r4 + r) * p.k_in) = w[r];
          }
        }
      };
      // 512 columns at a time, the first kN0 rows by warps 0-3 and the others by
      // warps 4-7 (one of each on every SM quadrant); the rest in units of 128
      // columns x 4 rows, a warp each (columns are multiples of 4)
      const int cb = (b + 1) * kB, nfull = (p.k_in - cb) / kCols;
      auto full = [&](auto rows, int r0) {
        if (r0 >= nr) return;
        int g = nfull ? (int)blockIdx.x % nfull : 0;
        for (int n = 0; n < nfull; ++n) {
          columns(cb + kCols * g + 4 * (tid & (kGqThreads / 2 - 1)), rows, r0);
          if (++g == nfull) g = 0;
        }
      };
      constexpr int kN0 = NR > 16 ? 16 : NR / 2;
      if (warp < 4) full(std::integral_constant<int, kN0>(), 0);
      else full(std::integral_constant<int, NR - kN0>(), kN0);
      const int ce = cb + kCols * nfull, units = nmine * ((p.k_in - ce + 127) / 128);
      for (int n = warp; n < units; n += kGqThreads / 32) {
        const int ca = ce + 128 * (n / nmine) + 4 * lane;
        if (ca < p.k_in) columns(ca, std::integral_constant<int, 4>(), 4 * (n % nmine));
      }
    }
  }
}

using GptqKernel = void (*)(GptqParams);
// nq: 32-pair columns of the samples, PT at a time for each of a row group's warps.
template <int QB>
GptqKernel rows_kernel(int nr, int nq) {
  constexpr bool kWide = QB == 8;
  switch (nr) {
    case 8: return nq <= 4 && !kWide ? gptq_rows_kernel<8, QB, 1> : gptq_rows_kernel<8, QB, 1 + kWide>;
    case 16: return nq <= 4 && !kWide ? gptq_rows_kernel<16, QB, 1 + kWide> : gptq_rows_kernel<16, QB, 2>;
    case 28: return nq <= 4 && !kWide ? gptq_rows_kernel<28, QB, 2 + kWide> : gptq_rows_kernel<28, QB, 3>;
    default: return nq <= 4 && !kWide ? gptq_rows_kernel<32, QB, 2 + kWide> : gptq_rows_kernel<32, QB, 3>;
  }
}

// The row-owner kernel where it applies (*used = false otherwise): the
// half-shift table and whole words of codes per block as for the tile
// encoder, B = 64, 128 or 256.  Rows per CTA: the count with the least time
// over the waves, NR K / 2 multiply-add pairs per row and block column against
// the chains per block (in cycles, both measured).
cudaError_t launch_gptq_rows(const sdq_plan_s* pl, const float* W, const float* U, uint32_t* codes, const float* alpha,
                             float* wc, cudaStream_t st, bool* used) {
  const Geometry& g = pl->geo;
  const size_t smem = sizeof(float) * gq_smem_floats(g.block, g.n_b);
  *used = pl->half_shift && (g.block == 64 || g.block == 128 || g.block == 256) && g.n_b % 16 == 0 &&
          (g.n_b * g.bits) % 32 == 0 && smem <= 226 * 1024;
  if (!*used) return cudaSuccess;
  GptqParams p;
  p.W = W; p.wc = wc; p.U = U; p.alpha = alpha; p.codes = codes; p.at = pl->d_at; p.g32 = pl->d_g32;
  p.n_out = g.n_out; p.k_in = g.k_in; p.B = g.block; p.n_b = g.n_b; p.nblk = g.nblk; p.wpr = g.words_per_row;
  p.quantizer = pl->desc.quantizer;
  p.pad0 = (uint32_t)(g.k_eff * g.bits / 32);
  const int cand[4] = {32, 28, 16, 8};
  const int64_t sms = std::max(1, pl->sm_count);
  int nr = 32;
  double best = 0;
  for (int i = 0; i < 4; ++i) {
    const int64_t groups = (g.n_out + cand[i] - 1) / cand[i], waves = (groups + sms - 1) / sms;
    const double c = (double)waves * (g.block / 128.0) * (1.0 * cand[i] * g.k_in + 45000.0 * g.block / 128.0);
    if (i == 0 || c < best) {
      best = c;
      nr = cand[i];
    }
  }
  const int nq = (g.n_b / 2 + 31) / 32;
  GptqKernel kern = g.block == 256   ? rows_kernel<8>(nr, nq)
                    : g.block == 128 ? rows_kernel<4>(nr, nq)
                                     : rows_kernel<2>(nr, nq);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)std::min<int64_t>((g.n_out + nr - 1) / nr, sms), kGqThreads, smem, st>>>(p);
  return cudaGetLastError();
}

inline size_t align256(size_t v) { return (v + 255) / 256 * 256; }

}  // namespace

cudaError_t launch_gptq_update(const sdq_plan_s* pl, float* W, const float* et, const float* U, int b,
                               cudaStream_t st) {
  const Geometry& g = pl->geo;
  const int f0 = b * g.block, col0 = f0 + g.block;
  if (col0 >= g.k_in) return cudaSuccess;
  const dim3 grid((g.k_in - col0 + kUpT - 1) / kUpT, (g.n_out + kUpT - 1) / kUpT);
  if (grid.y > 65535) return cudaErrorInvalidConfiguration;
  gptq_update_kernel<<<grid, kUpThreads, 0, st>>>(W, et, U, g.n_out, g.k_in, g.block, f0, col0);
  return cudaGetLastError();
}

}  // namespace sdq

using namespace sdq;

extern "C" size_t sdq_gptq_workspace_bytes(sdq_plan p) {
  if (!p) return 0;
  const Geometry& g = p->geo;
  return align256(sizeof(float) * (size_t)g.n_out * g.k_in) + align256(sizeof(float) * (size_t)g.n_out * g.block);
}

extern "C" int sdq_encode_rows_gptq(sdq_plan p, const float* W, const float* U, uint32_t* codes_plain,
                                    float* alpha, void* ws, size_t ws_bytes, void* stream) {
  if (!p || !W || !U || !codes_plain || !alpha || !ws) return SDQ_ERR_INVALID_ARG;
  const uintptr_t mis = (reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(U) |
                         reinterpret_cast<uintptr_t>(codes_plain) | reinterpret_cast<uintptr_t>(alpha) |
                         reinterpret_cast<uintptr_t>(ws)) & 15u;
  if (mis) return SDQ_ERR_INVALID_ARG;
  const Geometry& g = p->geo;
  if (g.block % 4) return SDQ_ERR_UNSUPPORTED;
  if (ws_bytes < sdq_gptq_workspace_bytes(p)) return SDQ_ERR_WORKSPACE;
  const int dv = sdq_check_device(p);
  if (dv != SDQ_OK) return dv;
  cudaStream_t st = (cudaStream_t)stream;
  float* wc = static_cast<float*>(ws);
  float* et = reinterpret_cast<float*>(static_cast<uint8_t*>(ws) + align256(sizeof(float) * (size_t)g.n_out * g.k_in));
  // alpha from the original weights (pass 0 over every block)
  cudaError_t e = launch_encode_alpha(p, W, codes_plain, alpha, st);
  bool used = false;
  if (e == cudaSuccess) e = launch_gptq_rows(p, W, U, codes_plain, alpha, wc, st, &used);
  if (used || e != cudaSuccess) return e == cudaSuccess ? SDQ_OK : SDQ_ERR_CUDA;
  // a launch per block and one per update, on a copy of W
  e = cudaMemcpyAsync(wc, W, sizeof(float) * (size_t)g.n_out * g.k_in, cudaMemcpyDeviceToDevice, st);
  for (int b = 0; b < g.nblk && e == cudaSuccess; ++b) {
    e = launch_encode_range(p, wc, codes_plain, alpha, st, 1, 2, b, b + 1, U, et);
    if (e == cudaSuccess && b + 1 < g.nblk) e = launch_gptq_update(p, wc, et, U, b, st);
  }
  return e == cudaSuccess ? SDQ_OK : SDQ_ERR_CUDA;
}
