// GPTQ block compensation for the Sigma-Delta encoder (SDQ-LLM Algorithm 1:
// the outer loop over blocks of B columns, with the inverse Hessian H^-1 =
// (2 X X^T + lambda I)^-1 given through its upper Cholesky factor U,
// U^T U = H^-1).
//
// Blocks are encoded in order on a working copy of W.  After block b is
// encoded (encode_kernel, one block per launch), each row's block error E =
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
//              (tile_upsample: half of A_enc in shared memory)
//   scan       one warp, lane = row (eq. 8), the codes left in shared memory
//              as floats in place of the samples, sample-major
//   rebuild    s_k = sum_j c_j G[j][k], E = W_F - alpha s: a warp 4 rows x all
//              columns (lane: l + 32 q), one FMA per term (c_j in {-1, 0,
//              1}: the product is exact, so fma(c, g, s) = fl(s + fl(c g)))
//   solve      E~ = E U_FF^-1 by forward substitution on the same registers,
//              U_FF's rows staged 32 at a time
//   update     W_R -= E~ U_FR: thread = 4 columns x half of the rows, U from
//              the L2 with 8 rows' loads in flight (staged by cp.async it was
//              slower, 226 against 178 k cycles a block), E~ broadcast from
//              shared memory.  A broadcast 16-byte load still returns 512 bytes to
//              its warp, 4 cycles of the SM's one shared-memory pipe: with 2
//              columns x all rows a thread that pipe was as busy as the
//              multiplies and adds
// The update's multiplies and adds bound it (no FMA: both are rounded), 60 %
// of the time of a 4096 x 4096 layer; the steps before it are chains of
// dependent operations, 40 us a block.  CTAs start at different column
// chunks: in step they all ask the same few L2 lines at once (88 -> 72 k
// cycles a block of updates for 8 rows).  The launch per block and per update
// that this replaces took 12.6 ms for that layer, this 4.4.
// W_F and W_R come from W itself at block 0 and from the working copy after
// it; the values and their order are those of a launch per block.
constexpr int kGqThreads = 256;
constexpr int kGqRp = 36;        // floats per sample / column of up to 32 rows (16-byte rows, 4-way bank spread)
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

// Shared memory in floats: half table, weights, samples (later U_FF chunks),
// E~, a U_FF chunk, the diagonal and its reciprocals.
__host__ __device__ inline size_t gq_xs_floats(int B, int n_b) {
  const size_t a = (size_t)n_b * kGqRp, b = (size_t)kGqChunk * B;
  return a > b ? a : b;
}
__host__ __device__ inline size_t gq_smem_floats(int B, int n_b) {
  return (size_t)B * (n_b / 2) + 4 * tile_weight_floats(B) + gq_xs_floats(B, n_b) + (size_t)B * kGqRp +
         (size_t)kGqChunk * B + 2 * B;
}

// e[i] = t[i] / d, correctly rounded, given r = 1 / d correctly rounded (0
// where |d| is outside [2^-30, 2^30]): a first quotient and two corrections by
// its exact remainder (Markstein, IBM J. Res. Dev. 34, 1990: the second
// starts within one unit in the last place of the quotient, so it ends
// correctly rounded).  Where something could over- or underflow, the division
// itself.  The same for all lanes, so the branch is uniform.
__device__ __forceinline__ void quotients(const float (&t)[4], float d, float r, float (&e)[4]) {
  bool safe = r != 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) safe = safe && fabsf(t[i]) >= 0x1p-60f && fabsf(t[i]) <= 0x1p60f;
  if (safe) {
#pragma unroll
    for (int i = 0; i < 4; ++i) e[i] = __fmul_rn(t[i], r);
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) e[i] = __fmaf_rn(__fmaf_rn(-e[i], d, t[i]), r, e[i]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) e[i] = __fdiv_rn(t[i], d);
  }
}

template <int NR, int QB, int PT>
__global__ void __launch_bounds__(kGqThreads, 1) gptq_rows_kernel(GptqParams p) {
  constexpr int kB = 32 * QB;              // block columns
  constexpr int kVg = (NR + 7) / 8;        // groups of 8 rows, 8 / kVg (rounded down) warps each for the upsampling
  constexpr int kHw = kVg == 3 ? 2 : 8 / kVg;
  extern __shared__ __align__(16) float smem[];
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int np = p.n_b / 2;
  float* ts = smem;
  float* wt = ts + (size_t)kB * np;                  // 4 groups of 8 rows, transposed
  float* xs = wt + 4 * tile_weight_floats(kB);       // samples / codes [n_b][kGqRp]; then U_FF rows
  float* et = xs + gq_xs_floats(kB, p.n_b);          // E, then E~ [B][kGqRp]
  float* ub = et + kB * kGqRp;                       // U_FF rows
  float* dg = ub + kGqChunk * kB;                    // diagonal, reciprocals
  tile_load_table(ts, p.at, kB, p.n_b);
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
      stage_u(ub, 0);
      if (tid < kB) {
        const float d = __ldg(uff + (size_t)tid * ldu + tid);
        dg[tid] = d;
        dg[kB + tid] = fabsf(d) >= 0x1p-30f && fabsf(d) <= 0x1p30f ? __frcp_rn(d) : 0.f;
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
      if (hw < kHw && 8 * vw < nr && 32 * PT * hw < np) {
        const int j0 = 32 * PT * hw + lane, left = np - j0;
        float acc[kTv][PT], acc2[kTv][PT];
        tile_upsample<PT>(ts + j0, np, left, wt + vw * tile_weight_floats(kB), kB, acc, acc2);
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
      if (warp == 0) {
        // Eq. (8); the codes replace the samples (rows past nr: zeros)
        const bool live = lane < nr;
        const float a = live ? p.alpha[row0 + lane] : 0.f, theta = 0.5f * a;
        float integ = 0.f, yp = 0.f;
        float* x = xs + lane;
        uint32_t* out = p.codes + (size_t)(row0 + lane) * p.wpr + (size_t)b * p.n_b * p.quantizer / 32;
        if (p.quantizer == SDQ_TERNARY) {
          for (int j = 0; j < p.n_b; j += 16) {
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
          for (int j = 0; j < p.n_b; j += 32) {
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
        if (live && b == p.nblk - 1)   // the row's padding words
          for (int w = (int)p.pad0; w < p.wpr; ++w) p.codes[(size_t)(row0 + lane) * p.wpr + w] = 0u;
      }
      if (b == p.nblk - 1) break;   // no later columns
      __syncthreads();
      // warp w's rows 4 w .. 4 w + 3, columns l + 32 q of lane l, in registers
      // from here to E~
      const bool mine = 4 * warp < nr;
      float t[4][QB];
      if (mine) {
        // s_k: one term per sample, in order, the next 16 samples' G in flight
        // (n_b is a multiple of 16)
        float gn[16][QB];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int q = 0; q < QB; ++q) t[i][q] = 0.f;
        const float* gk = p.g32 + lane;
#pragma unroll
        for (int j = 0; j < 16; ++j)
#pragma unroll
          for (int q = 0; q < QB; ++q) gn[j][q] = __ldg(gk + j * kB + 32 * q);
        const float* c = xs + 4 * warp;
#pragma unroll 1
        for (int j = 0; j < p.n_b; j += 16, c += 16 * kGqRp) {
          gk += 16 * kB;
          const bool more = j + 16 < p.n_b;
#pragma unroll
          for (int l = 0; l < 16; ++l) {
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
#pragma unroll 4
        for (int l = 0; l < 32; ++l) {
          const float d = dg[32 * c + l], r = dg[kB + 32 * c + l];
          float uv[QB], tl[4], e[4];
#pragma unroll
          for (int q = c; q < QB; ++q) uv[q] = u[l * kB + 32 * q + lane];
#pragma unroll
          for (int i = 0; i < 4; ++i) tl[i] = __shfl_sync(0xffffffffu, t[i][c], l);
          quotients(tl, d, r, e);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float n0 = __fsub_rn(t[i][c], __fmul_rn(e[i], uv[c]));
            t[i][c] = lane > l ? n0 : (lane == l ? e[i] : t[i][c]);
#pragma unroll
            for (int q = c + 1; q < QB; ++q) t[i][q] = __fsub_rn(t[i][q], __fmul_rn(e[i], uv[q]));
          }
        }
      }
      if (mine) {
#pragma unroll
        for (int q = 0; q < QB; ++q)
          *reinterpret_cast<float4*>(et + (size_t)(lane + 32 * q) * kGqRp + 4 * warp) =
              make_float4(t[0][q], t[1][q], t[2][q], t[3][q]);
      }
      __syncthreads();
      // W_R -= E~ U_FR: a thread's kC adjacent columns from ca, kN rows from r0
      const float* uf = p.U + (size_t)b * kB * ldu;
      auto columns = [&](int ca, auto cols, auto rows, int r0) {
        constexpr int kC = decltype(cols)::value, kN = decltype(rows)::value;
        using Vec = std::conditional_t<kC == 4, float4, float>;
        auto get = [](const Vec& v, int c) { return reinterpret_cast<const float*>(&v)[c]; };
        const float* u0 = uf + ca;
        float acc[kC][kN];
        Vec u[8];   // U of 8 rows: the L2's round trip under this load is over 1000 cycles
#pragma unroll
        for (int c = 0; c < kC; ++c)
#pragma unroll
          for (int r = 0; r < kN; ++r) acc[c][r] = -0.0f;   // -0 + p == p: the first product is taken as is
#pragma unroll
        for (int i = 0; i < 8; ++i) u[i] = __ldg(reinterpret_cast<const Vec*>(u0 + (size_t)i * ldu));
#pragma unroll 1
        for (int k = 0; k < kB; k += 8) {
          u0 += 8 * ldu;
          const bool more = k + 8 < kB;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float4* e4 = reinterpret_cast<const float4*>(et + (size_t)(k + i) * kGqRp + r0);
#pragma unroll
            for (int r = 0; r < kN; r += 4) {
              const float4 e = e4[r / 4];
#pragma unroll
              for (int c = 0; c < kC; ++c) {
                acc[c][r] = __fadd_rn(acc[c][r], __fmul_rn(e.x, get(u[i], c)));
                acc[c][r + 1] = __fadd_rn(acc[c][r + 1], __fmul_rn(e.y, get(u[i], c)));
                acc[c][r + 2] = __fadd_rn(acc[c][r + 2], __fmul_rn(e.z, get(u[i], c)));
                acc[c][r + 3] = __fadd_rn(acc[c][r + 3], __fmul_rn(e.w, get(u[i], c)));
              }
            }
            if (more) u[i] = __ldg(reinterpret_cast<const Vec*>(u0 + (size_t)i * ldu));
          }
        }
        const float* wr = (b == 0 ? p.W : p.wc) + (size_t)(row0 + r0) * p.k_in + ca;
        float* wo = p.wc + (size_t)(row0 + r0) * p.k_in + ca;
#pragma unroll
        for (int r = 0; r < kN; ++r) {
          if (r0 + r >= nr) break;
          Vec w = __ldcg(reinterpret_cast<const Vec*>(wr + (size_t)r * p.k_in));
#pragma unroll
          for (int c = 0; c < kC; ++c)
            reinterpret_cast<float*>(&w)[c] = __fsub_rn(get(w, c), acc[c][r]);
          *reinterpret_cast<Vec*>(wo + (size_t)r * p.k_in) = w;
        }
      };
      // warps 0-3 the first kN0 rows, warps 4-7 the others (one of each on
      // every SM quadrant): 4 columns a thread, the last ones 1
      auto update = [&](auto rows, int r0) {
        if (r0 >= nr) return;
        constexpr int kHalf = kGqThreads / 2;
        const int i = tid & (kHalf - 1);
        const int cb = (b + 1) * kB, nfull = (p.k_in - cb) / (4 * kHalf);
        int g = nfull ? (int)blockIdx.x % nfull : 0;
        for (int n = 0; n < nfull; ++n) {
          columns(cb + 4 * kHalf * g + 4 * i, std::integral_constant<int, 4>(), rows, r0);
          if (++g == nfull) g = 0;
        }
        for (int c0 = cb + 4 * kHalf * nfull; c0 < p.k_in; c0 += kHalf)
          if (c0 + i < p.k_in) columns(c0 + i, std::integral_constant<int, 1>(), rows, r0);
      };
      constexpr int kN0 = NR > 16 ? 16 : NR / 2;
      if (warp < 4) update(std::integral_constant<int, kN0>(), 0);
      else update(std::integral_constant<int, NR - kN0>(), kN0);
    }
  }
}

using GptqKernel = void (*)(GptqParams);
// nq: 32-pair columns of the samples; every warp takes ceil(nq / kHw) of them.
template <int QB>
GptqKernel rows_kernel(int nr, int nq) {
  switch (nr) {
    case 8: return gptq_rows_kernel<8, QB, 1>;
    case 16: return nq <= 4 ? gptq_rows_kernel<16, QB, 1> : gptq_rows_kernel<16, QB, 2>;
    case 28: return nq <= 4 ? gptq_rows_kernel<28, QB, 2> : gptq_rows_kernel<28, QB, 3>;
    default: return nq <= 4 ? gptq_rows_kernel<32, QB, 2> : gptq_rows_kernel<32, QB, 3>;
  }
}

// The row-owner kernel where it applies (*used = false otherwise): the
// half-shift table and whole words of codes per block as for the tile
// encoder, B = 64 or 128.  Rows per CTA: the count with the least time over
// the waves, NR K / 2 multiply-add pairs per row and block column against a
// fixed part per block (in cycles, both measured).
cudaError_t launch_gptq_rows(const sdq_plan_s* pl, const float* W, const float* U, uint32_t* codes, const float* alpha,
                             float* wc, cudaStream_t st, bool* used) {
  const Geometry& g = pl->geo;
  const size_t smem = sizeof(float) * gq_smem_floats(g.block, g.n_b);
  *used = pl->half_shift && (g.block == 64 || g.block == 128) && g.n_b / 2 <= 192 && (g.n_b * g.bits) % 32 == 0 &&
          smem <= 226 * 1024;
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
    const double c = (double)waves * (1.2 * cand[i] * g.k_in * g.block / 128.0 + 40000.0);
    if (i == 0 || c < best) {
      best = c;
      nr = cand[i];
    }
  }
  const int nq = (g.n_b / 2 + 31) / 32;
  GptqKernel kern = g.block == 128 ? rows_kernel<4>(nr, nq) : rows_kernel<2>(nr, nq);
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
