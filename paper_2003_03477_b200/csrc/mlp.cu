// Bottom MLP -> concat -> top MLP -> sigmoid/BCE, its backward pass and the dense Adagrad update.
#include <cooperative_groups.h>
#include <string.h>
#include "gemm.cuh"
#include "profile.cuh"
#include "mlp.cuh"
#include "mlp_plan.cuh"

namespace ss {

// ---------------------------------------------------------------------------------------------
// Reductions over the batch that are no dense contraction: bias gradients, the gradient of the
// single-logit layer and of the 13-input layer.  All have the form
//     out[c * s_cols + j] = sum_b M[b, c] * S[b, j]          (S absent: s_cols = 1, S = 1)
// One launch takes a list of such jobs.  A block owns 256 or 64 columns c and a slice of the batch; its 8
// row groups add their rows in ascending order, the groups are added in order, and a second kernel
// adds the slices in order: every sum has a fixed association.
// What bounds it is the latency of a block's loads, so a thread keeps 8 rows (of 8 columns) or 16 rows (of one or two) in flight:
// with 4 it took 13.8 / 34 us (the sums of the 2048- and the 4096-sample model), with 8 and 16 rows 8.5 / 28.  Where the first
// layer's gradients are bf16, a thread takes two columns of them (a row of S read from shared memory serves both; its loads start
// while the S tile is filled) and all threads add the row groups: half as many blocks, of which two fit beside a tensor-core CTA
// (its 21 504 registers and theirs of 20 480).  28 -> 24 us for the 4096-sample model, the same for the other, but four replicas of
// it take 455 us a round instead of 460.  Three blocks per SM leave a thread 80 registers, which costs 12 bytes of spills; without
// them, the job's fields read from shared memory at each use, a pass takes 0.3 us more.  A block's job is found by one thread and
// read from shared memory: read by every thread from the list itself, where only the kernel's parameters hold it, forward and
// backward of 320-256-1 behind 13-512-64 took 57 us instead of 55 at 2048 samples.
// ---------------------------------------------------------------------------------------------
constexpr int kMaxJobs = 2 * kMaxLayers + 2;
constexpr int kMaxSCols = 16;

struct RedJob {
  const void* M; const void* S;
  int64_t ldm, lds;
  int m_kind, s_kind;      // OperandKind
  int ncols, s_cols;
  int tile0;               // first column tile of this job in grid.x
  int part_off;            // offset of this job's outputs in a partial row
  int64_t out_off;         // offset into the flat gradient vector
};
struct RedJobs {
  RedJob job[kMaxJobs];
  int njobs, ntiles, total;   // total = outputs over all jobs
};

__device__ __forceinline__ float load_kind(const void* p, int kind, int64_t i) {
  if (kind == OP_BF16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[i]);
  const float v = reinterpret_cast<const float*>(p)[i];
  return kind == OP_F32 ? v : __bfloat162float(__float2bfloat16_rn(v));
}

constexpr int kRedRows = 256;     // most rows of the batch a block takes (bounds the staged S tile)
constexpr int kRedWide = 256;     // columns per block of a job without a second factor matrix (s_cols = 1)

// Eight consecutive elements M[row, c .. c+7] as floats; elements at or beyond ncols read as zero.  One
// 128-bit load (bf16) or two (float) when the address allows it, element loads otherwise.
__device__ __forceinline__ void load8_kind(const void* p, int kind, int64_t row, int64_t ld, int c, int ncols, bool vec_ok,
                                           float (&v)[8]) {
  if (vec_ok && c + 8 <= ncols) {
    if (kind == OP_BF16) {
      const uint4 q = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p) + row * ld + c);
      const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[2 * j] = __uint_as_float(w[j] << 16);                // a bf16 is the upper half of a float
        v[2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
      }
    } else {
      const float4* q = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p) + row * ld + c);
      const float4 a = q[0], b = q[1];
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
      if (kind == OP_F32_ROUND_BF16) {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = __bfloat162float(__float2bfloat16_rn(v[j]));
      }
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = (c + j < ncols) ? load_kind(p, kind, row * ld + c + j) : 0.f;
  }
}

// Rows ry, ry + 8, ... of C neighbouring columns, in ascending order, times the rows of S in s_tile: F rows in flight, the
// first ones while stage() fills s_tile.
template <int C, int F, typename Raw, typename Stage, typename Load, typename Value>
__device__ __forceinline__ void column_sums(const float* s_tile, int ry, int nrows, float2 (&acc)[C][kMaxSCols / 2], Stage stage, Load load,
                                            Value value) {
  Raw m[F];
  auto fetch = [&](int rr) {
#pragma unroll
    for (int u = 0; u < F; ++u) m[u] = rr + 8 * u < nrows ? load(rr + 8 * u) : Raw{};
  };
  fetch(ry);
  stage();
  for (int rr = ry; rr < nrows; rr += 8 * F) {
    if (rr != ry) fetch(rr);
#pragma unroll
    for (int u = 0; u < F; ++u) {
      if (rr + 8 * u >= nrows) break;
      float v[C];
      value(m[u], v);
      const float4* srow = reinterpret_cast<const float4*>(s_tile + (rr + 8 * u) * kMaxSCols);
#pragma unroll
      for (int q4 = 0; q4 < kMaxSCols / 4; ++q4) {
        const float4 sv = srow[q4];                            // one 128-bit broadcast read for four columns of S
#pragma unroll
        for (int h = 0; h < C; ++h) {
          acc[h][2 * q4] = fma2(make_float2(v[h], v[h]), make_float2(sv.x, sv.y), acc[h][2 * q4]);
          acc[h][2 * q4 + 1] = fma2(make_float2(v[h], v[h]), make_float2(sv.z, sv.w), acc[h][2 * q4 + 1]);
        }
      }
    }
  }
}

// kCols: columns a thread takes of a job with a second factor matrix, 2 where that job's gradients are bf16
template <int kCols>
__global__ void __launch_bounds__(256, 3)
batch_reduce_partial_kernel(const __grid_constant__ RedJobs jobs, int B, int rows_per_split, float* __restrict__ partial) {
  wait_for_previous_kernel();
  // S rows of this block's batch slice, as float; then the row groups' sums (8 x 256 or 8 x 32 x 17 floats)
  constexpr int kPartFloats = 8 * 32 * (kMaxSCols + 1);
  static_assert(kPartFloats >= kRedRows * kMaxSCols && kPartFloats >= 8 * kRedWide, "one buffer serves all three uses");
  __shared__ __align__(16) float s_tile[kPartFloats];
  __shared__ RedJob s_job;
  if (threadIdx.x == 0) {
    int j = 0;
    while (j + 1 < jobs.njobs && (int)blockIdx.x >= jobs.job[j + 1].tile0) ++j;
    s_job = jobs.job[j];
  }
  __syncthreads();
  const RedJob J = s_job;                                    // the job's fields in registers
  const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5;
  const int sc = J.s_cols;
  const int r0 = blockIdx.y * rows_per_split;
  const int r1 = min(B, r0 + rows_per_split);
  const int nrows = r1 - r0;

  if (sc == 1) {
    // ---- no second factor, or a single column of one (S[b]): a warp reads 256 consecutive columns of a row,
    // eight per lane; warp ry adds rows ry, ry+8, ... in ascending order, then the eight warps are added in order.
    const int c = ((int)blockIdx.x - J.tile0) * kRedWide + 8 * cx;
    const bool vec_ok = J.m_kind == OP_BF16 ? ((J.ldm & 7) == 0 && (reinterpret_cast<uintptr_t>(J.M) & 15u) == 0)
                                            : ((J.ldm & 3) == 0 && (reinterpret_cast<uintptr_t>(J.M) & 15u) == 0);
    float acc[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = 0.f;
    if (J.m_kind == OP_BF16 && vec_ok && c + 8 <= J.ncols) {
      // eight rows in flight per thread, kept as loaded: a block is a chain of load latencies (256 rows: four rounds)
      const __nv_bfloat16* M = reinterpret_cast<const __nv_bfloat16*>(J.M) + (int64_t)r0 * J.ldm + c;
      for (int rr = ry; rr < nrows; rr += 64) {
        uint4 q[8];
        float sv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int r = rr + 8 * u;
          q[u] = make_uint4(0u, 0u, 0u, 0u);
          sv[u] = 0.f;
          if (r < nrows) {
            q[u] = *reinterpret_cast<const uint4*>(M + (int64_t)r * J.ldm);
            sv[u] = J.S ? load_kind(J.S, J.s_kind, (int64_t)(r0 + r) * J.lds) : 1.f;
          }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const uint32_t w[4] = {q[u].x, q[u].y, q[u].z, q[u].w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {                        // a bf16 is the upper half of a float; x * 1 + a rounds as x + a
            acc[2 * j] = fmaf(__uint_as_float(w[j] << 16), sv[u], acc[2 * j]);
            acc[2 * j + 1] = fmaf(__uint_as_float(w[j] & 0xFFFF0000u), sv[u], acc[2 * j + 1]);
          }
        }
      }
    } else if (c < J.ncols) {
      for (int rr = ry; rr < nrows; rr += 32) {
        float m[4][8], sv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {                          // four rows in flight per thread
          const int r = rr + 8 * u;
          if (r < nrows) {
            load8_kind(J.M, J.m_kind, r0 + r, J.ldm, c, J.ncols, vec_ok, m[u]);
            sv[u] = J.S ? load_kind(J.S, J.s_kind, (int64_t)(r0 + r) * J.lds) : 1.f;
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) m[u][j] = 0.f;
            sv[u] = 0.f;
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (J.S) {
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] = fmaf(m[u][j], sv[u], acc[j]);
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] += m[u][j];
          }
        }
      }
    }
    float* part = s_tile;                                      // [8][256]
    float4* pw = reinterpret_cast<float4*>(part + ry * kRedWide + 8 * cx);
    pw[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    pw[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    __syncthreads();
    const int co = ((int)blockIdx.x - J.tile0) * kRedWide + (int)threadIdx.x;
    if (co < J.ncols) {
      float t = 0.f;
#pragma unroll
      for (int r = 0; r < 8; ++r) t += part[r * kRedWide + threadIdx.x];
      partial[(int64_t)blockIdx.y * jobs.total + J.part_off + co] = t;
    }
    return;
  }

  // ---- a second factor with several columns (the layer with few inputs): 32 or 64 columns c per block, one or two neighbours a
  // thread, which keeps one sum per column of S for each; a row of S read from shared memory serves both
  const int c0 = ((int)blockIdx.x - J.tile0) * 32 * kCols, c = c0 + kCols * cx;
  float2 acc[kCols][kMaxSCols / 2];
#pragma unroll
  for (int h = 0; h < kCols; ++h)
#pragma unroll
    for (int q = 0; q < kMaxSCols / 2; ++q) acc[h][q] = make_float2(0.f, 0.f);
  auto stage = [&] {
    // S rows as float, padded with zeros to kMaxSCols columns so that the inner product needs no column test
    for (int i = threadIdx.x; i < nrows * kMaxSCols; i += 256) {
      const int rr = i / kMaxSCols, q = i % kMaxSCols;
      s_tile[i] = q < sc ? load_kind(J.S, J.s_kind, (int64_t)(r0 + rr) * J.lds + q) : 0.f;
    }
    __syncthreads();
  };
  if constexpr (kCols == 1) {
    column_sums<1, 16, float>(
        s_tile, ry, nrows, acc, stage,
        [&](int r) { return c < J.ncols ? load_kind(J.M, J.m_kind, (int64_t)(r0 + r) * J.ldm + c) : 0.f; },
        [](float m, float (&v)[1]) { v[0] = m; });
  } else {                                                     // bf16, and a layer's width is a multiple of 8: pairs are whole and aligned
    const __nv_bfloat16* M = reinterpret_cast<const __nv_bfloat16*>(J.M) + (int64_t)r0 * J.ldm + c;
    column_sums<2, 16, uint32_t>(
        s_tile, ry, nrows, acc, stage,
        [&](int r) { return c < J.ncols ? *reinterpret_cast<const uint32_t*>(M + (int64_t)r * J.ldm) : 0u; },
        [](uint32_t w, float (&v)[2]) { v[0] = __uint_as_float(w << 16); v[1] = __uint_as_float(w & 0xFFFF0000u); });   // a bf16 is the upper half of a float
  }
  __syncthreads();                                             // the S tile is no longer read
  // of two columns a thread the even ones first, then the odd ones, in the same buffer
  float (*part)[32][kMaxSCols + 1] = reinterpret_cast<float (*)[32][kMaxSCols + 1]>(s_tile);   // [8][32][17]
  float* dst = partial + (int64_t)blockIdx.y * jobs.total + J.part_off;
#pragma unroll
  for (int h = 0; h < kCols; ++h) {
    if (h > 0) __syncthreads();
#pragma unroll
    for (int q = 0; q < kMaxSCols; ++q) part[ry][cx][q] = q & 1 ? acc[h][q >> 1].y : acc[h][q >> 1].x;
    __syncthreads();
    for (int i = threadIdx.x; i < 32 * sc; i += 256) {
      const int col = i / sc, q = i - col * sc, co = c0 + kCols * col + h;
      if (co >= J.ncols) break;
      float t = 0.f;
#pragma unroll
      for (int r = 0; r < 8; ++r) t += part[r][col][q];
      dst[(int64_t)co * sc + q] = t;
    }
  }
}

// The single-logit layer, the sigmoid and the loss in one launch:
//   logit[b] = sum_k X[b, k] * w[k] + bias;  prob[b] = sigmoid(logit[b]);
//   loss = mean_b( max(z,0) - z*y + log(1+exp(-|z|)) ).
// One warp per sample (eight consecutive k per lane and round, fixed shuffle tree); a block adds the loss terms of
// its eight samples in order and leaves the sum in part[block]; the block that draws the last ticket adds the
// blocks' sums in a fixed order (which block that is does not matter) and clears the ticket for the next call.
// back.dX given: the layer's backward pass at once, while the sample's activations are at hand (see LogitBack).
struct LogitBack {
  void* dz; void* dX;          // dz: [B]; dX: [B, K], both in the precision of X
};

// dz of a sample, as the later products read it; lane 0 stores it.
template <bool BF16>
__device__ __forceinline__ float store_dz(float prob, float label, int B, int b, bool writes, const LogitBack& o) {
  float d = (prob - label) / (float)B;
  if (BF16) {
    const __nv_bfloat16 dh = __float2bfloat16_rn(d);
    d = __bfloat162float(dh);
    if (writes) reinterpret_cast<__nv_bfloat16*>(o.dz)[b] = dh;
  } else if (writes) {
    reinterpret_cast<float*>(o.dz)[b] = d;
  }
  return d;
}

// dX[b, c .. c + 7] = d * w[c ..], gated by X[b, c ..] > 0.
template <bool BF16>
__device__ __forceinline__ void outer_mask8(float d, const void* w, const void* X, int64_t ldx, int b, int c, int K, void* dX) {
  if (BF16) {
    const uint4 xq = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(X) + (int64_t)b * ldx + c);
    const uint4 wq = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(w) + c);
    const uint32_t xw[4] = {xq.x, xq.y, xq.z, xq.w}, ww[4] = {wq.x, wq.y, wq.z, wq.w};
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float x0 = __uint_as_float(xw[j] << 16), x1 = __uint_as_float(xw[j] & 0xFFFF0000u);
      const float w0 = __uint_as_float(ww[j] << 16), w1 = __uint_as_float(ww[j] & 0xFFFF0000u);
      const float v0 = x0 > 0.f ? d * w0 : 0.f, v1 = x1 > 0.f ? d * w1 : 0.f;
      __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
      o[j] = *reinterpret_cast<uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(dX) + (int64_t)b * K + c) = make_uint4(o[0], o[1], o[2], o[3]);
  } else {
    const float4* xq = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(X) + (int64_t)b * ldx + c);
    const float4* wq = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(w) + c);
    float4* oq = reinterpret_cast<float4*>(reinterpret_cast<float*>(dX) + (int64_t)b * K + c);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 x = xq[h], ww = wq[h];
      oq[h] = make_float4(x.x > 0.f ? d * ww.x : 0.f, x.y > 0.f ? d * ww.y : 0.f, x.z > 0.f ? d * ww.z : 0.f,
                          x.w > 0.f ? d * ww.w : 0.f);
    }
  }
}

__global__ void __launch_bounds__(256)
logit_loss_kernel(const void* __restrict__ X, int x_kind, int64_t ldx, const void* __restrict__ w, int w_kind, int K,
                  const float* __restrict__ bias, const float* __restrict__ labels, int B, float* __restrict__ logit,
                  float* __restrict__ prob, float* __restrict__ loss, float* part, unsigned int* ticket, LogitBack back) {
  wait_for_previous_kernel();
  __shared__ float s_term[8];
  __shared__ float s_red[256];
  __shared__ int s_last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * 8 + warp;
  float s = 0.f;
  if (b < B) {
    const bool al_x = (reinterpret_cast<uintptr_t>(X) & 15u) == 0, al_w = (reinterpret_cast<uintptr_t>(w) & 15u) == 0;
    const bool vec_x = al_x && (x_kind == OP_BF16 ? (ldx & 7) == 0 : (ldx & 3) == 0);
    for (int k0 = 8 * lane; k0 < K; k0 += 256) {
      float xv[8], wv[8];
      load8_kind(X, x_kind, b, ldx, k0, K, vec_x, xv);
      load8_kind(w, w_kind, 0, 0, k0, K, al_w, wv);
#pragma unroll
      for (int j = 0; j < 8; ++j) s = fmaf(xv[j], wv[j], s);
    }
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  float d = 0.f;
  if (lane == 0) {
    float t = 0.f;
    if (b < B) {
      const float z = s + bias[0], y = labels[b];
      const float e = expf(-fabsf(z));
      const float pr = (z >= 0.f) ? 1.f / (1.f + e) : e / (1.f + e);
      logit[b] = z;
      prob[b] = pr;
      t = fmaxf(z, 0.f) - z * y + log1pf(e);
      if (back.dX) d = x_kind == OP_BF16 ? store_dz<true>(pr, y, B, b, true, back) : store_dz<false>(pr, y, B, b, true, back);
    }
    s_term[warp] = t;
  }
  if (back.dX) {
    d = __shfl_sync(0xffffffffu, d, 0);
    for (int c = 8 * lane; b < B && c < K; c += 256) {       // K is a multiple of 8: hidden widths are
      if (x_kind == OP_BF16) outer_mask8<true>(d, w, X, ldx, b, c, K, back.dX);
      else outer_mask8<false>(d, w, X, ldx, b, c, K, back.dX);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
#pragma unroll
    for (int r = 0; r < 8; ++r) t += s_term[r];
    part[blockIdx.x] = t;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  float a = 0.f;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += 256) a += __ldcg(part + i);
  s_red[threadIdx.x] = a;
  __syncthreads();
  for (int off = 128; off >= 1; off >>= 1) {
    if (threadIdx.x < off) s_red[threadIdx.x] += s_red[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    loss[0] = s_red[0] / (float)B;
    *ticket = 0u;
  }
}

// The backward of the single-logit layer with the loss gradient folded in:
//   dz[b] = (prob[b] - y[b]) / B   (rounded to bf16 in bf16 mode, and stored: the reductions read it)
//   dX[b, k] = dz[b] * w[k], gated by X[b, k] > 0.
// One thread per eight consecutive k of a row (K is a multiple of 8: hidden widths are).
template <bool BF16>
__global__ void __launch_bounds__(256)
dz_outer_mask_kernel(const float* __restrict__ prob, const float* __restrict__ labels, const void* __restrict__ w,
                     const void* __restrict__ X, int B, int K, LogitBack back) {
  wait_for_previous_kernel();
  const int kc = K >> 3;
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= (int64_t)B * kc) return;
  const int b = (int)(i / kc), c = (int)(i - (int64_t)b * kc) * 8;
  const float d = store_dz<BF16>(prob[b], labels[b], B, b, c == 0, back);
  outer_mask8<BF16>(d, w, X, K, b, c, K, back.dX);
}

// dz alone, as a [B, 1] gradient matrix (a single top layer: its input gradient is a product's).
template <bool BF16>
__global__ void dz_kernel(const float* __restrict__ prob, const float* __restrict__ labels, int B, LogitBack back) {
  wait_for_previous_kernel();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < B) store_dz<BF16>(prob[b], labels[b], B, b, true, back);
}

// Where the gradient of each parameter tensor is found when the update kernel runs.
//   GRAD_FLAT    in the flat gradient vector itself (a GEMM wrote it there)
//   GRAD_SLICES  nsplit K slices of a weight-gradient GEMM: src[off + z*stride + i]
//   GRAD_BATCH   nsplit batch slices of the batched reduction (bias, skinny weights): src[off + z*stride + i]
// Elements that belong to no tensor (pads of the layout) have gradient zero.
enum { GRAD_FLAT = 0, GRAD_SLICES = 1, GRAD_BATCH = 2 };
constexpr int kMaxGradRanges = 2 * kMaxLayers;
struct GradTable {
  int n;
  int64_t begin[kMaxGradRanges], end[kMaxGradRanges], off[kMaxGradRanges], stride[kMaxGradRanges];
  int kind[kMaxGradRanges], nsplit[kMaxGradRanges];
};

// Element-wise Adagrad over the flat parameter vector; refreshes the bf16 mirror.  The slices of a
// gradient are added in slice order.  A zero gradient (pads, dead units) leaves the element
// untouched.  g_out (nullable, may alias g) receives the assembled gradient.
// A thread owns two float4 positions, 256 apart; the parameter and accumulator loads of both go out
// before the gradient is looked up, so one round of memory latency covers all of a thread's loads.
constexpr int kAdaPerThread = 2;

__device__ __forceinline__ float4 assemble_grad(const GradTable& tab, int64_t i, const float* g, const float* __restrict__ gpart,
                                                const float* __restrict__ bpart) {
  const int64_t e = i * 4;
  float4 gv = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int t = 0; t < tab.n; ++t) {
    if (e >= tab.begin[t] && e < tab.end[t]) {               // tensors start on multiples of 32: no float4 straddles a start
      const int64_t rel = e - tab.begin[t];
      if (tab.kind[t] == GRAD_FLAT) {
        gv = reinterpret_cast<const float4*>(g)[i];
      } else if (tab.kind[t] == GRAD_SLICES) {               // sizes are multiples of 8: aligned float4 loads
        const float4* p = reinterpret_cast<const float4*>(gpart + tab.off[t] + rel);
        const int ns = tab.nsplit[t];
        const int64_t st4 = tab.stride[t] >> 2;
        gv = p[0];
        if (ns == 2) {
          const float4 q = p[st4];
          gv.x += q.x; gv.y += q.y; gv.z += q.z; gv.w += q.w;
        } else {
          for (int z = 1; z < ns; ++z) {
            const float4 q = p[(int64_t)z * st4];
            gv.x += q.x; gv.y += q.y; gv.z += q.z; gv.w += q.w;
          }
        }
      } else {                                               // any size: scalar loads, elements past the end stay zero
        const int64_t left = tab.end[t] - e;
        const float* p = bpart + tab.off[t] + rel;
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        for (int z = 0; z < tab.nsplit[t]; ++z) {
          const float* q = p + (int64_t)z * tab.stride[t];
#pragma unroll
          for (int k = 0; k < 4; ++k) if (k < left) v[k] += q[k];
        }
        gv = make_float4(v[0], v[1], v[2], v[3]);
      }
      break;
    }
  }
  return gv;
}

__global__ void __launch_bounds__(256)
adagrad_kernel(float* __restrict__ w, float* __restrict__ acc, const float* g, const float* __restrict__ gpart,
               const float* __restrict__ bpart, const __grid_constant__ GradTable tab,
               __nv_bfloat16* __restrict__ mirror, int64_t n4, float lr, float eps, float* g_out, int apply) {
  wait_for_previous_kernel();
  const int64_t i0 = (int64_t)blockIdx.x * (256 * kAdaPerThread) + threadIdx.x;
  float4 wv[kAdaPerThread], av[kAdaPerThread], gv[kAdaPerThread];
#pragma unroll
  for (int u = 0; u < kAdaPerThread; ++u) {
    const int64_t i = i0 + 256 * u;
    if (apply && i < n4) {
      wv[u] = reinterpret_cast<float4*>(w)[i];
      av[u] = reinterpret_cast<float4*>(acc)[i];
    }
  }
#pragma unroll
  for (int u = 0; u < kAdaPerThread; ++u) {
    const int64_t i = i0 + 256 * u;
    if (i < n4) gv[u] = assemble_grad(tab, i, g, gpart, bpart);
  }
#pragma unroll
  for (int u = 0; u < kAdaPerThread; ++u) {
    const int64_t i = i0 + 256 * u;
    if (i >= n4) continue;
    if (g_out) reinterpret_cast<float4*>(g_out)[i] = gv[u];
    if (!apply) continue;
#define SS_UPD(F)                                        \
    if (gv[u].F != 0.f) {                                \
      av[u].F = fmaf(gv[u].F, gv[u].F, av[u].F);         \
      wv[u].F -= lr * gv[u].F / (sqrtf(av[u].F) + eps);  \
    }
    SS_UPD(x) SS_UPD(y) SS_UPD(z) SS_UPD(w)
#undef SS_UPD
    reinterpret_cast<float4*>(w)[i] = wv[u];
    reinterpret_cast<float4*>(acc)[i] = av[u];
    if (mirror) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(wv[u].x, wv[u].y), hi = __floats2bfloat162_rn(wv[u].z, wv[u].w);
      uint2 r;
      r.x = *reinterpret_cast<uint32_t*>(&lo);
      r.y = *reinterpret_cast<uint32_t*>(&hi);
      reinterpret_cast<uint2*>(mirror)[i] = r;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// The layer that reads the dense features (at most 16 inputs) is no dense contraction either:
//   Y[b, o] = ReLU( sum_k bf16(x[b, k]) * W[o, k] + bias[o] ),   stored as bf16.
// A thread keeps the weights of eight consecutive outputs in registers (K 16-byte loads: the rows of W are K elements and
// K is a template parameter) and walks the rows of its block: per row K / 2 128-bit shared-memory broadcasts of the sample,
// 4 x K paired FMAs in ascending k, one 16-byte store and one byte of sign bits.  What bounds it is instruction issue:
// four outputs a thread took 19 us at 8191 x 13 -> 1024, eight take 12.
// Its first block clears the control words of the pass (the workspace arrives uninitialised).
// ---------------------------------------------------------------------------------------------
constexpr int kFewInputs = 16;
constexpr int kFewRows = 64;        // most samples per block
constexpr int kFewThreads = 128;

template <int K>
__global__ void __launch_bounds__(kFewThreads)
few_inputs_layer_kernel(const float* __restrict__ x, const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias,
                        int relu, int B, int N, __nv_bfloat16* __restrict__ Y, int64_t ldy, int rows_per_block,
                        uint8_t* __restrict__ bits /*one bit per output "positive", rows of ld_bits bytes*/,
                        int64_t ld_bits, int* __restrict__ ctl, int ctl_words) {
  wait_for_previous_kernel();
  constexpr int KP = (K + 1) & ~1;
  __shared__ __align__(16) float2 s_x[kFewRows][KP];         // the block's samples, rounded to bf16; each value twice
  const int b0 = blockIdx.x * rows_per_block;
  const int rows = min(rows_per_block, B - b0);
  if (blockIdx.x == 0 && blockIdx.y == 0)
    for (int i = threadIdx.x; i < ctl_words; i += kFewThreads) ctl[i] = 0;
  for (int i = threadIdx.x; i < rows * KP; i += kFewThreads) {
    const int r = i / KP, k = i - r * KP;
    const float v = k < K ? __bfloat162float(__float2bfloat16_rn(x[(int64_t)(b0 + r) * K + k])) : 0.f;
    s_x[r][k] = make_float2(v, v);
  }
  const int n8 = N >> 3;                                     // octets of outputs
  const int q0 = blockIdx.y * kFewThreads, q_blk = min(n8 - q0, kFewThreads);
  const int groups = kFewThreads / q_blk;                    // row groups of the block
  const int grp = threadIdx.x / q_blk, q = q0 + threadIdx.x - grp * q_blk;
  const bool active = grp < groups;
  float2 w[4][K];                                            // outputs (0, 1), (2, 3), (4, 5), (6, 7)
  float bv[8];
  if (active) {
    uint32_t raw[4 * K];                                     // 8 rows of K bf16
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(W + (int64_t)8 * q * K) + i);   // tensors start on multiples of 32 elements
      raw[4 * i] = v.x; raw[4 * i + 1] = v.y; raw[4 * i + 2] = v.z; raw[4 * i + 3] = v.w;
    }
    auto weight = [&](int e) { return __uint_as_float((e & 1) ? raw[e >> 1] & 0xFFFF0000u : raw[e >> 1] << 16); };
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int k = 0; k < K; ++k) w[j][k] = make_float2(weight(2 * j * K + k), weight((2 * j + 1) * K + k));
#pragma unroll
    for (int j = 0; j < 8; ++j) bv[j] = bias[8 * q + j];
  }
  __syncthreads();
  if (!active) return;
  for (int r = grp; r < rows; r += groups) {
    float2 acc[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < K; k += 2) {
      const float4 xv = *reinterpret_cast<const float4*>(&s_x[r][k]);
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[j] = fma2(make_float2(xv.x, xv.y), w[j][k], acc[j]);
      if (k + 1 < K) {
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j] = fma2(make_float2(xv.z, xv.w), w[j][k + 1 < K ? k + 1 : 0], acc[j]);
      }
    }
    uint32_t out[4], pos = 0;
    const uint32_t zero = 0u;
    const __nv_bfloat162 z2 = *reinterpret_cast<const __nv_bfloat162*>(&zero);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float v0 = acc[j].x + bv[2 * j], v1 = acc[j].y + bv[2 * j + 1];
      if (relu) { v0 = fmaxf(v0, 0.f); v1 = fmaxf(v1, 0.f); }
      __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
      out[j] = *reinterpret_cast<uint32_t*>(&h);
      pos |= (__hgt2_mask(h, z2) & 0x00020001u) << (2 * j);  // column 2j at bit 2j, column 2j + 1 at bit 2j + 17
    }
    *reinterpret_cast<uint4*>(Y + (int64_t)(b0 + r) * ldy + 8 * q) = make_uint4(out[0], out[1], out[2], out[3]);
    bits[(int64_t)(b0 + r) * ld_bits + q] = (uint8_t)(pos | pos >> 16);
  }
}

// Collects the tensor-core products of a pass into flows (one persistent launch each, see gemm.cuh) and remembers
// which job of the open flow writes which tensor, so that a later product reading that tensor waits for its row
// blocks inside the launch instead of for a kernel boundary.
static_assert(kTcMaxFlow == kFlowProducts, "the control-word region of the workspace is sized for this many products per flow");
struct FlowBuilder {
  TcJob jobs[kTcMaxFlow];
  int n = 0;
  int writer[kMaxLayers];      // writer[l]: job of the open flow whose output is the tensor attached to layer l, or -1
  int* ctrl;
  int max_rows, sharers;
  cudaStream_t st;
  FlowBuilder(int* ctrl_, int max_rows_, int sharers_, cudaStream_t st_)
      : ctrl(ctrl_), max_rows(max_rows_), sharers(sharers_), st(st_) {
    for (int l = 0; l < kMaxLayers; ++l) writer[l] = -1;
  }
  // launches what has been collected; everything it writes is complete for whatever follows on the stream
  ss_status flush() {
    if (n == 0) return SS_OK;
    const ss_status r = gemm_tc_flow(jobs, n, (n == 1 && jobs[0].dep < 0) ? nullptr : ctrl, max_rows, sharers, st);
    n = 0;
    for (int l = 0; l < kMaxLayers; ++l) writer[l] = -1;
    return r;
  }
  // adds a job; `reads` is the layer whose tensor is its A operand (or -1); returns the job's index or a negative status
  int add(TcJob j, int reads, int dep_mode, int dep_k) {
    if (n == kTcMaxFlow) {
      const ss_status r = flush();
      if (r != SS_OK) return r;
    }
    if (reads >= 0 && writer[reads] >= 0) {
      j.dep = writer[reads]; j.dep_mode = dep_mode; j.dep_k = dep_k;
    }
    jobs[n] = j;
    return n++;
  }
};

// How layer l (not the last) of the forward pass is computed, and with which operands: the forward pass runs it, the
// backward pass asks the same question to know whether the layer left the sign bits of its output (bits[l]).
enum { FWD_FEW_INPUTS = 0, FWD_TENSOR_CORE = 1, FWD_SIMT = 2 };
struct FwdLayer { Operand A, Bm; Epilogue ep; int how; };
static FwdLayer describe_fwd_layer(const MlpPlan& p, int l, int B, const float* w, const void* w_bf16, const float* dense,
                                   const float* concat_f32, const void* concat_bf16, char* ws) {
  const LayerInfo& L = p.layer[l];
  const int act_kind = p.bf16 ? OP_BF16 : OP_F32;
  FwdLayer f;
  if (l == 0) f.A = Operand{dense, p.bf16 ? OP_F32_ROUND_BF16 : OP_F32, p.n_dense, 1};
  else if (l == p.nb) f.A = Operand{p.bf16 ? (const void*)concat_bf16 : (const void*)concat_f32, act_kind, p.W, 1};
  else f.A = Operand{ws + p.act[l - 1], act_kind, L.in, 1};
  f.Bm = p.bf16 ? Operand{reinterpret_cast<const __nv_bfloat16*>(w_bf16) + L.w_off, OP_BF16, L.in, 1}
                : Operand{w + L.w_off, OP_F32, L.in, 1};
  f.ep.bias = w + L.b_off;
  f.ep.relu = L.relu;
  f.ep.lo_cols = L.out;
  if (l == p.nb - 1) {
    f.ep.out_lo = p.bf16 ? const_cast<void*>(concat_bf16) : (void*)concat_f32; f.ep.lo_bf16 = p.bf16; f.ep.ld_lo = p.W;
  } else {
    f.ep.out_lo = ws + p.act[l]; f.ep.lo_bf16 = p.bf16; f.ep.ld_lo = L.out;
  }
  if (p.bf16 && l == 0 && L.in <= kFewInputs)
    f.how = FWD_FEW_INPUTS;
  else if (gemm_tc_eligible(B, L.out, L.in, f.A, f.Bm, f.ep))
    f.how = FWD_TENSOR_CORE;
  else
    f.how = FWD_SIMT;
  return f;
}

static ss_status check_common(const MlpPlan& p, int B, const void* concat_f32, const void* concat_bf16,
                              const void* w_bf16, void* ws, size_t ws_bytes) {
  if (B < 1) return SS_ERR_SHAPE;
  if (!ws) return SS_ERR_NULL;
  if (p.bf16 && (!concat_bf16 || !w_bf16)) return SS_ERR_DTYPE;
  if (!p.bf16 && !concat_f32) return SS_ERR_NULL;
  if (!aligned16(ws) || (concat_f32 && !aligned16(concat_f32)) || (concat_bf16 && !aligned16(concat_bf16)) ||
      (w_bf16 && !aligned16(w_bf16)))
    return SS_ERR_ALIGN;
  if (ws_bytes < p.total) return SS_ERR_WORKSPACE;
  return check_arch();
}

// The operands of the logit layer's backward pass.
static LogitBack logit_back(const MlpPlan& p, char* ws) {
  const int last = p.nl - 1;
  return LogitBack{ws + p.dact[last], last == p.nb ? nullptr : ws + p.dact[last - 1]};
}

ss_status mlp_fwd(const ss_mlp_desc* desc, const float* w, const void* w_bf16, const float* dense, float* concat_f32,
                  void* concat_bf16, int B, const float* labels, float* logit, float* prob, float* loss, void* workspace,
                  size_t workspace_bytes, ss_stream stream, const PassOptions& opt) {
  if (!w || !dense || !labels || !logit || !prob || !loss) return SS_ERR_NULL;
  MlpPlan p;
  ss_status st = make_mlp_plan(desc, B, &p);
  if (st != SS_OK) return st;
  st = check_common(p, B, concat_f32, concat_bf16, w_bf16, workspace, workspace_bytes);
  if (st != SS_OK) return st;
  if (!aligned16(w)) return SS_ERR_ALIGN;
  cudaStream_t cs = as_stream(stream);
  char* ws = reinterpret_cast<char*>(workspace);
  // the loss kernel's ticket and the control words of the tensor-core flows start at zero (the workspace arrives
  // uninitialised): the first layer's kernel clears them where it can, else clear_words; both clear themselves after use
  int* const ctl = reinterpret_cast<int*>(ws + p.ctrl);
  const int ctl_words = (int)(p.bf16 ? p.ctrl_bytes / 4 : kTicketWords);
  FlowBuilder flow(ctl + kTicketWords, p.ctrl_rows, opt.sharers, cs);

  for (int l = 0; l < p.nl; ++l) {
    const LayerInfo& L = p.layer[l];
    const FwdLayer f = describe_fwd_layer(p, l, B, w, w_bf16, dense, concat_f32, concat_bf16, ws);
    const Operand& A = f.A;
    const Operand& Bm = f.Bm;
    const Epilogue& ep = f.ep;
    if (l == 0 && f.how != FWD_FEW_INPUTS && p.bf16 && (st = clear_words(ctl, ctl_words, cs)) != SS_OK) return st;
    if (l == p.nl - 1) {   // one output unit: a dot product per sample
      st = flow.flush();
      if (st != SS_OK) return st;
      LogitBack back{};
      if (opt.logit_backward && l != p.nb) back = logit_back(p, ws);
      { SS_TIMED("logit_loss_kernel", cs);
      launch_dependent(logit_loss_kernel, (B + 7) / 8, 256, 0, cs, A.p, A.kind, A.s_row, Bm.p, Bm.kind, L.in, w + L.b_off, labels, B, logit,
                                                     prob, loss, reinterpret_cast<float*>(ws + p.loss_part),
                                                     reinterpret_cast<unsigned int*>(ctl), back);
      }
      SS_LAUNCH_OK();
      break;
    }
    if (f.how == FWD_FEW_INPUTS) {
      // about three blocks per SM, but at least 8 rows a thread where the batch allows it: a thread loads its weights first
      const int n8 = L.out / 8, q_blk = n8 < kFewThreads ? n8 : kFewThreads, groups = kFewThreads / q_blk;
      const int gy = (n8 + kFewThreads - 1) / kFewThreads;
      int rows = (B * gy + 3 * num_sms() - 1) / (3 * num_sms());
      if (rows < 8 * groups) rows = 8 * groups;
      if (rows > kFewRows) rows = kFewRows;
      const dim3 grid((B + rows - 1) / rows, gy);
      SS_TIMED("few_inputs_layer_kernel", cs);
#define SS_FEW(K_)                                                                                                     \
  case K_:                                                                                                             \
    launch_dependent(few_inputs_layer_kernel<K_>, grid, kFewThreads, 0, cs,                                                          \
        dense, reinterpret_cast<const __nv_bfloat16*>(w_bf16) + L.w_off, ep.bias, ep.relu, B, L.out,                   \
        reinterpret_cast<__nv_bfloat16*>(ep.out_lo), ep.ld_lo, rows, reinterpret_cast<uint8_t*>(ws + p.bits[l]),       \
        (int64_t)p.ld_bits[l] * 4, ctl, ctl_words);                                                                     \
    break
      switch (L.in) {
        SS_FEW(1); SS_FEW(2); SS_FEW(3); SS_FEW(4); SS_FEW(5); SS_FEW(6); SS_FEW(7); SS_FEW(8);
        SS_FEW(9); SS_FEW(10); SS_FEW(11); SS_FEW(12); SS_FEW(13); SS_FEW(14); SS_FEW(15); SS_FEW(16);
      }
#undef SS_FEW
      SS_LAUNCH_OK();
      continue;
    }
    if (f.how == FWD_TENSOR_CORE) {
      // The whole chain of tensor-core layers is ONE launch: layer l's tiles wait for the row blocks of layer l - 1
      // they read.  The first top layer reads the concat buffer, of which only the first D0 columns come from the
      // bottom MLP: it contracts the pooled embeddings first and waits for the bottom output only then.
      TcJob j;
      j.M = B; j.N = L.out; j.K = L.in; j.A = A; j.B = Bm; j.ep = ep;
      j.ep.bits_out = reinterpret_cast<uint32_t*>(ws + p.bits[l]);   // the backward pass masks with these
      j.ep.ld_bits_out = p.ld_bits[l];
      const int idx = flow.add(j, l - 1, 1, l == p.nb ? p.D0 : 0);
      if (idx < 0) return (ss_status)idx;
      flow.writer[l] = idx;
      continue;
    }
    st = flow.flush();
    if (st != SS_OK) return st;
    F32Jobs f32;
    if (f32.add(B, L.out, L.in, A, Bm, ep)) {
      if (l == 0) { f32.clear = ctl; f32.clear_words = ctl_words; }
      st = gemm_f32(f32, cs);
    } else {
      st = gemm_simt(B, L.out, L.in, A, Bm, ep, cs);
    }
    if (st != SS_OK) return st;
  }
  return SS_OK;
}

ss_status mlp_bwd(const ss_mlp_desc* desc, float* w, void* w_bf16, float* adagrad_acc, float* grads, const float* dense,
                  const float* concat_f32, const void* concat_bf16, const float* labels, const float* prob, int B, float lr,
                  float eps, int apply_update, float* grad_pooled, int64_t ld_grad, void* workspace, size_t workspace_bytes,
                  ss_stream stream, const PassOptions& opt) {
  if (!w || !dense || !labels || !prob || !grad_pooled) return SS_ERR_NULL;
  if (apply_update && !adagrad_acc) return SS_ERR_NULL;
  MlpPlan p;
  ss_status st = make_mlp_plan(desc, B, &p);
  if (st != SS_OK) return st;
  st = check_common(p, B, concat_f32, concat_bf16, w_bf16, workspace, workspace_bytes);
  if (st != SS_OK) return st;
  if (!aligned16(w) || (adagrad_acc && !aligned16(adagrad_acc)) || (grads && !aligned16(grads)) ||
      !aligned16(grad_pooled) || (ld_grad & 3))
    return SS_ERR_ALIGN;
  if (ld_grad < p.W - p.D0) return SS_ERR_SHAPE;
  if (!(lr >= 0.f) || !(eps >= 0.f)) return SS_ERR_RANGE;
  cudaStream_t cs = as_stream(stream);
  char* ws = reinterpret_cast<char*>(workspace);
  const int act_kind = p.bf16 ? OP_BF16 : OP_F32;
  float* g = grads ? grads : reinterpret_cast<float*>(ws + p.grads);

  const int last = p.nl - 1;
  const int dz_kind = p.bf16 ? OP_BF16 : OP_F32;
  const LogitBack back = logit_back(p, ws);
  if (last == p.nb) {   // a single top layer: its input gradient is a GEMM's; otherwise dz comes out of the fused kernel below
    SS_TIMED("dz_kernel", cs);
    if (p.bf16) launch_dependent(dz_kernel<true>, (B + 255) / 256, 256, 0, cs, prob, labels, B, back);
    else launch_dependent(dz_kernel<false>, (B + 255) / 256, 256, 0, cs, prob, labels, B, back);
  }
  SS_LAUNCH_OK();

  float* gpart = reinterpret_cast<float*>(ws + p.gpart);
  GradTable tab;
  memset(&tab, 0, sizeof(tab));                            // unused entries too: launches are compared byte by byte (step.cu)
  auto add_range = [&](int64_t begin, int64_t count, int kind, int64_t off, int64_t stride, int nsplit) {
    const int t = tab.n++;
    tab.begin[t] = begin; tab.end[t] = begin + count; tab.kind[t] = kind; tab.off[t] = off; tab.stride[t] = stride;
    tab.nsplit[t] = nsplit;
  };
  // Bias gradients and the first layer's and the logit layer's weight gradients are sums over the batch that are no dense
  // contraction; the batched reduction takes them.  (As products with a padded sample matrix inside the flow they cost 8 us
  // less for the ordinary model, but sum in another order: one float ulp in a parameter now and then moves its bf16 mirror
  // by an ulp, and the next step's ReLU gates with it.  The update is off the critical path of a step anyway.)
  RedJobs jobs;
  memset(&jobs, 0, sizeof(jobs));
  const int rows = ((B + p.red_splits - 1) / p.red_splits + 7) & ~7;   // <= kRedRows by the choice of red_splits
  const int nsplit = (B + rows - 1) / rows;
  // Columns a thread takes of the first layer's weight gradient.  Float rows are two loads for two columns, and the float model's
  // layers are narrow: one column (batch 1024, 64 wide 86.5 us for the pass, with two 89); bf16 pairs are one (87 and 82 us for the
  // 4096-sample model's).
  const int red_cols = p.bf16 ? 2 : 1;
  auto add_job = [&](const void* M, int m_kind, int64_t ldm, int ncols, const void* S, int s_kind, int64_t lds,
                     int s_cols, int64_t out_off) {
    RedJob& J = jobs.job[jobs.njobs++];
    J.M = M; J.m_kind = m_kind; J.ldm = ldm; J.ncols = ncols;
    J.S = S; J.s_kind = s_kind; J.lds = lds; J.s_cols = s_cols;
    J.tile0 = jobs.ntiles; J.part_off = jobs.total; J.out_off = out_off;
    jobs.ntiles += s_cols == 1 ? (ncols + kRedWide - 1) / kRedWide : (ncols + 32 * red_cols - 1) / (32 * red_cols);
    jobs.total += ncols * s_cols;
  };

  // All tensor-core products of the pass -- per layer the input gradient dX = dY W (which produces the next dY) and
  // the weight gradient dW = dY^T X -- form ONE flow, input gradient first: a product that reads a dY written inside
  // the flow waits for the row blocks it needs (dX by tile row, dW by k block, since it contracts over the batch).
  FlowBuilder flow(reinterpret_cast<int*>(ws + p.ctrl) + kTicketWords, p.ctrl_rows, opt.sharers, cs);   // writer[l]: the job that writes dact[l]
  for (int l = last; l >= 0; --l) {
    F32Jobs f32;
    const LayerInfo& L = p.layer[l];
    const void* G = ws + p.dact[l];
    // input of layer l
    Operand X;
    if (l == 0) X = Operand{dense, p.bf16 ? OP_F32_ROUND_BF16 : OP_F32, 1, p.n_dense};
    else if (l == p.nb) X = Operand{p.bf16 ? concat_bf16 : (const void*)concat_f32, act_kind, 1, p.W};
    else X = Operand{ws + p.act[l - 1], act_kind, 1, L.in};
    // dX[b, i] = sum_o G[b, o] * W[o, i], gated by the ReLU of the producing layer
    if (l == 0 || (l == last && l != p.nb && opt.logit_backward)) {
    } else if (l == last && l != p.nb) {
      const void* wl = p.bf16 ? (const void*)(reinterpret_cast<const __nv_bfloat16*>(w_bf16) + L.w_off) : (const void*)(w + L.w_off);
      const int64_t cnt = (int64_t)B * (L.in >> 3);            // L.in is a hidden width: a multiple of 8
      { SS_TIMED("dz_outer_mask_kernel", cs);
      if (p.bf16)
        launch_dependent(dz_outer_mask_kernel<true>, (unsigned)((cnt + 255) / 256), 256, 0, cs, prob, labels, wl, ws + p.act[l - 1], B, L.in, back);
      else
        launch_dependent(dz_outer_mask_kernel<false>, (unsigned)((cnt + 255) / 256), 256, 0, cs, prob, labels, wl, ws + p.act[l - 1], B, L.in, back);
      }
      SS_LAUNCH_OK();
    } else {
      Operand A{G, act_kind, L.out, 1};
      Operand Wt = p.bf16 ? Operand{reinterpret_cast<const __nv_bfloat16*>(w_bf16) + L.w_off, OP_BF16, 1, L.in}
                          : Operand{w + L.w_off, OP_F32, 1, L.in};
      Epilogue ep;
      ep.mask_bf16 = p.bf16;
      ep.out_lo = ws + p.dact[l - 1]; ep.lo_bf16 = p.bf16;
      if (l == p.nb) {
        ep.mask = p.bf16 ? concat_bf16 : (const void*)concat_f32; ep.ld_mask = p.W; ep.mask_cols = p.D0;
        ep.ld_lo = p.D0; ep.lo_cols = p.D0;
        ep.out_hi = grad_pooled; ep.ld_hi = ld_grad;
      } else {
        ep.mask = ws + p.act[l - 1]; ep.ld_mask = L.in; ep.mask_cols = L.in;
        ep.ld_lo = L.in; ep.lo_cols = L.in;
      }
      // the sign bits of the producing layer's output, where its forward kernel left them
      if (p.bf16 && describe_fwd_layer(p, l - 1, B, w, w_bf16, dense, concat_f32, concat_bf16, ws).how != FWD_SIMT) {
        ep.mask_bits = reinterpret_cast<const uint32_t*>(ws + p.bits[l - 1]);
        ep.ld_mask_bits = p.ld_bits[l - 1];
      }
      // On the tensor cores a product has one output matrix: below the concat buffer the columns of the bottom MLP (which
      // the rest of the pass waits for, so they come first) and those of the pooled embeddings are two products.
      const int n_lo = ep.lo_cols, n_hi = L.in - n_lo;
      Epilogue lo = ep, hi;
      lo.out_hi = nullptr;
      hi.out_lo = grad_pooled; hi.ld_lo = ld_grad; hi.lo_cols = n_hi;
      Operand Whi = Wt;
      Whi.p = reinterpret_cast<const char*>(Wt.p) + (size_t)n_lo * (p.bf16 ? 2 : 4);
      if (gemm_tc_eligible(B, n_lo, L.out, A, Wt, lo) && (n_hi == 0 || gemm_tc_eligible(B, n_hi, L.out, A, Whi, hi))) {
        TcJob j;
        j.M = B; j.N = n_lo; j.K = L.out; j.A = A; j.B = Wt; j.ep = lo;
        const int idx = flow.add(j, l, 1, 0);
        if (idx < 0) return (ss_status)idx;
        flow.writer[l - 1] = idx;
        if (n_hi > 0) {
          j.N = n_hi; j.B = Whi; j.ep = hi;
          const int i2 = flow.add(j, l, 1, 0);
          if (i2 < 0) return (ss_status)i2;
        }
      } else {
        st = flow.flush();
        if (st != SS_OK) return st;
        if (p.bf16 || !f32.add(B, L.in, L.out, A, Wt, ep)) {
          st = gemm_simt(B, L.in, L.out, A, Wt, ep, cs);
          if (st != SS_OK) return st;
        }
      }
    }
    // db[o] = sum_b G[b, o]
    add_job(G, act_kind, L.out, L.out, nullptr, 0, 0, 1, L.b_off);
    // dW[o, i] = sum_b G[b, o] * X[b, i]
    if (l == last) {
      add_job(X.p, X.kind, X.s_k, L.in, G, dz_kind, 1, 1, L.w_off);          // out = 1: dW[i] = sum_b X[b,i] dz[b]
    } else if (l == 0 && L.in <= kMaxSCols) {
      add_job(G, act_kind, L.out, L.out, X.p, X.kind, X.s_k, L.in, L.w_off);  // few inputs: dW[o, :] per column o
    } else {
      Operand A{G, act_kind, 1, L.out};
      Epilogue ep;
      ep.out_lo = g + L.w_off; ep.lo_bf16 = 0; ep.ld_lo = L.in; ep.lo_cols = L.in;
      if (gemm_tc_eligible(L.out, L.in, B, A, X, ep)) {
        // K = batch may be cut into slices; the update kernel adds them in slice order.
        const int64_t size = (int64_t)L.in * L.out;
        const int ks = p.k_splits[l];
        if (ks > 1) {
          ep.out_lo = gpart + p.gpart_off[l];
          add_range(L.w_off, size, GRAD_SLICES, p.gpart_off[l], size, ks);
        } else {
          add_range(L.w_off, size, GRAD_FLAT, 0, 0, 1);
        }
        TcJob j;
        j.M = L.out; j.N = L.in; j.K = B; j.A = A; j.B = X; j.ep = ep; j.k_splits = ks; j.split_stride = size;
        const int idx = flow.add(j, l, 2, 0);
        if (idx < 0) return (ss_status)idx;
      } else {
        st = flow.flush();
        if (st != SS_OK) return st;
        if (p.bf16 || !f32.add(L.out, L.in, B, A, X, ep)) {
          st = gemm_simt(L.out, L.in, B, A, X, ep, cs);
          if (st != SS_OK) return st;
        }
        add_range(L.w_off, (int64_t)L.in * L.out, GRAD_FLAT, 0, 0, 1);
      }
    }
    st = gemm_f32(f32, cs);                                  // float mode: both products of the layer side by side
    if (st != SS_OK) return st;
  }
  st = flow.flush();
  if (st != SS_OK) return st;
  if (opt.grads_ready) SS_CUDA(step_record(opt.grads_ready, cs));   // grad_pooled is complete
  float* partial = reinterpret_cast<float*>(ws + p.red_partial);
  if (jobs.njobs > 0) {
    // all batch reductions of the pass in one launch; the update kernel adds the batch slices
    { SS_TIMED("batch_reduce_partial_kernel", cs);
    launch_dependent(red_cols == 1 ? batch_reduce_partial_kernel<1> : batch_reduce_partial_kernel<2>, dim3(jobs.ntiles, nsplit), 256, 0,
                     cs, jobs, B, rows, partial);
    }
    SS_LAUNCH_OK();
    for (int j = 0; j < jobs.njobs; ++j)
      add_range(jobs.job[j].out_off, (int64_t)jobs.job[j].ncols * jobs.job[j].s_cols, GRAD_BATCH, jobs.job[j].part_off,
                jobs.total, nsplit);
  }
    const int64_t n4 = p.P / 4;
    SS_TIMED("adagrad_kernel", cs);
    launch_dependent(adagrad_kernel, (unsigned)((n4 + 256 * kAdaPerThread - 1) / (256 * kAdaPerThread)), 256, 0, cs, w, adagrad_acc, g, gpart, partial, tab,
                                                                 reinterpret_cast<__nv_bfloat16*>(w_bf16), n4, lr, eps,
                                                                 (grads || !apply_update) ? g : nullptr, apply_update);
    SS_LAUNCH_OK();
  return SS_OK;
}

}  // namespace ss

extern "C" {

int64_t ss_mlp_param_count(const ss_mlp_desc* desc) {
  ss::MlpPlan p;
  if (ss::make_mlp_plan(desc, 0, &p) != SS_OK) return -1;
  return p.P;
}

ss_status ss_mlp_param_offsets(const ss_mlp_desc* desc, int64_t* w_off, int64_t* b_off) {
  if (!w_off || !b_off) return SS_ERR_NULL;
  ss::MlpPlan p;
  ss_status st = ss::make_mlp_plan(desc, 0, &p);
  if (st != SS_OK) return st;
  for (int l = 0; l < p.nl; ++l) { w_off[l] = p.layer[l].w_off; b_off[l] = p.layer[l].b_off; }
  return SS_OK;
}

size_t ss_mlp_workspace_bytes(const ss_mlp_desc* desc, int B) {
  ss::MlpPlan p;
  if (ss::make_mlp_plan(desc, B, &p) != SS_OK) return 0;
  return p.total;
}

ss_status ss_mlp_fwd(const ss_mlp_desc* desc, const float* w, const void* w_bf16, const float* dense,
                     float* concat_f32, void* concat_bf16, int B, const float* labels, float* logit, float* prob,
                     float* loss, void* workspace, size_t workspace_bytes, ss_stream stream) {
  return ss::mlp_fwd(desc, w, w_bf16, dense, concat_f32, concat_bf16, B, labels, logit, prob, loss, workspace, workspace_bytes,
                     stream, ss::PassOptions());
}

ss_status ss_mlp_bwd(const ss_mlp_desc* desc, float* w, void* w_bf16, float* adagrad_acc, float* grads,
                     const float* dense, const float* concat_f32, const void* concat_bf16, const float* labels,
                     const float* prob, int B, float lr, float eps, int apply_update, float* grad_pooled,
                     int64_t ld_grad, void* workspace, size_t workspace_bytes, ss_stream stream) {
  return ss::mlp_bwd(desc, w, w_bf16, adagrad_acc, grads, dense, concat_f32, concat_bf16, labels, prob, B, lr, eps,
                     apply_update, grad_pooled, ld_grad, workspace, workspace_bytes, stream, ss::PassOptions());
}

// ---- normalised entropy (Section 4, "Evaluation Metrics") --------------------------------------
}  // extern "C"

namespace ss {
// acc[0] += sum_b cross-entropy(z_b, y_b), acc[1] += sum_b y_b, acc[2] += B; fixed tree, double.  One cluster of up to
// eight blocks (the double-precision logarithms are what takes the time: 9.4 us for 8191 samples in one block), whose sums
// the first block reads out of the others' shared memory.
__global__ void __launch_bounds__(1024)
ne_accumulate_kernel(const float* __restrict__ logit, const float* __restrict__ labels, int B, double* __restrict__ acc) {
  wait_for_previous_kernel();
  __shared__ double red[2][1024];
  double ce = 0.0, pos = 0.0;
  for (int b = blockIdx.x * 1024 + threadIdx.x; b < B; b += 1024 * gridDim.x) {
    const double z = logit[b], y = labels[b];
    ce += fmax(z, 0.0) - z * y + log1p(exp(-fabs(z)));
    pos += y;
  }
  red[0][threadIdx.x] = ce;
  red[1][threadIdx.x] = pos;
  __syncthreads();
  for (int off = 512; off >= 1; off >>= 1) {
    if (threadIdx.x < off) {
      red[0][threadIdx.x] += red[0][threadIdx.x + off];
      red[1][threadIdx.x] += red[1][threadIdx.x + off];
    }
    __syncthreads();
  }
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  cluster.sync();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    double c = red[0][0], p = red[1][0];
    for (unsigned r = 1; r < gridDim.x; ++r) {
      c += *cluster.map_shared_rank(&red[0][0], r);
      p += *cluster.map_shared_rank(&red[1][0], r);
    }
    acc[0] += c; acc[1] += p; acc[2] += (double)B;
  }
  cluster.sync();                                          // no block leaves while its sums may still be read
}

// NE = (mean cross-entropy) / (entropy of the empirical click rate p = acc[1]/acc[2])
__global__ void ne_value_kernel(const double* __restrict__ acc, double* __restrict__ out) {
  const double n = acc[2], p = acc[1] / n;
  out[0] = (acc[0] / n) / -(p * log(p) + (1.0 - p) * log(1.0 - p));
}
}  // namespace ss

extern "C" {

ss_status ss_ne_accumulate(const float* logit, const float* labels, int B, double* acc, ss_stream stream) {
  if (!logit || !labels || !acc) return SS_ERR_NULL;
  if (B < 1) return SS_ERR_SHAPE;
  if (reinterpret_cast<uintptr_t>(acc) & 7u) return SS_ERR_ALIGN;
  ss_status st = ss::check_arch();
  if (st != SS_OK) return st;
  SS_TIMED("ne_accumulate_kernel", ss::as_stream(stream));
  const int blocks = B >= 8 * 1024 ? 8 : (B + 1023) / 1024;
  ss::launch_cluster_dependent(ss::ne_accumulate_kernel, blocks, 1024, 0, blocks, ss::as_stream(stream), logit, labels, B, acc);
  SS_LAUNCH_OK();
  return SS_OK;
}

ss_status ss_ne_value(const double* acc, double* out, ss_stream stream) {
  if (!acc || !out) return SS_ERR_NULL;
  if ((reinterpret_cast<uintptr_t>(acc) | reinterpret_cast<uintptr_t>(out)) & 7u) return SS_ERR_ALIGN;
  ss_status st = ss::check_arch();
  if (st != SS_OK) return st;
  ss::ne_value_kernel<<<1, 1, 0, ss::as_stream(stream)>>>(acc, out);
  SS_LAUNCH_OK();
  return SS_OK;
}

}  // extern "C"
