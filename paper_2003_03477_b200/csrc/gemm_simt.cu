// SIMT matrix products: float operands (the float path of the small configurations) on a pipelined kernel that takes one
// or two products per launch, and a plain kernel with arbitrary operand kinds for bf16 layers the tensor cores cannot take
// (unaligned or too narrow).
#include "gemm.cuh"
#include "profile.cuh"

namespace ss {

// ---------------------------------------------------------------------------------------------- float operands
// C[m, n] = sum_k A(m, k) * B(n, k) in fp32 FMAs, k ascending in one chain per output (so results do not depend on the
// tile).  The products of the float path are small: what bounded them was one round trip to memory per 16 k (a 256 x 64
// product over 144 k took 15 us, one of 1024 x 256 over 3000 k 190 us).  Here the operand tiles of four K steps of 32 are
// in flight at a time (cp.async, 16 bytes where the rows are aligned, else 4), and the tile size follows the number of
// tiles (gemm_f32).
// Either operand may be K-major (k contiguous) or MN-major (m or n contiguous); tiles keep that layout in shared memory:
// K-major rows of 32 k, 36 floats apart (128-bit reads of four k, rows a thread apart: no bank conflicts), MN-major rows
// of one k.
constexpr int kFK = 32, kFStages = 4, kFRow = kFK + 4;

__device__ __forceinline__ void cp_async16(void* dst, const void* src, int bytes) {   // bytes < 16: the rest is zero
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}

// Requests the tiles of an operand, rows [r0, r0 + R), one K step of 32 after the other; elements outside [0, rows) x [0, K)
// become zero.  The addresses of a thread's 16-byte pieces are computed once and then only advance.
template <int R, int NT>
struct TileLoader {
  static constexpr int kPieces = R * kFK / 4 / NT;
  const F32Operand& o;
  int r0, rows, K, k0 = 0;
  const float* src[kPieces];
  int bytes[kPieces];              // of a piece inside the matrix: K-major: 16 or 0 by its row; MN-major: by its columns
  __device__ __forceinline__ TileLoader(const F32Operand& op, int first, int n_rows, int n_k) : o(op), r0(first), rows(n_rows), K(n_k) {
#pragma unroll
    for (int i = 0; i < kPieces; ++i) {
      const int e = threadIdx.x + NT * i;
      const int r = o.k_major ? e / (kFK / 4) : 4 * (e % (R / 4)), k = o.k_major ? 4 * (e % (kFK / 4)) : e / (R / 4);
      src[i] = o.p + (o.k_major ? (int64_t)(r0 + r) * o.ld + k : (int64_t)k * o.ld + r0 + r);
      bytes[i] = o.k_major ? (r0 + r < rows ? 16 : 0) : max(0, min(16, 4 * (rows - r0 - r)));
    }
  }
  __device__ __forceinline__ void next(float* tile) {
    if (o.vec) {
#pragma unroll
      for (int i = 0; i < kPieces; ++i) {
        const int e = threadIdx.x + NT * i;
        if (o.k_major) {
          const int r = e / (kFK / 4), k = 4 * (e % (kFK / 4));
          const int n = min(bytes[i], max(0, 4 * (K - k0 - k)));
          cp_async16(tile + r * kFRow + k, n > 0 ? src[i] : o.p, n);
          src[i] += kFK;
        } else {
          const int n = k0 + e / (R / 4) < K ? bytes[i] : 0;
          cp_async16(tile + 4 * e, n > 0 ? src[i] : o.p, n);          // (k, r) -> k * R + r
          src[i] += (int64_t)kFK * o.ld;
        }
      }
    } else {
#pragma unroll 4
      for (int i = 0; i < 4 * kPieces; ++i) {
        const int e = threadIdx.x + NT * i;
        const int r = o.k_major ? e / kFK : e % R, k = o.k_major ? e % kFK : e / R;
        const bool in = r0 + r < rows && k0 + k < K;
        const int64_t at = o.k_major ? (int64_t)(r0 + r) * o.ld + k0 + k : (int64_t)(k0 + k) * o.ld + r0 + r;
        cp_async4(o.k_major ? tile + r * kFRow + k : tile + k * R + r, in ? o.p + at : o.p, in ? 4 : 0);
      }
    }
    k0 += kFK;
  }
};

// v[i][j] = element (slot i, k + j) of a tile, j < 4.  Slot i of thread coordinate x (of NX) stands for row x + NX * i of a
// K-major tile, x * T + i of an MN-major one.
template <bool KM, int T, int NX>
__device__ __forceinline__ int slot_row(int x, int i) { return KM ? x + NX * i : x * T + i; }
template <bool KM, int T, int NX>
__device__ __forceinline__ void read_frag(const float* tile, int x, int k, float (&v)[T][4]) {
  if (KM) {
#pragma unroll
    for (int i = 0; i < T; ++i) {
      const float4 q = *reinterpret_cast<const float4*>(tile + (x + NX * i) * kFRow + k);
      v[i][0] = q.x; v[i][1] = q.y; v[i][2] = q.z; v[i][3] = q.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float* p = tile + (k + j) * (NX * T) + x * T;
      if (T == 1) {
        v[0][j] = p[0];
      } else if (T == 4) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        v[0][j] = q.x; v[1][j] = q.y; v[2 % T][j] = q.z; v[3 % T][j] = q.w;
      } else {
        const float2 q = *reinterpret_cast<const float2*>(p);
        v[0][j] = q.x; v[1 % T][j] = q.y;
      }
    }
  }
}

// A warp covers 8 x TN columns and 4 x TM rows: its 128-bit reads of either operand are one pass over the banks.
template <int BM, int BN, int TM, int TN, bool AK, bool BK>
__device__ __forceinline__ void f32_tile(const F32Job& J, int m0, int n0, float* smem) {
  constexpr int NX = BN / TN, NY = BM / TM, NT = NX * NY, kA = BM * kFRow, kStage = (BM + BN) * kFRow;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tx = warp % (NX / 8) * 8 + (lane & 7), ty = warp / (NX / 8) * 4 + (lane >> 3);
  const int steps = (J.K + kFK - 1) / kFK;
  TileLoader<BM, NT> la(J.A, m0, J.M, J.K);
  TileLoader<BN, NT> lb(J.B, n0, J.N, J.K);
  auto request = [&](int s) {
    if (s < steps) {
      float* st = smem + (s % kFStages) * kStage;
      la.next(st);
      lb.next(st + kA);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int s = 0; s < kFStages - 1; ++s) request(s);
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
#pragma unroll 1
  for (int s = 0; s < steps; ++s) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kFStages - 2) : "memory");
    __syncthreads();                                       // step s is here, and everybody is done with the stage refilled next
    const float* at = smem + (s % kFStages) * kStage;
    const float* bt = at + kA;
    float a[2][TM][4], b[2][TN][4];                        // four k at a time, the next four on their way
    read_frag<AK, TM, NY>(at, ty, 0, a[0]);
    read_frag<BK, TN, NX>(bt, tx, 0, b[0]);
    request(s + kFStages - 1);
#pragma unroll
    for (int g = 0; g < kFK / 4; ++g) {                    // zeros beyond K add nothing
      if (g + 1 < kFK / 4) {
        read_frag<AK, TM, NY>(at, ty, 4 * g + 4, a[(g + 1) & 1]);
        read_frag<BK, TN, NX>(bt, tx, 4 * g + 4, b[(g + 1) & 1]);
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[g & 1][i][kk], b[g & 1][j][kk], acc[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + slot_row<AK, TM, NY>(ty, i);
    if (m >= J.M) continue;
    float v[TN];
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int n = n0 + slot_row<BK, TN, NX>(tx, j);
      v[j] = n < J.N ? epilogue_value(J.ep, acc[i][j], m, n) : 0.f;
    }
    const int n = n0 + tx * TN;                            // neighbouring columns on one side of lo_cols leave together
    float* const out = n < J.ep.lo_cols ? reinterpret_cast<float*>(J.ep.out_lo) + m * J.ep.ld_lo + n
                                        : J.ep.out_hi + m * J.ep.ld_hi + (n - J.ep.lo_cols);
    if (!BK && TN == 4 && n + 4 <= J.N && !J.ep.lo_bf16 && (J.ep.lo_cols & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15u) == 0) {
      *reinterpret_cast<float4*>(out) = make_float4(v[0], v[1 % TN], v[2 % TN], v[3 % TN]);
      continue;
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int nj = n0 + slot_row<BK, TN, NX>(tx, j);
      if (nj < J.N) epilogue_store(J.ep, v[j], m, nj);
    }
  }
}

template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__(BM / TM * (BN / TN))
gemm_f32_kernel(const __grid_constant__ F32Jobs jobs) {
  wait_for_previous_kernel();
  extern __shared__ __align__(16) float f32_smem[];
  if (jobs.clear && blockIdx.x == 0 && threadIdx.x < jobs.clear_words) jobs.clear[threadIdx.x] = 0;
  int j = 0;
  while (j + 1 < jobs.n && (int)blockIdx.x >= jobs.job[j + 1].tile0) ++j;
  const F32Job& J = jobs.job[j];
  const int t = (int)blockIdx.x - J.tile0, gx = (J.N + BN - 1) / BN;
  const int m0 = t / gx * BM, n0 = t % gx * BN;
  if (J.A.k_major) {
    if (J.B.k_major) f32_tile<BM, BN, TM, TN, true, true>(J, m0, n0, f32_smem);
    else f32_tile<BM, BN, TM, TN, true, false>(J, m0, n0, f32_smem);
  } else {
    if (J.B.k_major) f32_tile<BM, BN, TM, TN, false, true>(J, m0, n0, f32_smem);
    else f32_tile<BM, BN, TM, TN, false, false>(J, m0, n0, f32_smem);
  }
}

bool f32_operand(const Operand& o, F32Operand* f) {
  if (o.kind != OP_F32 || (o.s_k != 1 && o.s_row != 1)) return false;
  f->p = reinterpret_cast<const float*>(o.p);
  f->k_major = o.s_k == 1;
  f->ld = f->k_major ? o.s_row : o.s_k;
  f->vec = aligned16(o.p) && (f->ld & 3) == 0;
  return true;
}

template <int BM, int BN, int TM, int TN>
static ss_status launch_f32(F32Jobs& jobs, int blocks, cudaStream_t st) {
  constexpr size_t smem = (size_t)kFStages * (BM + BN) * kFRow * 4;
  static bool attr_set[64];
  int dev = 0;
  SS_CUDA(current_device(&dev));
  if (smem > 48 * 1024 && dev >= 0 && dev < 64 && !attr_set[dev]) {
    SS_CUDA(cudaFuncSetAttribute(gemm_f32_kernel<BM, BN, TM, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    attr_set[dev] = true;
  }
  SS_TIMED("gemm_f32_kernel", st);
  launch_dependent(gemm_f32_kernel<BM, BN, TM, TN>, blocks, BM / TM * (BN / TN), smem, st, jobs);
  SS_LAUNCH_OK();
  return SS_OK;
}

ss_status gemm_f32(F32Jobs& jobs, cudaStream_t st) {
  auto tiles = [&](int bm, int bn, bool place) {
    int64_t t = 0;
    for (int i = 0; i < jobs.n; ++i) {
      F32Job& J = jobs.job[i];
      if (place) J.tile0 = (int)t;
      t += (int64_t)((J.M + bm - 1) / bm) * ((J.N + bn - 1) / bn);
    }
    return t;
  };
  if (jobs.n < 1) return SS_OK;
  // Tiles as small as needed for every SM to have one: a K step of a 16 x 16 tile (128 threads, 1 x 2 outputs each) takes
  // about 800 cycles, of a 32 x 32 one (128 threads, 2 x 4) 1350, of a 64 x 64 one (256 threads, 4 x 4) 2400.  Measured, us
  // with 16 / 32 / 64: 78 x 176 over 3072 k 39 / 67 / 118; 1000 x 256 over 2976 k 140 / 99 / 119; 1000 x 2976 over 256 k
  // together with 256 x 2976 over 1000 k 281 / 150 / 121.
  int64_t blocks = tiles(64, 64, false);
  const bool large = blocks >= 4 * num_sms(), small = !large && tiles(32, 32, false) < num_sms();
  blocks = large ? tiles(64, 64, true) : (small ? tiles(16, 16, true) : tiles(32, 32, true));
  if (blocks > 0x7fffffff) return SS_ERR_SHAPE;
  if (large) return launch_f32<64, 64, 4, 4>(jobs, (int)blocks, st);
  if (small) return launch_f32<16, 16, 1, 2>(jobs, (int)blocks, st);
  return launch_f32<32, 32, 2, 4>(jobs, (int)blocks, st);
}

// ---------------------------------------------------------------------------------------------- any operand kinds
constexpr int kTM = 64, kTN = 64, kTK = 16;

template <int KIND>
__device__ __forceinline__ float load_op(const void* p, int64_t i) {
  if (KIND == OP_F32) return reinterpret_cast<const float*>(p)[i];
  if (KIND == OP_BF16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[i]);
  return __bfloat162float(__float2bfloat16_rn(reinterpret_cast<const float*>(p)[i]));
}

template <int KA, int KB>
__global__ void __launch_bounds__(256)
gemm_simt_kernel(int M, int N, int K, const void* __restrict__ A, int64_t sam, int64_t sak,
                 const void* __restrict__ B, int64_t sbn, int64_t sbk, Epilogue ep) {
  wait_for_previous_kernel();
  __shared__ float As[kTK][kTM + 4];
  __shared__ float Bs[kTK][kTN + 4];
  const int tid = threadIdx.x;
  const int m0 = blockIdx.y * kTM, n0 = blockIdx.x * kTN;
  const int ty = tid >> 4, tx = tid & 15;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

  for (int k0 = 0; k0 < K; k0 += kTK) {
    // stage the two operand tiles; the thread->element map follows the contiguous dimension
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int r, k;
      if (sak == 1) { r = (tid >> 4) + 16 * i; k = tid & 15; } else { r = tid & 63; k = (tid >> 6) + 4 * i; }
      const int gm = m0 + r, gk = k0 + k;
      As[k][r] = (gm < M && gk < K) ? load_op<KA>(A, (int64_t)gm * sam + (int64_t)gk * sak) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int r, k;
      if (sbk == 1) { r = (tid >> 4) + 16 * i; k = tid & 15; } else { r = tid & 63; k = (tid >> 6) + 4 * i; }
      const int gn = n0 + r, gk = k0 + k;
      Bs[k][r] = (gn < N && gk < K) ? load_op<KB>(B, (int64_t)gn * sbn + (int64_t)gk * sbk) : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kTK; ++k) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[k][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[k][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty * 4 + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n >= N) continue;
      epilogue_store(ep, epilogue_value(ep, acc[i][j], m, n), m, n);
    }
  }
}

ss_status gemm_simt(int M, int N, int K, const Operand& A, const Operand& B, const Epilogue& ep, cudaStream_t st) {
  if (M <= 0 || N <= 0) return SS_OK;
  F32Jobs jobs;
  if (jobs.add(M, N, K, A, B, ep)) return gemm_f32(jobs, st);
  dim3 grid((N + kTN - 1) / kTN, (M + kTM - 1) / kTM);
#define SS_GO(KA, KB)                                                                                         \
  launch_dependent(gemm_simt_kernel<KA, KB>, grid, 256, 0, st, M, N, K, A.p, A.s_row, A.s_k, B.p, B.s_row, B.s_k, ep)
  const int key = A.kind * 3 + B.kind;
  SS_TIMED("gemm_simt_kernel", st);
  switch (key) {
    case OP_F32 * 3 + OP_F32: SS_GO(OP_F32, OP_F32); break;
    case OP_BF16 * 3 + OP_BF16: SS_GO(OP_BF16, OP_BF16); break;
    case OP_F32_ROUND_BF16 * 3 + OP_BF16: SS_GO(OP_F32_ROUND_BF16, OP_BF16); break;
    case OP_BF16 * 3 + OP_F32_ROUND_BF16: SS_GO(OP_BF16, OP_F32_ROUND_BF16); break;
    default: return SS_ERR_DTYPE;
  }
#undef SS_GO
  SS_LAUNCH_OK();
  return SS_OK;
}

}  // namespace ss
