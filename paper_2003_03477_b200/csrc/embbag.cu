// Embedding-bag forward (sum pooling) and the deterministic backward fused with row-wise Adagrad.
//
// Forward: a group of G = D/4 lanes owns one bag; every lane keeps one float4 column slice of the
// pooled vector in registers and walks the bag's rows with 128-bit loads (rows are D*4 contiguous
// bytes, so a group reads whole rows, fully coalesced).  Row loads of six lookups (four of
// wide rows) are issued together so several gathers are in flight per lane.
//
// Backward: (1-3) stable LSD radix sort by key t*N+row, unique keys and segment offsets, in one launch: ranges of each
// table in shared memory, or, for tables too long or too skewed for that, tiled passes over all SMs; (4) the sorted lookups are cut
// into windows of 16 consecutive positions; a lane group sums the gradients of each run of equal keys inside its window in position
// order.  A run that lies inside one window is final and is updated at once; a run that crosses a window edge leaves partial sums,
// added in window order by the group in which it starts, or by a second kernel where the run leaves the block or covers more than
// eight windows.  (Rows of more than 256 floats, and of more than 128 where windows are few or rows popular, are summed in memory
// and updated by a kernel of their own.)
// Work per group is the same whatever the skew of the row distribution, and every sum has a fixed
// association, so results do not depend on scheduling.
#include <type_traits>
#include "common.cuh"
#include "profile.cuh"

namespace ss {

// ======================================================================================
// forward
// ======================================================================================
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

__device__ __forceinline__ uint2 bf16x4(float4 v) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y);
  __nv_bfloat162 hi = __floats2bfloat162_rn(v.z, v.w);
  uint2 r;
  r.x = *reinterpret_cast<uint32_t*>(&lo);
  r.y = *reinterpret_cast<uint32_t*>(&hi);
  return r;
}

// G lanes per bag (power of two <= 32); NV float4 slices per lane (NV*G*4 >= D).
// Grid: x over the samples of a table (256 / G bags per block), y = table: no division finds (t, b), and all
// addressing inside a table is 32-bit (N * D / 4 < 2^32 is checked by the host).
template <int G, int NV>
__global__ void __launch_bounds__(256)
embbag_fwd_kernel(const float* __restrict__ tables, int T, uint32_t N, int D,
                  const int32_t* __restrict__ indices, const int32_t* __restrict__ offsets, int B,
                  float* __restrict__ out_f32, int64_t ld_f32,
                  __nv_bfloat16* __restrict__ out_bf16, int64_t ld_bf16, int col0,
                  int32_t* __restrict__ d_status) {
  wait_for_previous_kernel();
  const int b = blockIdx.x * (256 / G) + threadIdx.x / G;
  const int lane = threadIdx.x % G;
  const int t = blockIdx.y;
  if (b >= B) return;
  const int32_t* off = offsets + (int64_t)t * B + b;
  int lo = off[0], hi = off[1];
  // the index list ends where the last bag ends; a bag that is not inside [0, L] in ascending order is treated as empty
  const int L = __ldg(offsets + (int64_t)T * B);
  int bad = 0;
  if (lo < 0 || hi < lo || hi > L) { bad |= SS_DEV_BAD_OFFSET; lo = hi = 0; }
  const uint32_t nvec = (uint32_t)D >> 2;
  const float4* tab = reinterpret_cast<const float4*>(tables + (int64_t)t * N * D);

  float4 acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);

  // kRows lookups per round: their indices are loaded first, then their rows; a lookup beyond the bag's end or with
  // an index outside the table reads nothing and adds zeros.  Six rows (one float4 each) or four (two float4 each) in
  // flight per lane still fit 32 registers and were the fastest of 4 / 6 / 8 and 2 / 3 / 4.
  constexpr int kRows = NV >= 2 ? 4 : 6;
  for (int j = lo; j < hi; j += kRows) {
    uint32_t idx[kRows];
#pragma unroll
    for (int u = 0; u < kRows; ++u) idx[u] = (j + u < hi) ? (uint32_t)indices[j + u] : 0xffffffffu;
    float4 rowv[kRows][NV];
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const bool ok = idx[u] < N;                            // one unsigned compare: negative indices are huge
      if (!ok && j + u < hi) bad |= SS_DEV_BAD_INDEX;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const uint32_t c = lane + v * G;
        rowv[u][v] = (ok && c < nvec) ? __ldg(tab + (idx[u] * nvec + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int u = 0; u < kRows; ++u)      // lookups are added in bag order
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = add4(acc[v], rowv[u][v]);
  }

#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int c = lane + v * G;
    if (c < (int)nvec) {
      const int64_t col = (int64_t)col0 + (int64_t)t * D + 4 * c;
      if (out_f32) *reinterpret_cast<float4*>(out_f32 + (int64_t)b * ld_f32 + col) = acc[v];
      if (out_bf16) *reinterpret_cast<uint2*>(out_bf16 + (int64_t)b * ld_bf16 + col) = bf16x4(acc[v]);
    }
  }
  if (bad && d_status) atomicOr(d_status, bad);
}

// Rows of 65 to 256 floats, many bags: a block takes a stretch of consecutive bags, and the blocks that land on an SM at launch
// take neighbouring stretches, so an SM stays with one table and finds its popular rows in L1; with half of the threads there
// are enough registers for every row of a round to be in flight.  What bounds the form above there is the latency of rows from
// L2, half of which another SM has just read as well; narrower rows gain nothing (64 floats 28.7 -> 30 us, 16 floats 45 -> 47).
// Nothing evens the blocks out once they run, so a stretch is cut by work, not by bags.  us in a row, form above / equal numbers of
// bags / equal work, rows of 128 floats of 26 tables, batch 4096, ids of Zipf 1.05: 8 lookups a bag 55.6 / 41.9 / 43.4; one
// table 40 and the others 2 30.8 / 112 / 23.4; one twice the others 59.5 / 70 / 48.8; 1 to 100 by table 79 / 269 / 55; one
// lookup a bag 14.5 / 14.8 / 15.2 (batch 8191 34.6 / 36.0 / 30.7).  256 floats, 8 tables, batch 2048, 2 a bag: 6.3 / 8.7 / 8.0.
constexpr int kStretchThreads = 512, kStretchBlocks = 2;   // blocks per SM
constexpr uint32_t kBagWork = 3;                           // what a bag takes beside its lookups, in lookups (of 1 to 4)

// Bags [first, end) of stretch k of `stretches`: a stretch begins at the first bag i with offsets[i] + kBagWork * i at or above k
// equal shares of the whole.  Each half of the block looks for one end: among up to 1024 bags all at once, among more at 256
// places first (one load after the other; 1.3 us).  Whatever the offsets hold, a larger share is not found earlier, and the
// stretch before ends where this one begins: every bag is in one stretch.
__device__ __forceinline__ void stretch_of(int k, int stretches, const int32_t* __restrict__ offsets, uint32_t bags, uint32_t& first,
                                           uint32_t& end) {
  constexpr uint32_t kHalf = kStretchThreads / 2, kEach = 4, kWarps = kHalf / 32;
  __shared__ uint32_t s_below[2][2][kWarps], s_cut[2];
  const uint32_t half = threadIdx.x / kHalf, at = threadIdx.x % kHalf, lane = threadIdx.x & 31;
  const int32_t last = offsets[bags];
  uint32_t lo = 0, hi = bags, step;                        // the place is in [lo, hi]
  int round = 0;
  do {
    step = hi - lo > kEach * kHalf ? (hi - lo + kHalf - 1) / kHalf : 1u;
    int32_t value[kEach];
#pragma unroll
    for (uint32_t u = 0; u < kEach; ++u) {
      const uint32_t i = lo + (at + u * kHalf + 1) * step - 1;
      value[u] = i < hi ? offsets[i] : 0;
    }
    const uint64_t want = (uint64_t)((uint32_t)max(last, 0) + kBagWork * bags) * (uint32_t)(k + half);   // `stretches` times as much
    uint32_t below = 0;
#pragma unroll
    for (uint32_t u = 0; u < kEach; ++u) {
      if (lo + u * kHalf * step >= hi) break;              // (the same for all threads of the half)
      const uint32_t i = lo + (at + u * kHalf + 1) * step - 1;
      below += i < hi && (uint64_t)((uint32_t)max(value[u], 0) + kBagWork * i) * (uint32_t)stretches < want;
    }
    below = __reduce_add_sync(0xffffffffu, below);
    if (lane == 0) s_below[round & 1][half][at >> 5] = below;
    if (half == 0) asm volatile("bar.sync 1, %0;" ::"n"(kStretchThreads / 2) : "memory");
    else asm volatile("bar.sync 2, %0;" ::"n"(kStretchThreads / 2) : "memory");
    below = __reduce_add_sync(0xffffffffu, lane < kWarps ? s_below[round & 1][half][lane] : 0u);
    lo += below * step;
    hi = min(hi, lo + step - 1);
    ++round;
  } while (step > 1);
  if (at == 0) s_cut[half] = lo;
  __syncthreads();
  first = k > 0 ? s_cut[0] : 0u;
  end = k + 1 < stretches ? s_cut[1] : bags;
}

template <int G>
__global__ void __launch_bounds__(kStretchThreads, kStretchBlocks)
embbag_fwd_stretch_kernel(const float* __restrict__ tables, int T, uint32_t N, int D,
                          const int32_t* __restrict__ indices, const int32_t* __restrict__ offsets, int B,
                          float* __restrict__ out_f32, int64_t ld_f32,
                          __nv_bfloat16* __restrict__ out_bf16, int64_t ld_bf16, int col0,
                          int sms, int32_t* __restrict__ d_status) {
  wait_for_previous_kernel();
  constexpr int kGroups = kStretchThreads / G, NV = 2, kRows = 4;
  const int grp = threadIdx.x / G, lane = threadIdx.x % G;
  const uint32_t bags = (uint32_t)T * (uint32_t)B;
  uint32_t first, end;
  stretch_of((int)blockIdx.x % sms * kStretchBlocks + (int)blockIdx.x / sms, sms * kStretchBlocks, offsets, bags, first, end);
  const int L = __ldg(offsets + bags);
  const uint32_t nvec = (uint32_t)D >> 2;
  int t = (int)(first / (uint32_t)B), b = (int)(first % (uint32_t)B) + grp, bad = 0;
  // A lane group's bags of the stretch, P of them side by side.  (The round is written out: as a function that the other form
  // shares, the compiler makes 10 % more of it here, 43.4 -> 47 to 49 us.)
  auto sum_bags = [&](auto bags_at_once) {
    constexpr int P = decltype(bags_at_once)::value, kEach = kRows / P;
    for (uint32_t i = first + grp; i < end; i += P * kGroups, b += P * kGroups) {
      while (b >= B) { b -= B; ++t; }
      int lo[P], hi[P];
      float4 acc[P][NV];
#pragma unroll
      for (int p = 0; p < P; ++p) {
        lo[p] = hi[p] = 0;
        if (p == 0 || i + p * kGroups < end) {
          lo[p] = offsets[i + p * kGroups];
          hi[p] = offsets[i + p * kGroups + 1];
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[p][v] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      const float4* tab[P];
      int tp[P], bp[P];
#pragma unroll
      for (int p = 0; p < P; ++p) {
        tp[p] = t; bp[p] = b + p * kGroups;
        while (p > 0 && bp[p] >= B) { bp[p] -= B; ++tp[p]; }
        tab[p] = reinterpret_cast<const float4*>(tables + (int64_t)tp[p] * N * D);
        if (lo[p] < 0 || hi[p] < lo[p] || hi[p] > L) { bad |= SS_DEV_BAD_OFFSET; lo[p] = hi[p] = 0; }   // as above: an empty bag
      }
      while (lo[0] < hi[0] || (P > 1 && lo[P - 1] < hi[P - 1])) {
        uint32_t idx[P][kEach];
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
          for (int u = 0; u < kEach; ++u) idx[p][u] = (lo[p] + u < hi[p]) ? (uint32_t)__ldg(indices + lo[p] + u) : 0xffffffffu;
        float4 rowv[P][kEach][NV];
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
          for (int u = 0; u < kEach; ++u) {
            const bool ok = idx[p][u] < N;
            if (!ok && lo[p] + u < hi[p]) bad |= SS_DEV_BAD_INDEX;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
              const uint32_t c = lane + v * G;
              rowv[p][u][v] = (ok && c < nvec) ? __ldg(tab[p] + (idx[p][u] * nvec + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
          }
#pragma unroll
        for (int p = 0; p < P; ++p) {
#pragma unroll
          for (int u = 0; u < kEach; ++u)
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[p][v] = add4(acc[p][v], rowv[p][u][v]);
          lo[p] += kEach;
        }
      }
#pragma unroll
      for (int p = 0; p < P; ++p) {
        if (p > 0 && i + p * kGroups >= end) break;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int c = lane + v * G;
          if (c < (int)nvec) {
            const int64_t col = (int64_t)col0 + (int64_t)tp[p] * D + 4 * c;
            if (out_f32) *reinterpret_cast<float4*>(out_f32 + (int64_t)bp[p] * ld_f32 + col) = acc[p][v];
            if (out_bf16) *reinterpret_cast<uint2*>(out_bf16 + (int64_t)bp[p] * ld_bf16 + col) = bf16x4(acc[p][v]);
          }
        }
      }
    }
  };
  if (first >= end) return;
  // short bags: the latency of a bag's offsets, indices and rows is all there is (one lookup a bag: 16.4 -> 15.2 us, 37 -> 31)
  if (max(offsets[end], 0) - max(offsets[first], 0) <= 2 * (int64_t)(end - first)) sum_bags(std::integral_constant<int, 2>());
  else sum_bags(std::integral_constant<int, 1>());
  if (bad && d_status) atomicOr(d_status, bad);
}

template <int G, int NV>
static void launch_fwd(const float* tables, int T, int64_t N, int D, const int32_t* indices,
                       const int32_t* offsets, int B, float* out_f32, int64_t ld_f32, __nv_bfloat16* out_bf16,
                       int64_t ld_bf16, int col0, int32_t* d_status, cudaStream_t st) {
  // rows of 65..128 floats: two float4 per lane and 16 lanes per bag (measured faster than 32 lanes with one each;
  // for narrower rows the single-float4 form is the faster one)
  constexpr int FG = (NV == 1 && G == 32) ? 16 : G, FNV = (NV == 1 && G == 32) ? 2 : NV;
  if constexpr (FNV == 2) {
    // from the point on where the bags fill every SM once, two of them or more for a lane group of a stretch (and up to where
    // the work of all of them fits 32 bits)
    const int64_t bags = (int64_t)T * B;
    if (bags * FG >= 2048ll * num_sms() && bags < (1ll << 28)) {
      SS_TIMED("embbag_fwd_kernel", st);
      launch_dependent(embbag_fwd_stretch_kernel<FG>, (unsigned)(num_sms() * kStretchBlocks), kStretchThreads, 0, st, tables, T,
                       (uint32_t)N, D, indices, offsets, B, out_f32, ld_f32, out_bf16, ld_bf16, col0, num_sms(), d_status);
      return;
    }
  }
  const int per_block = 256 / FG;
  const dim3 blocks((unsigned)((B + per_block - 1) / per_block), (unsigned)T);
  { SS_TIMED("embbag_fwd_kernel", st);
  launch_dependent(embbag_fwd_kernel<FG, FNV>, blocks, 256, 0, st, tables, T, (uint32_t)N, D, indices, offsets, B, out_f32, ld_f32,
                                                      out_bf16, ld_bf16, col0, d_status);
  }
}

// ======================================================================================
// backward: keys, radix sort, unique, windowed segment reduction, row-wise Adagrad
// ======================================================================================
constexpr int kSortThreads = 256;
constexpr int kSortIPT = 16;                              // items per thread
constexpr int kSortTile = kSortThreads * kSortIPT;        // 4096 items per block
constexpr int kMaxBins = 512;
constexpr int kWin = 16;                                  // sorted positions per reduction window

// words of the control region: the bucket sort's fallback flag and tickets, the tiled sort's counters, the bucket counts
enum { kCtlFallback = 0, kCtlTicket = 1, kCtlTiled = 4, kCtlCounts = 8 };
constexpr int kBsMaxBuckets = 8;

constexpr int kListTicket = 5;                            // word of the scalars: blocks of the combine kernel that have read the list's length

struct BwdPlan {
  int64_t L;
  int nblk;          // sort tiles
  int bits, passes, digit_bits, bins;
  int nwin;
  size_t off_keys_a, off_keys_b, off_pos_a, off_pos_b, off_bag, off_hist, off_bintot, off_heads, off_uniq, off_seg,
      off_uidx, off_sbag, off_partial, off_long, off_gsum, off_scalars, off_ctl, total;
  size_t ctl_bytes;  // control words of the sort kernels, cleared before them: see kCtlFallback ...
};

static inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

static BwdPlan make_plan(int T, int64_t N, int D, int64_t L) {
  BwdPlan p{};
  p.L = L;
  p.nblk = (int)((L + kSortTile - 1) / kSortTile);
  if (p.nblk < 1) p.nblk = 1;
  const uint64_t maxkey = (uint64_t)T * (uint64_t)N;     // sentinel for skipped lookups
  p.bits = 1;
  while ((maxkey >> p.bits) != 0) ++p.bits;
  p.passes = (p.bits + 8) / 9;
  p.digit_bits = (p.bits + p.passes - 1) / p.passes;
  p.bins = 1 << p.digit_bits;
  p.nwin = (int)((L + kWin - 1) / kWin);
  if (p.nwin < 1) p.nwin = 1;
  size_t o = 0;
  const size_t l4 = align256((size_t)(L > 0 ? L : 1) * 4);
  p.off_keys_a = o; o += l4;
  p.off_keys_b = o; o += l4;
  p.off_pos_a = o; o += l4;
  p.off_pos_b = o; o += l4;
  p.off_bag = o; o += l4;
  p.off_hist = o; o += align256((size_t)p.nblk * p.bins * 4);
  p.off_bintot = o; o += align256((size_t)kMaxBins * 4);
  p.off_heads = o; o += align256((size_t)p.nblk * 4);
  p.off_uniq = o; o += l4;
  p.off_seg = o; o += align256((size_t)(L + 1) * 4);
  p.off_uidx = o; o += l4;
  p.off_sbag = o; o += l4;
  p.off_partial = o; o += align256((size_t)p.nwin * 2 * (size_t)D * 4);
  p.off_long = o; o += align256((size_t)p.nwin * 4);
  const uint64_t umax = (uint64_t)L < maxkey ? (uint64_t)L : maxkey;   // distinct rows cannot exceed either
  p.off_gsum = o; o += align256((size_t)(umax > 0 ? umax : 1) * (size_t)D * 4);
  p.off_scalars = o; o += 256;
  p.ctl_bytes = ((size_t)kCtlCounts + (size_t)T * kBsMaxBuckets) * 4;
  p.off_ctl = o; o += align256(p.ctl_bytes);
  p.total = o;
  return p;
}

// ---- (1) keys ---------------------------------------------------------------------------
// One thread per bag: key = t*N + row for each of its lookups, and the bag id of each position.
// Every position in [0, L) is written by somebody: a bag owns [lo, hi) with both ends clamped to
// [0, L] (consecutive bags share an end, so the clamped ranges tile [clamp(off[0]), clamp(off[T*B])) even
// when the offsets are not monotone), the first and the last bag also take what lies before and after.
// Positions of a malformed bag, and lookups with a row index outside the table, get the sentinel key.
template <int NT>
__device__ __forceinline__ void build_keys_block(int blk, const int32_t* __restrict__ indices,
                                                 const int32_t* __restrict__ offsets, int T, int64_t N, int B, int64_t L,
                                                 uint32_t* __restrict__ keys, int32_t* __restrict__ bag_of,
                                                 int32_t* __restrict__ d_status) {
  const int64_t bag = (int64_t)blk * NT + threadIdx.x;
  const int64_t nbags = (int64_t)T * B;
  if (bag >= nbags) return;
  const uint32_t sentinel = (uint32_t)((uint64_t)T * (uint64_t)N);
  const int t = (int)(bag / B);
  const int lo = offsets[bag], hi = offsets[bag + 1];
  const int64_t clo = lo < 0 ? 0 : (lo > L ? L : lo), chi = hi < 0 ? 0 : (hi > L ? L : hi);
  const bool well_formed = (lo == clo) && (hi == chi) && (lo <= hi);
  int bad = well_formed ? 0 : SS_DEV_BAD_OFFSET;
  for (int64_t j = clo; j < chi; ++j) {
    uint32_t key = sentinel;
    if (well_formed) {
      const int idx = indices[j];
      if (idx >= 0 && idx < N) key = (uint32_t)((uint64_t)t * (uint64_t)N + (uint64_t)idx);
      else bad |= SS_DEV_BAD_INDEX;
    }
    keys[j] = key;
    bag_of[j] = (int32_t)bag;
  }
  if (bag == 0) {
    if (lo != 0) bad |= SS_DEV_BAD_OFFSET;
    for (int64_t j = 0; j < clo; ++j) { keys[j] = sentinel; bag_of[j] = 0; }
  }
  if (bag == nbags - 1) {
    if (hi != L) bad |= SS_DEV_BAD_OFFSET;
    for (int64_t j = chi; j < L; ++j) { keys[j] = sentinel; bag_of[j] = 0; }
  }
  if (bad && d_status) atomicOr(d_status, bad);
}

// ---- (2) radix sort pass ----------------------------------------------------------------
// Lanes of the warp that hold the same digit, from one ballot per digit bit (cost independent of how many
// distinct digits the warp holds).  `digit` is below 2^nbits, or exactly 2^nbits for a lane past the end.
__device__ __forceinline__ uint32_t same_digit_lanes(uint32_t digit, int nbits) {
  uint32_t peers = 0xffffffffu;
  for (int b = 0; b <= nbits; ++b) {
    const bool bit = (digit >> b) & 1u;
    const uint32_t m = __ballot_sync(0xffffffffu, bit);
    peers &= bit ? m : ~m;
  }
  return peers;
}

// hist[bin * nblk + blk] = number of keys of tile blk whose digit is bin.  Lanes holding the same
// digit are counted together, so a hot row does not serialise on one counter.
// Reads of data that other blocks of the same launch may have written (the single-launch form below) bypass L1.
template <int NT>
__device__ __forceinline__ void sort_hist_block(int blk, uint32_t* cnt /*shared, kMaxBins*/, const uint32_t* keys, int64_t L,
                                                int shift, int bins, int nblk, uint32_t* hist) {
  for (int i = threadIdx.x; i < bins; i += NT) cnt[i] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t base = (int64_t)blk * (NT * kSortIPT);
  const uint32_t mask = (uint32_t)bins - 1u;
  const int nbits = 31 - __clz(bins);
  uint32_t digit[kSortIPT];
#pragma unroll
  for (int k = 0; k < kSortIPT; ++k) {                      // all loads first, then the counting
    const int64_t i = base + (int64_t)k * NT + threadIdx.x;
    digit[k] = (i < L) ? ((__ldcg(keys + i) >> shift) & mask) : (uint32_t)bins;
  }
#pragma unroll
  for (int k = 0; k < kSortIPT; ++k) {
    const uint32_t peers = same_digit_lanes(digit[k], nbits);
    if (digit[k] < (uint32_t)bins && lane == (__ffs(peers) - 1))
      atomicAdd(&cnt[digit[k]], (uint32_t)__popc(peers));   // integer counts: order-free
  }
  __syncthreads();
  for (int i = threadIdx.x; i < bins; i += NT) hist[(int64_t)i * nblk + blk] = cnt[i];
}

// One warp per bin: exclusive scan of that bin's per-tile counts in place, bin total to bintot[bin].
template <int NT>
__device__ __forceinline__ void bin_scan_block(int blk, uint32_t* hist, int bins, int nblk, uint32_t* bintot) {
  const int bin = blk * (NT / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (bin >= bins) return;
  uint32_t* row = hist + (int64_t)bin * nblk;
  uint32_t carry = 0;
  for (int b0 = 0; b0 < nblk; b0 += 32) {
    const int b = b0 + lane;
    const uint32_t v = (b < nblk) ? __ldcg(row + b) : 0u;
    uint32_t inc = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t n = __shfl_up_sync(0xffffffffu, inc, off);
      if (lane >= off) inc += n;
    }
    if (b < nblk) row[b] = carry + inc - v;
    carry += __shfl_sync(0xffffffffu, inc, 31);
  }
  if (lane == 0) bintot[bin] = carry;
}

// Stable scatter: warp w of the block owns the contiguous items [w*512, (w+1)*512) of the tile and
// walks them 32 at a time; rank inside a round comes from the lanes holding the same digit, across rounds and warps from
// per-warp running counters that start at (bins before this digit) + (this digit in earlier tiles).
template <int NT>
__device__ __forceinline__ void sort_scatter_block(int blk, uint32_t* cnt /*shared: [(NT / 32)][bins], binbase[bins], wtot[8]*/,
                                                   const uint32_t* keys_in, const int32_t* pos_in, uint32_t* keys_out,
                                                   int32_t* pos_out, int64_t L, int shift, int bins, int nblk,
                                                   const uint32_t* hist_scanned, const uint32_t* bintot) {
  uint32_t* binbase = cnt + (NT / 32) * bins;
  uint32_t* wtot = binbase + bins;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < (NT / 32) * bins; i += NT) cnt[i] = 0;
  // exclusive scan of the bin totals (bins <= 512 = 2 per thread)
  {
    const int i0 = 2 * threadIdx.x, i1 = i0 + 1;
    const uint32_t v0 = (i0 < bins) ? __ldcg(bintot + i0) : 0u, v1 = (i1 < bins) ? __ldcg(bintot + i1) : 0u;
    uint32_t inc = v0 + v1;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t n = __shfl_up_sync(0xffffffffu, inc, off);
      if (lane >= off) inc += n;
    }
    if (lane == 31) wtot[warp] = inc;
    __syncthreads();
    uint32_t wbase = 0;
    for (int w = 0; w < warp; ++w) wbase += wtot[w];
    const uint32_t excl = wbase + inc - (v0 + v1);
    if (i0 < bins) binbase[i0] = excl;
    if (i1 < bins) binbase[i1] = excl + v0;
  }
  __syncthreads();
  const uint32_t mask = (uint32_t)bins - 1u;
  const int nbits = 31 - __clz(bins);
  const int64_t wbase = (int64_t)blk * (NT * kSortIPT) + (int64_t)warp * (32 * kSortIPT);
  uint32_t key[kSortIPT];
  uint32_t* mycnt = cnt + warp * bins;
#pragma unroll
  for (int k = 0; k < kSortIPT; ++k) {
    const int64_t i = wbase + k * 32 + lane;
    const bool valid = i < L;
    key[k] = valid ? __ldcg(keys_in + i) : 0u;
    const uint32_t digit = valid ? ((key[k] >> shift) & mask) : (uint32_t)bins;   // invalid lanes pair up apart
    const uint32_t peers = same_digit_lanes(digit, nbits);
    if (valid && lane == (__ffs(peers) - 1)) mycnt[digit] += __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  for (int bin = threadIdx.x; bin < bins; bin += NT) {
    uint32_t run = binbase[bin] + __ldcg(hist_scanned + (int64_t)bin * nblk + blk);
#pragma unroll
    for (int w = 0; w < (NT / 32); ++w) {
      const uint32_t c = cnt[w * bins + bin];
      cnt[w * bins + bin] = run;
      run += c;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kSortIPT; ++k) {
    const int64_t i = wbase + k * 32 + lane;
    const bool valid = i < L;
    const uint32_t digit = valid ? ((key[k] >> shift) & mask) : (uint32_t)bins;
    const uint32_t peers = same_digit_lanes(digit, nbits);
    uint32_t dst = 0;
    if (valid) dst = mycnt[digit] + __popc(peers & ((1u << lane) - 1u));
    __syncwarp();
    if (valid && lane == (__ffs(peers) - 1)) mycnt[digit] += __popc(peers);
    __syncwarp();
    if (valid) {
      keys_out[dst] = key[k];
      pos_out[dst] = pos_in ? __ldcg(pos_in + i) : (int32_t)i;
    }
  }
}

// ---- (3) unique, as items of the tiled sort ---------------------------------------------------
// Where the results of the sort half go.  Outputs a caller asked for are written beside the workspace's own.
struct SortOut {
  uint32_t* keys; int32_t* perm;                           // sorted keys and lookup positions [L]
  int32_t* uidx; int32_t* sbag;                            // segment and bag of every sorted position [L]; sbag nullable
  int32_t* uniq; int32_t* seg;                             // distinct keys [U], segment starts [U + 1]
  int32_t *perm_out, *uniq_out, *seg_out, *d_num_unique;   // the caller's, all nullable
  int32_t* scalars; int32_t* d_status;
  int64_t L; uint32_t sentinel;
};

// scalars[2..3] stamp the workspace with the problem it holds a finished sort of; the reduction kernels
// refuse a workspace whose stamp does not match their arguments.
__device__ __forceinline__ int32_t ws_stamp(uint32_t sentinel) { return (int32_t)(sentinel ^ 0x53484144u); }

__device__ __forceinline__ void put_unique(const SortOut& o, uint32_t u, uint32_t key, int64_t pos) {
  o.uniq[u] = (int32_t)key;
  o.seg[u] = (int32_t)pos;
  if (o.uniq_out) o.uniq_out[u] = (int32_t)key;
  if (o.seg_out) o.seg_out[u] = (int32_t)pos;
}
__device__ __forceinline__ void put_segment_end(const SortOut& o, uint32_t u, int64_t pos) {
  o.seg[u] = (int32_t)pos;
  if (o.seg_out) o.seg_out[u] = (int32_t)pos;
}
// U distinct keys: close the segment list when there is none, publish U, stamp the workspace.
__device__ __forceinline__ void finish_unique(const SortOut& o, uint32_t U) {
  if (U == 0) put_segment_end(o, 0, 0);
  if (o.d_num_unique) *o.d_num_unique = (int32_t)U;
  o.scalars[0] = (int32_t)U;
  o.scalars[1] = 0;                                        // rows whose run crosses a window edge (filled by the window kernel)
  o.scalars[kListTicket] = 0;
  o.scalars[2] = (int32_t)o.L;
  o.scalars[3] = ws_stamp(o.sentinel);
}

// Inclusive sum of v over the block's NT threads (s: NT / 32 words of shared memory).
template <int NT>
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t n = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += n;
  }
  __syncthreads();
  if (lane == 31) s[warp] = v;
  __syncthreads();
  uint32_t t = lane < NT / 32 ? s[lane] : 0u;              // every warp scans the warps' totals
  const uint32_t own = t;
#pragma unroll
  for (int off = 1; off < NT / 32; off <<= 1) {
    const uint32_t n = __shfl_up_sync(0xffffffffu, t, off);
    if (lane >= off) t += n;
  }
  return v + __shfl_sync(0xffffffffu, t - own, warp);
}

// A warp's part of a sort tile: kSortIPT rounds of 32 consecutive positions.  Their keys (the sentinel beyond the end), and
// per round the lanes whose key differs from the one before: the heads of segments.
__device__ __forceinline__ uint32_t tile_heads_of(const SortOut& o, int64_t w0, uint32_t (&key)[kSortIPT], uint32_t (&heads)[kSortIPT]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < kSortIPT; ++k) {
    const int64_t i = w0 + 32 * k + lane;
    key[k] = i < o.L ? __ldcg(o.keys + i) : o.sentinel;
  }
  uint32_t last = w0 > 0 && w0 <= o.L ? __ldcg(o.keys + w0 - 1) : 0xffffffffu;   // (no key: a key is at most the sentinel)
  uint32_t total = 0;
#pragma unroll
  for (int k = 0; k < kSortIPT; ++k) {
    uint32_t before = __shfl_up_sync(0xffffffffu, key[k], 1);
    if (lane == 0) before = last;
    last = __shfl_sync(0xffffffffu, key[k], 31);
    heads[k] = __ballot_sync(0xffffffffu, key[k] < o.sentinel && key[k] != before);
    total += __popc(heads[k]);
  }
  return total;
}

template <int NT>
__device__ __forceinline__ void unique_count_block(int blk, uint32_t* s, const SortOut& o, uint32_t* tile_heads) {
  uint32_t key[kSortIPT], heads[kSortIPT];
  const int64_t w0 = (int64_t)blk * (NT * kSortIPT) + (threadIdx.x >> 5) * (32 * kSortIPT);
  const uint32_t c = tile_heads_of(o, w0, key, heads);
  const uint32_t inc = block_scan<NT>((threadIdx.x & 31) == 0 ? c : 0u, s);
  if (threadIdx.x == NT - 1) tile_heads[blk] = inc;
}

// Exclusive scan of the tiles' head counts; closes the unique pass.
template <int NT>
__device__ __forceinline__ void unique_scan_block(uint32_t* s, const SortOut& o, uint32_t* tile_heads, int nblk) {
  uint32_t carry = 0;
  for (int b0 = 0; b0 < nblk; b0 += NT) {
    const int b = b0 + threadIdx.x;
    const uint32_t v = b < nblk ? __ldcg(tile_heads + b) : 0u;
    const uint32_t inc = block_scan<NT>(v, s);
    if (b < nblk) tile_heads[b] = carry + inc - v;
    __syncthreads();
    if (threadIdx.x == NT - 1) s[0] = inc;
    __syncthreads();
    carry += s[0];
    __syncthreads();
  }
  if (threadIdx.x == 0) finish_unique(o, carry);
}

// Segment and bag of every sorted position, distinct keys and segment starts.
template <int NT>
__device__ __forceinline__ void unique_write_block(int blk, uint32_t* s, const SortOut& o, const uint32_t* tile_heads,
                                                   const int32_t* bag_of) {
  const int lane = threadIdx.x & 31;
  uint32_t key[kSortIPT], heads[kSortIPT];
  const int64_t w0 = (int64_t)blk * (NT * kSortIPT) + (threadIdx.x >> 5) * (32 * kSortIPT);
  const uint32_t c = tile_heads_of(o, w0, key, heads);
  uint32_t before = block_scan<NT>(lane == 0 ? c : 0u, s) - (lane == 0 ? c : 0u);
  before = __ldcg(tile_heads + blk) + __shfl_sync(0xffffffffu, before, 0);   // heads before this warp's part
  // the last valid position closes the last segment: seg[U] = number of valid lookups
  const uint32_t after = w0 + 32 * kSortIPT < o.L ? __ldcg(o.keys + w0 + 32 * kSortIPT) : o.sentinel;
#pragma unroll
  for (int k0 = 0; k0 < kSortIPT; k0 += 8) {               // eight rounds' loads in flight
    int pj[8], bag[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int64_t i = w0 + 32 * (k0 + k) + lane;
      pj[k] = i < o.L ? __ldcg(o.perm + i) : -1;
    }
    if (o.sbag) {
#pragma unroll
      for (int k = 0; k < 8; ++k) bag[k] = (pj[k] >= 0 && pj[k] < o.L) ? __ldcg(bag_of + pj[k]) : -1;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int64_t i = w0 + 32 * (k0 + k) + lane;
      const uint32_t m = heads[k0 + k], kk = key[k0 + k];
      const uint32_t inc = before + __popc(m & (0xffffffffu >> (31 - lane)));   // heads up to and including position i
      before += __popc(m);
      uint32_t next = __shfl_down_sync(0xffffffffu, kk, 1);
      const uint32_t first = k0 + k + 1 < kSortIPT ? __shfl_sync(0xffffffffu, key[(k0 + k + 1) % kSortIPT], 0) : after;
      if (lane == 31) next = first;
      if (i >= o.L) continue;
      if ((m >> lane) & 1u) put_unique(o, inc - 1u, kk, i);
      o.uidx[i] = (int32_t)inc - 1;
      if (o.perm_out) o.perm_out[i] = pj[k];
      if (o.sbag) o.sbag[i] = bag[k];
      if (kk < o.sentinel && next >= o.sentinel) put_segment_end(o, inc, i + 1);
    }
  }
}

// ---- (2a) the tiled sort and the unique pass as ONE launch ---------------------------------------
// Work items -- key building per 256 bags, then per digit pass: a histogram per tile, a scan per group of bins, a ranked
// scatter per tile; then head counts per tile, their scan, the outputs per tile -- are numbered in that order and drawn by
// the blocks from a counter.  An item of one phase needs every item of the phases before it; it waits until that many
// items have been reported complete.  The items it waits for have lower numbers, so they were drawn earlier by blocks that
// are running: the wait ends however few blocks the device keeps resident (a single block does everything in turn).
// ctl = {next item, items complete, blocks gone}, zero at launch and left zero.  The wait is bounded (about a second);
// when it runs out the block reports SS_DEV_BAD_WORKSPACE and leaves.
struct TiledSort {
  const int32_t* indices; const int32_t* offsets;
  int T, B; int64_t N;
  uint32_t *keys_a, *keys_b; int32_t *pos_a, *pos_b, *bag_of;
  uint32_t *hist, *bintot, *tile_heads;
  const int32_t* run_if; int* ctl;
  int passes, digit_bits, bins;
  SortOut out;
};
__host__ __device__ constexpr size_t sort_smem_words(int nt) { return (size_t)(nt / 32) * kMaxBins + kMaxBins + nt / 32; }

template <int NT>
__device__ __forceinline__ void tiled_sort_items(const TiledSort& a, uint32_t* smem /*sort_smem_words(NT)*/, int n_blocks) {
  __shared__ int s_item;
  const int64_t L = a.out.L;
  const int nblk = (int)((L + NT * kSortIPT - 1) / (NT * kSortIPT));
  const int n_key_items = (int)(((int64_t)a.T * a.B + NT - 1) / NT), bins_per_item = NT / 32;
  const int n_scan_items = (a.bins + bins_per_item - 1) / bins_per_item;
  const int per_pass = 2 * nblk + n_scan_items, sort_items = n_key_items + a.passes * per_pass;
  const int total = sort_items + 2 * nblk + 1;
  for (;;) {
    __syncthreads();                                       // the previous item's shared memory is no longer in use
    if (threadIdx.x == 0) s_item = atomicAdd(a.ctl, 1);
    __syncthreads();
    const int item = s_item;
    if (item >= total) break;
    // phase of the item, and how many items precede that phase
    int need = 0, pass = -1, phase = 0, idx = item;
    if (item >= sort_items) {
      pass = a.passes;
      idx = item - sort_items;
      need = sort_items;
      if (idx >= nblk) { idx -= nblk; need += nblk; phase = 1; }
      if (phase == 1 && idx >= 1) { idx -= 1; need += 1; phase = 2; }
    } else if (item >= n_key_items) {
      const int r = item - n_key_items;
      pass = r / per_pass;
      idx = r - pass * per_pass;
      need = n_key_items + pass * per_pass;
      if (idx >= nblk) { idx -= nblk; need += nblk; phase = 1; }
      if (phase == 1 && idx >= n_scan_items) { idx -= n_scan_items; need += n_scan_items; phase = 2; }
    }
    if (threadIdx.x == 0 && need > 0) {
      const long long t0 = clock64();
      int seen;
      do {
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(a.ctl + 1) : "memory");
        if (seen < need && clock64() - t0 > 2000000000ll) { s_item = -1; break; }
      } while (seen < need);
    }
    __syncthreads();
    if (s_item < 0) {                                      // gave up: report, and do not touch the item
      if (threadIdx.x == 0 && a.out.d_status) atomicOr(a.out.d_status, SS_DEV_BAD_WORKSPACE);
      break;
    }
    // buffers of this pass: pass 0 reads keys_a (positions = indices), every pass swaps
    const uint32_t* kin = (pass & 1) ? a.keys_b : a.keys_a;
    uint32_t* kout = (pass & 1) ? a.keys_a : a.keys_b;
    const int32_t* pin = pass <= 0 ? nullptr : ((pass & 1) ? a.pos_b : a.pos_a);
    int32_t* pout = (pass & 1) ? a.pos_a : a.pos_b;
    const int shift = pass * a.digit_bits;
    if (pass < 0) build_keys_block<NT>(idx, a.indices, a.offsets, a.T, a.N, a.B, L, a.keys_a, a.bag_of, a.out.d_status);
    else if (pass == a.passes) {
      if (phase == 0) unique_count_block<NT>(idx, smem, a.out, a.tile_heads);
      else if (phase == 1) unique_scan_block<NT>(smem, a.out, a.tile_heads, nblk);
      else unique_write_block<NT>(idx, smem, a.out, a.tile_heads, a.bag_of);
    } else if (phase == 0) sort_hist_block<NT>(idx, smem, kin, L, shift, a.bins, nblk, a.hist);
    else if (phase == 1) bin_scan_block<NT>(idx, a.hist, a.bins, nblk, a.bintot);
    else sort_scatter_block<NT>(idx, smem, kin, pin, kout, pout, L, shift, a.bins, nblk, a.hist, a.bintot);
    __threadfence();                                       // this thread's stores, before the item is reported
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(a.ctl + 1, 1);
  }
  // the last block to leave clears the control words for the next launch
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(a.ctl + 2, 1) == n_blocks - 1) { a.ctl[0] = 0; a.ctl[1] = 0; a.ctl[2] = 0; __threadfence(); }
  }
}

__global__ void __launch_bounds__(kSortThreads)
tiled_sort_kernel(const __grid_constant__ TiledSort a) {
  wait_for_previous_kernel();
  __shared__ uint32_t smem[sort_smem_words(kSortThreads)];
  if (a.run_if && *a.run_if == 0) return;                  // the bucket sort has produced the result
  tiled_sort_items<kSortThreads>(a, smem, gridDim.x);
}

// ---- (2b) bucket sort in shared memory ------------------------------------------------------------
// The lookups arrive grouped by table (bags are table-major), so the sort by key = t*N + row is T independent sorts by
// row.  A table is cut into ranges of rows and a block takes one range: it reads the table's whole index list (a few bytes
// of L2 traffic per lookup), keeps the lookups of its range in order, and sorts them in shared memory with
// stable LSD passes over the bits of the range alone.  Ranges share no row, so the block also finds its distinct rows by
// itself; only the number of distinct rows before it comes from the other blocks (a published count per range, summed by
// everybody), and all outputs of the sort half leave from here: one launch instead of sort, count, scan and write.
// Blocks take their ranges from a ticket, so the counts a block waits for come from blocks that are running.  There are as
// many blocks as tables of any lengths could need; those without a range leave at once.
//
// The cut follows the data, so it does not matter whether popular rows are scattered or neighbours, or one table is longer
// than another.  A table gets a range per `per_range` of its own lookups: equal slices of its rows at first.  While a block
// collects its slice it counts all slices of the table, and if one of them does not fit into a block, every block of the
// table comes to know that; they collect again, ranges whose edges are quantiles of 2048 lookups spread over the table,
// which they all read alike.  A popular row on an edge goes to the side that has less of it; where a range is too full all
// the same, because its first or last row draws so much, that row is not sorted but copied out, in order, by one more walk
// over the index list.  (Quantiles in the first place, or samples that tell whether slices will do, cost 2-4 us a call.)
// What bounds it is instruction issue and the latency of a block's rounds.  Measured alone, the whole sort half, ids scattered /
// ordered by popularity / one row drawing 80 % (in brackets slices with a fixed reserve for a popular row, and the tiled
// passes behind them where those overflowed): 26 tables of 21 500 lookups 44 / 60 / 67 us (43 / 152 / 147), 26 of 32 800
// 58 / 77 / 103 (49 / 164 / 161), 40 of 32 900 56 / 85 / 115 (74 / 272 / 258).
//
// A block that cannot take the path (a range with more lookups than `cap` after all, a table of more than 65536, offsets
// that are not monotone within [0, L], a row index outside the table) raises *fallback.  Only a range can be too full if
// L > cap: then the caller launches tiled_sort_kernel behind this kernel, which returns at once when the flag is down.
// Otherwise the input is malformed, and the last block to leave runs the tiled sort's items by itself: slow, and nothing
// to launch.
constexpr int kBsThreads = 1024;
constexpr int kBsWarps = kBsThreads / 32;
constexpr int kBsChunk = 8 * kBsThreads;                   // index positions looked at together, 8 per thread
constexpr int kBsDigit = 10;                               // most bits of a digit
constexpr int kBsMaxLookups = 65536;                       // of a table: positions inside it take 16 bits
constexpr size_t kBsSmemMax = 226 * 1024;                  // leaves room for the static part
constexpr int kBsRounds = 16;                              // most rounds of 32 lookups per warp: a block sorts up to 16384
// Lookups a range is meant to hold: with kBsSamples the share of a range of C equal ones is off by sqrt((C - 1) / 2048) of
// itself (one standard deviation), so 13400 stays below 16384 by five of them for up to five ranges.
constexpr int kBsSamples = 2 * kBsThreads, kBsRange = 13400;
// dynamic shared memory: row, position, bag and index of the kept lookups (10 bytes each), then a region that first
// holds a chunk of the index list and its bags and later the digit counters
__host__ __device__ constexpr size_t bs_counter_bytes(int nb) { return (size_t)kBsWarps * ((1 << nb) + 2) * 2; }
__host__ __device__ constexpr size_t bs_region(int nb) {
  return bs_counter_bytes(nb) > (size_t)kBsChunk * 6 ? bs_counter_bytes(nb) : (size_t)kBsChunk * 6;
}
__host__ __device__ constexpr size_t bs_smem(int cap, int nb) {
  const size_t own = (size_t)cap * 10 + bs_region(nb), tiled = sort_smem_words(kBsThreads) * 4;
  return own > tiled ? own : tiled;
}
constexpr int kBsCap = kBsRounds * kBsThreads;
static_assert(bs_smem(kBsCap, kBsDigit) <= kBsSmemMax, "the largest range and the widest digit fit");

struct BucketSort {
  const int32_t* indices; const int32_t* offsets;
  int64_t N;
  int T, B;
  int per_range, cap;                                      // lookups per range, lookups one can hold
  int ranges, serial_fallback;                             // ranges > 0: that many for every table (more tables than threads)
  int32_t* fallback;                                       // zero at launch
  int* ticket;                                             // {next range, blocks gone}: zero at launch
  uint32_t* counts;                                        // [T * kBsMaxBuckets], zero at launch: distinct rows of a range | 1 << 31
};

template <int NB>
__device__ __forceinline__ uint32_t same_digit_lanes_n(uint32_t digit) {
  uint32_t peers = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const bool bit = (digit >> b) & 1u;
    const uint32_t m = __ballot_sync(0xffffffffu, bit);
    peers &= bit ? m : ~m;
  }
  return peers;
}

// One stable LSD pass over NB bits of the kept lookups' rows: order -> order.  A pass looks at every lookup once: the lanes
// of a round that hold the same digit give its rank among the warp's lookups with that digit, kept in a register until the
// counters have been scanned.
template <int NB>
__device__ __forceinline__ void bucket_sort_pass(const uint32_t* okey, uint16_t* order, uint16_t* cnt, uint32_t* s_w, int shift,
                                                 int i0, int iend) {
  constexpr int bins = 1 << NB, kStride = bins + 2;        // padded: the scan reads one digit of all warps
  constexpr uint32_t mask = (uint32_t)bins - 1u;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint16_t* mycnt = cnt + warp * kStride;
  uint32_t held[kBsRounds];                                // lookup | rank << 16
  for (int i = tid; i < kBsWarps * kStride / 2; i += kBsThreads) reinterpret_cast<uint32_t*>(cnt)[i] = 0u;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kBsRounds; ++r) {                    // whole rounds: the bounds are the same for all lanes
    const int i = i0 + 32 * r + lane;
    if (i - lane >= iend) break;
    const uint32_t pay = shift == 0 ? (uint32_t)i : order[i];
    const uint32_t digit = (okey[pay] >> shift) & mask;
    const uint32_t peers = same_digit_lanes_n<NB>(digit);
    const uint32_t lower = peers & ((1u << lane) - 1u);
    const uint32_t base = mycnt[digit];
    __syncwarp();
    if (lower == 0) mycnt[digit] = (uint16_t)(base + __popc(peers));
    __syncwarp();
    held[r] = pay | (base + __popc(lower)) << 16;
  }
  __syncthreads();
  // exclusive scan in (digit, warp) order: thread tid owns bins / 32 consecutive entries of that order
  {
    constexpr int per = bins >> 5;
    uint32_t v[per], sum = 0;
#pragma unroll
    for (int u = 0; u < per; ++u) {
      const int e = tid * per + u;
      v[u] = cnt[(e & 31) * kStride + (e >> 5)];
      sum += v[u];
    }
    uint32_t run = block_scan<kBsThreads>(sum, s_w) - sum;
#pragma unroll
    for (int u = 0; u < per; ++u) {
      const int e = tid * per + u;
      cnt[(e & 31) * kStride + (e >> 5)] = (uint16_t)run;
      run += v[u];
    }
  }
  __syncthreads();
  // stable scatter
#pragma unroll
  for (int r = 0; r < kBsRounds; ++r) {
    if (i0 + 32 * r >= iend) break;
    const uint32_t pay = held[r] & 0xffffu;
    order[mycnt[(okey[pay] >> shift) & mask] + (held[r] >> 16)] = (uint16_t)pay;
  }
  __syncthreads();
}

// The range in hand: what one phase finds out and a later one needs stays in shared memory rather than in registers.
struct BucketRange {
  uint32_t w[kBsWarps], m[kBsWarps];                       // scratch of the scans
  uint32_t total, id;                                      // ranges of all tables, this one
  int t, c, ranges, seg0, seg1;                            // its table, its number there, how many there are, the table's segment
  uint32_t edge[2], rank[2];                               // while the edges are looked for
  uint32_t base, span, hot_row;                            // rows [base, base + span) are sorted, one beside them may be copied out
  uint32_t edges[kBsMaxBuckets - 1], part[kBsMaxBuckets - 1][kBsWarps];   // rows; lookups of rows before them, per warp
  int n_edges, lt[kBsMaxBuckets - 1];                      // and in all
  int kept, hot, out0;                                     // lookups sorted and copied out, where the sorted ones go
  uint32_t mine, before;                                   // distinct rows of this range and of those before it
};

__device__ __forceinline__ bool sound_table(const BucketSort& a, int64_t L, int t, int seg0, int seg1) {
  return seg0 >= 0 && seg1 >= seg0 && (int64_t)seg1 <= L && seg1 - seg0 <= kBsMaxLookups && (t != 0 || seg0 == 0) &&
         (t != a.T - 1 || (int64_t)seg1 == L);
}

// Two edges of a table's ranges, into r.edge: the k0-th and k1-th smallest (from 0) of the threads' 2 x 1024 values, below
// 2^bits, each plus one if more of the values equal to it come before that place than after.  A histogram of the highest ten
// bits tells in which bin each lies, one of the next ten bits of that bin's values the bin inside it, and so on.  Counts of
// the two share a word.  hist: 1024 words of shared memory.
__device__ __forceinline__ void select_two(BucketRange& r, uint32_t* hist, const uint32_t (&value)[2], int bits, int k0, int k1) {
  const int tid = threadIdx.x;
  if (tid == 0) { r.edge[0] = r.edge[1] = 0u; r.rank[0] = (uint32_t)k0; r.rank[1] = (uint32_t)k1; }
  for (int shift = bits; shift > 0;) {
    const int d = shift < 10 ? shift : 10;
    shift -= d;
    hist[tid] = 0u;
    __syncthreads();
    const uint32_t e0 = r.edge[0], e1 = r.edge[1], want0 = r.rank[0], want1 = r.rank[1];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const uint32_t high = value[i] >> shift >> d, add = (high == e0 ? 1u : 0u) + (high == e1 ? 0x10000u : 0u);
      if (add) atomicAdd(&hist[(value[i] >> shift) & ((1u << d) - 1u)], add);
    }
    __syncthreads();
    const uint32_t own = hist[tid];                        // (bins beyond 2^d are empty)
    const uint32_t upto = block_scan<kBsThreads>(own, r.w), before = upto - own;
    const uint32_t at0 = want0 - (before & 0xffffu), at1 = want1 - (before >> 16);
    if (at0 < (own & 0xffffu)) { r.edge[0] = (e0 << d | (uint32_t)tid) + (shift == 0 && 2 * at0 > (own & 0xffffu)); r.rank[0] = at0; }
    if (at1 < own >> 16) { r.edge[1] = (e1 << d | (uint32_t)tid) + (shift == 0 && 2 * at1 > own >> 16); r.rank[1] = at1; }
    __syncthreads();
  }
}

constexpr uint32_t kNoRow = 0xffffffffu;                   // no row id is that large
// What a thread has in flight before a walk: the first chunk of the index list (kNoRow beyond its end), the offsets of bag `tid`.
struct WalkStart {
  uint32_t next[8];
  int l, h;
  __device__ __forceinline__ WalkStart(const BucketSort& a, const BucketRange& r, int n) {
    const int tid = threadIdx.x;
    const int32_t* off = a.offsets + (int64_t)r.t * a.B;
    l = h = 0;
    if (tid < a.B) { l = off[tid]; h = off[tid + 1]; }
#pragma unroll
    for (int k = 0; k < 8; ++k) next[k] = tid + k * kBsThreads < n ? (uint32_t)__ldg(a.indices + r.seg0 + tid + k * kBsThreads) : kNoRow;
  }
};

// Walks the index list of table r.t, n long, and hands the lookups of rows [from, from + rows) to put(number, number in the
// chunk, row, position, bag), in order, and after each chunk their numbers to flush(first, count); their count, or -1: the
// list is malformed.  Per thread, byte j % 4 of seen[j / 4] counts the lookups of rows before r.edges[j] (a thread looks at
// 64 positions at most).  The list goes through shared memory so that its loads are coalesced; a chunk's loads are in flight
// while the chunk before is worked on.
template <typename Put, typename Flush>
__device__ __forceinline__ int walk_table(const BucketSort& a, BucketRange& r, uint32_t* crow, uint16_t* cbag, int n, WalkStart& start,
                                          uint32_t from, uint32_t rows, int n_edges, uint32_t (&seen)[2], Put put, Flush flush) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int seg0 = r.seg0, seg1 = seg0 + n;
  const int32_t* off = a.offsets + (int64_t)r.t * a.B;
  int kept = 0;
  uint32_t bag_carry = 0;                                  // 1 + the last bag that starts before the chunk
  for (int p0 = 0; p0 == 0 || p0 < n; p0 += kBsChunk) {    // (once for an empty table: its offsets are checked here)
    const int p1 = min(n, p0 + kBsChunk);
    const int w0 = p0 + 8 * tid;                           // a thread looks at eight consecutive positions
    int bad = 0;
    // every bag that starts in the chunk leaves its number at its first position; the bag of a position is the highest
    // number at or before it
    auto mark = [&](int b, int l, int h) {
      if (l < seg0 || h < l || h > seg1) bad = 1;
      else if (h > l && l - seg0 >= p0 && l - seg0 < p1) cbag[l - seg0 - p0] = (uint16_t)(b + 1);
    };
    *reinterpret_cast<uint4*>(cbag + 8 * tid) = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    if (tid < a.B) mark(tid, start.l, start.h);
#pragma unroll 2
    for (int b = tid + kBsThreads; b < a.B; b += kBsThreads) mark(b, off[b], off[b + 1]);
#pragma unroll
    for (int k = 0; k < 8; ++k) crow[tid + k * kBsThreads] = start.next[k];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int p = p0 + kBsChunk + tid + k * kBsThreads;
      start.next[k] = p < n ? (uint32_t)__ldg(a.indices + seg0 + p) : kNoRow;
    }
    __syncthreads();
    const uint4 r0 = *reinterpret_cast<const uint4*>(crow + 8 * tid), r1 = *reinterpret_cast<const uint4*>(crow + 8 * tid + 4);
    const uint32_t row[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
    int mine = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (row[k] >= (uint32_t)a.N && w0 + k < p1) bad = 1; // one unsigned compare: negative indices are huge
      mine += row[k] - from < rows;
    }
    for (int j = 0; j < n_edges; ++j) {
      const uint32_t edge = r.edges[j];
      uint32_t c = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) c += row[k] < edge;
      if (j < 4) seen[0] += c << 8 * j; else seen[1] += c << 8 * (j - 4);
    }
    if (__syncthreads_or(bad)) return -1;
    const uint4 mk = *reinterpret_cast<const uint4*>(cbag + 8 * tid);
    const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
    uint32_t top = 0;                                      // the highest number at this thread's positions
#pragma unroll
    for (int k = 0; k < 4; ++k) top = max(top, max(mw[k] & 0xffffu, mw[k] >> 16));
    // scan over the threads: kept lookups (sum) and bag numbers (maximum)
    uint32_t sum = (uint32_t)mine, mx = top;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, sum, d), v = __shfl_up_sync(0xffffffffu, mx, d);
      if (lane >= d) { sum += u; mx = max(mx, v); }
    }
    if (lane == 31) { r.w[warp] = sum; r.m[warp] = mx; }
    __syncthreads();
    uint32_t ws = r.w[lane], wm = r.m[lane];               // kBsWarps == 32: every warp scans the warps' totals
    const uint32_t ws0 = ws;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, ws, d), v = __shfl_up_sync(0xffffffffu, wm, d);
      if (lane >= d) { ws += u; wm = max(wm, v); }
    }
    const int chunk = (int)__shfl_sync(0xffffffffu, ws, 31);
    int at = kept + (int)(__shfl_sync(0xffffffffu, ws - ws0, warp) + sum) - mine;
    uint32_t bag = __shfl_up_sync(0xffffffffu, mx, 1);
    if (lane == 0) bag = 0;
    const uint32_t wbag = __shfl_sync(0xffffffffu, wm, max(warp - 1, 0));
    bag = max(bag, max(bag_carry, warp ? wbag : 0u));
    bag_carry = max(bag_carry, __shfl_sync(0xffffffffu, wm, 31));
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      bag = max(bag, (k & 1) ? mw[k >> 1] >> 16 : mw[k >> 1] & 0xffffu);
      if (row[k] - from < rows) {
        put(at, at - kept, row[k], w0 + k, (int)bag - 1);
        ++at;
      }
    }
    __syncthreads();                                       // the chunk's bags and the scans' scratch are free again
    flush(kept, chunk);
    kept += chunk;
  }
  return kept;
}

__device__ __forceinline__ void write_sorted(const SortOut& o, int j, uint32_t key, int pos, int bag, uint32_t u) {
  o.keys[j] = key;
  if (o.perm_out) o.perm_out[j] = pos;                     // (o.perm is the tiled passes' own)
  o.uidx[j] = (int32_t)u;
  o.sbag[j] = bag;
}

// The range's rows by quantiles of samples: r.base, r.span, r.hot_row, and the rows whose lookups the walk is to count.
__device__ __forceinline__ void recut(const BucketSort& a, BucketRange& r, uint32_t* hist) {
  const int tid = threadIdx.x, n = r.seg1 - r.seg0, c = r.c, C = r.ranges;
  uint32_t sample[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) sample[i] = min((uint32_t)__ldg(a.indices + r.seg0 + (((2 * tid + i) * n) >> 11)), (uint32_t)a.N - 1u);
  select_two(r, hist, sample, max(1, 32 - __clz((uint32_t)a.N - 1u)), c * kBsSamples / C, min((c + 1) * kBsSamples / C, kBsSamples - 1));
  const uint32_t lo = c > 0 ? r.edge[0] : 0u, hi = c < C - 1 ? r.edge[1] : (uint32_t)a.N;
  auto count = [&](uint32_t from, uint32_t rows) {         // samples of rows [from, from + rows)
    return __syncthreads_count(sample[0] - from < rows) + __syncthreads_count(sample[1] - from < rows);
  };
  // what a block holds, less five standard deviations of the samples' share (1 / 18 = 2.5 / sqrt(2048)), in samples
  uint32_t hot = kNoRow;
  if (count(lo, hi - lo) > (int)((int64_t)(a.cap - n / 18) * kBsSamples / n)) hot = count(lo, 1u) >= count(hi - 1u, 1u) ? lo : hi - 1u;
  if (tid == 0) {
    r.base = lo + (hot == lo);
    r.span = hi - r.base - (hot != lo && hot != kNoRow);
    r.hot_row = hot;
    r.edges[0] = r.base; r.edges[1] = hot; r.edges[2] = hot + 1u;
    r.n_edges = hot == kNoRow ? 1 : 3;
  }
}

// Collects the range's lookups (rows [r.base, r.base + r.span)) in shared memory, as many as fit, and counts those of rows
// before each of r.edges into r.lt; their number, or -1: the list is malformed.
__device__ __forceinline__ int collect(const BucketSort& a, BucketRange& r, int n, uint32_t* okey, uint16_t* opos, uint16_t* obag,
                                       uint32_t* crow, uint16_t* cbag) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cap = a.cap;
  WalkStart start(a, r, n);
  __syncthreads();                                         // the range is set
  const uint32_t base = r.base;
  const int n_edges = r.n_edges;
  uint32_t seen[2] = {0u, 0u};
  const int kept = walk_table(a, r, crow, cbag, n, start, base, r.span, n_edges, seen,
                              [&](int at, int, uint32_t row, int position, int bag) {
                                if (at >= cap) return;
                                okey[at] = row - base;
                                opos[at] = (uint16_t)position;
                                obag[at] = (uint16_t)bag;
                              }, [](int, int) {});
  for (int j = 0; j < n_edges; ++j) {
    const uint32_t c = __reduce_add_sync(0xffffffffu, (seen[j >> 2] >> 8 * (j & 3)) & 0xffu);
    if (lane == 0) r.part[j][warp] = c;
  }
  __syncthreads();
  if (warp < n_edges) {
    const int c = (int)__reduce_add_sync(0xffffffffu, r.part[warp][lane]);
    if (lane == 0) r.lt[warp] = c;
  }
  __syncthreads();
  return kept;
}

// The same once more, by quantiles.  Out of line, like copy_row: few tables need it, and inside the kernel its registers cost
// every range (26 tables of 21 500 lookups 43 -> 45 us).
__device__ __noinline__ int collect_again(const BucketSort& a, BucketRange& r, int n, uint32_t* okey, uint16_t* opos, uint16_t* obag,
                                          uint32_t* crow, uint16_t* cbag) {
  recut(a, r, okey);
  return collect(a, r, n, okey, opos, obag, crow, cbag);
}

// Outputs of the row of a range that is not sorted.
__device__ __noinline__ void copy_row(const BucketSort& a, const SortOut& o, BucketRange& r, uint16_t* opos, uint16_t* obag,
                                      uint32_t* crow, uint16_t* cbag) {
  const int tid = threadIdx.x, seg0 = r.seg0, n = r.seg1 - seg0, bag0 = r.t * a.B;
  const bool before = r.hot_row < r.base;                  // the sorted rows
  const int first = before ? r.out0 - r.hot : r.out0 + r.kept;
  const uint32_t key = (uint32_t)((uint64_t)r.t * (uint64_t)a.N) + r.hot_row, u = before ? r.before : r.before + r.mine - 1u;
  WalkStart start(a, r, n);
  uint32_t unused[2] = {0u, 0u};
  __syncthreads();                                         // everybody is done with what the block kept and with the counters
  walk_table(a, r, crow, cbag, n, start, r.hot_row, 1u, 0, unused,
             [&](int, int i, uint32_t, int position, int bag) {
               opos[i] = (uint16_t)position;
               obag[i] = (uint16_t)bag;
             },
             [&](int done, int count) {
               for (int i = tid; i < count; i += kBsThreads) write_sorted(o, first + done + i, key, seg0 + opos[i], bag0 + obag[i], u);
             });
  if (tid == 0 && (int64_t)u < o.L) put_unique(o, u, key, first);
}

template <int NB>                                          // digit bits, 5..kBsDigit
__global__ void __launch_bounds__(kBsThreads, 1)
bucket_sort_kernel(const __grid_constant__ BucketSort a, const __grid_constant__ TiledSort tiled) {
  wait_for_previous_kernel();
  extern __shared__ __align__(16) unsigned char bs_raw[];
  __shared__ BucketRange r;
  const SortOut& o = tiled.out;
  const int cap = a.cap;
  uint32_t* okey = reinterpret_cast<uint32_t*>(bs_raw);    // row, relative to the range, of kept lookup i
  uint16_t* opos = reinterpret_cast<uint16_t*>(okey + cap);           // its position in the table
  uint16_t* obag = opos + cap;                             // its bag, inside the table
  uint16_t* order = obag + cap;                            // the kept lookups in the order reached so far
  uint16_t* cnt = order + cap;                             // [kBsWarps][bins + 2]
  uint32_t* crow = reinterpret_cast<uint32_t*>(cnt);       // the chunk's row ids (cap is a multiple of 32: 16-byte aligned)
  uint16_t* cbag = reinterpret_cast<uint16_t*>(crow + kBsChunk);      // and bags
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  do {                                                     // (a break: nothing to do for this block)
    // ---- how many ranges every table has, by its lookups, and which range is this block's; thread t looks after table t
    constexpr int kBad = 1 << 20;                          // more than all ranges
    auto ranges_of = [&](int t, int first, int last) {
      return sound_table(a, o.L, t, first, last) ? max(1, min(kBsMaxBuckets, (last - first + a.per_range - 1) / a.per_range)) : kBad;
    };
    auto take = [&](int id, int t, int end, int ranges, int first, int last) {
      if (id < end && id >= end - ranges) { r.t = t; r.c = id - (end - ranges); r.ranges = ranges; r.seg0 = first; r.seg1 = last; }
    };
    if (a.ranges == 0 && a.T <= 64) {
      if (warp == 0) {                                     // one warp, two tables a lane: the others issue nothing meanwhile
        int first[2] = {0, 0}, last[2] = {0, 0}, ranges[2] = {0, 0}, id = 0;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int t = lane + 32 * i;
          if (t < a.T) { first[i] = a.offsets[(int64_t)t * a.B]; last[i] = a.offsets[(int64_t)(t + 1) * a.B]; }
        }
        if (lane == 0) id = atomicAdd(a.ticket, 1);
        int end = 0;
        id = __shfl_sync(0xffffffffu, id, 0);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int t = lane + 32 * i;
          if (t < a.T) ranges[i] = ranges_of(t, first[i], last[i]);
          int upto = ranges[i];
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, upto, d);
            if (lane >= d) upto += x;
          }
          take(id, t, end + upto, ranges[i], first[i], last[i]);
          end += __shfl_sync(0xffffffffu, upto, 31);
        }
        if (lane == 0) {
          r.id = (uint32_t)id; r.total = (uint32_t)end;
          if (end >= kBad) atomicOr(a.fallback, 1);
        }
      }
      __syncthreads();
      if (r.id >= r.total || r.total >= (uint32_t)kBad) break;
    } else if (a.ranges == 0) {
      int first = 0, last = 0, ranges = 0;
      if (tid < a.T) { first = a.offsets[(int64_t)tid * a.B]; last = a.offsets[(int64_t)(tid + 1) * a.B]; }
      if (tid == 0) r.id = (uint32_t)atomicAdd(a.ticket, 1);
      if (tid < a.T) ranges = ranges_of(tid, first, last);
      const int end = (int)block_scan<kBsThreads>((uint32_t)ranges, r.w);
      if (tid == kBsThreads - 1) {
        r.total = (uint32_t)end;
        if (end >= kBad) atomicOr(a.fallback, 1);
      }
      take((int)r.id, tid, end, ranges, first, last);
      __syncthreads();
      if (r.id >= r.total || r.total >= (uint32_t)kBad) break;
    } else {
      if (tid == 0) {
        r.id = (uint32_t)atomicAdd(a.ticket, 1);
        const int t = (int)r.id / a.ranges;
        r.total = gridDim.x;
        r.t = t; r.c = (int)r.id - t * a.ranges; r.ranges = a.ranges;
        r.seg0 = a.offsets[(int64_t)t * a.B]; r.seg1 = a.offsets[(int64_t)(t + 1) * a.B];
      }
      __syncthreads();
    }
    // ---- the range's rows, and its lookups into shared memory
    {
      const bool sound = sound_table(a, o.L, r.t, r.seg0, r.seg1);
      const int n = sound ? r.seg1 - r.seg0 : 0, C = r.ranges;
      if (tid < kBsMaxBuckets) {
        const uint32_t width = ((uint32_t)a.N + C - 1u) / C, edge = min((tid + 1u) * width, (uint32_t)a.N);
        if (tid < kBsMaxBuckets - 1) r.edges[tid] = edge;
        if (tid == r.c) { r.base = min(tid * width, (uint32_t)a.N); r.span = edge - r.base; r.hot_row = kNoRow; r.n_edges = C - 1; }
      }
      int kept = collect(a, r, n, okey, opos, obag, crow, cbag);
      int fullest = kept, before = r.c > 0 ? r.lt[r.c - 1] : 0, hot = 0;
      for (int c = 0; c < C; ++c) fullest = max(fullest, (c < C - 1 ? r.lt[c] : n) - (c > 0 ? r.lt[c - 1] : 0));   // of all slices
      if (kept >= 0 && C > 1 && fullest > cap) {
        fullest = kept = collect_again(a, r, n, okey, opos, obag, crow, cbag);
        before = r.lt[0];
        hot = r.hot_row == kNoRow ? 0 : r.lt[2] - r.lt[1];
      }
      const bool ok = sound && kept >= 0 && fullest <= cap;
      const int q = ok ? kept : 0;
      // pads of the last round: the largest digits and the last places, so every stable pass leaves them at the end
      if (tid < ((q + 31) & ~31) - q) okey[q + tid] = 0xffffffffu;
      if (tid == 0) {
        if (!ok) atomicOr(a.fallback, 1);
        r.kept = q;
        r.hot = ok ? hot : 0;
        r.out0 = r.seg0 + before;
      }
      __syncthreads();
    }
    // ---- sort
    const int q = r.kept, q32 = (q + 31) & ~31;
    const int rounds = (q32 + kBsThreads - 1) / kBsThreads;  // rounds of 32 consecutive items per warp
    const int i0 = warp * rounds * 32, iend = min(i0 + rounds * 32, q32);
    if (q > 0) {
      const int bits = max(1, 32 - __clz(r.span - 1u));    // (something was kept: there is a row)
      for (int shift = 0; shift < bits; shift += NB) bucket_sort_pass<NB>(okey, order, cnt, r.w, shift, i0, iend);
    }
    // ---- distinct rows: a warp walks its sorted positions 32 at a time; a position is a head when its row differs from the one before
    auto head_at = [&](int j, uint32_t k) {                // all lanes; k: row at j (anything beyond the end)
      uint32_t before = __shfl_up_sync(0xffffffffu, k, 1);
      if (lane == 0) before = j > 0 && j <= q ? okey[order[j - 1]] : 0u;
      return j < q && (j == 0 || k != before);
    };
    uint32_t heads = 0;
    for (int j = i0 + lane; j < iend; j += 32) heads += __popc(__ballot_sync(0xffffffffu, head_at(j, okey[order[j]])));
    const uint32_t inc = block_scan<kBsThreads>(lane == 0 ? heads : 0u, r.w);   // heads of the warps up to this one
    if (tid == kBsThreads - 1) {
      r.mine = inc + (r.hot > 0);
      atomicExch(a.counts + r.id, r.mine | 0x80000000u);   // for the ranges behind this one
    }
    __syncthreads();
    // distinct rows of the ranges before this one
    {
      uint32_t sum = 0;
      bool gave_up = false;
      const long long t0 = clock64();
      for (int i = tid; i < (int)r.id; i += kBsThreads) {
        uint32_t v;
        while (!((v = *reinterpret_cast<volatile uint32_t*>(a.counts + i)) >> 31)) {
          if (clock64() - t0 > 2000000000ll) { gave_up = true; break; }
          __nanosleep(64);
        }
        sum += v & 0x7fffffffu;
      }
      if (gave_up && o.d_status) atomicOr(o.d_status, SS_DEV_BAD_WORKSPACE);
      const uint32_t all = block_scan<kBsThreads>(sum, r.w);
      if (tid == kBsThreads - 1) r.before = all;
    }
    __syncthreads();
    // ---- outputs: the sorted rows, and the row copied out before or behind them
    const int seg0 = r.seg0, bag0 = r.t * a.B, out0 = r.out0;
    const uint32_t key0 = (uint32_t)((uint64_t)r.t * (uint64_t)a.N);
    {
      const uint32_t base = key0 + r.base;
      uint32_t u_next = r.before + (r.hot > 0 && r.hot_row < r.base) + __shfl_sync(0xffffffffu, inc - (lane == 0 ? heads : 0u), 0);
#pragma unroll 4
      for (int j = i0 + lane; j < iend; j += 32) {
        const int pay = j < q ? order[j] : 0;
        const uint32_t k = okey[pay];
        const int pos = seg0 + opos[pay];
        const int bag = bag0 + obag[pay];
        const bool head = head_at(j, k);
        const uint32_t m = __ballot_sync(0xffffffffu, head);
        const uint32_t u = u_next + __popc(m & (0xffffffffu >> (31 - lane))) - 1u;
        u_next += __popc(m);
        if (j < q) {
          write_sorted(o, out0 + j, base + k, pos, bag, u);
          // (u < L unless another table's offsets are malformed; then the fallback writes all of this again)
          if (head && (int64_t)u < o.L) put_unique(o, u, base + k, out0 + j);
        }
      }
    }
    if (r.hot > 0) copy_row(a, o, r, opos, obag, crow, cbag);
    if (r.id == r.total - 1 && tid == 0) {
      put_segment_end(o, min(r.before + r.mine, (uint32_t)o.L), o.L);
      finish_unique(o, r.before + r.mine);
    }
  } while (false);
  if (a.serial_fallback) {
    __threadfence();
    __syncthreads();
    if (tid == 0) r.id = (uint32_t)atomicAdd(a.ticket + 1, 1);
    __syncthreads();
    if (r.id != gridDim.x - 1) return;
    __threadfence();
    if (*reinterpret_cast<volatile int32_t*>(a.fallback) != 0)
      tiled_sort_items<kBsThreads>(tiled, reinterpret_cast<uint32_t*>(bs_raw), 1);
  }
}

__device__ __forceinline__ bool ws_matches(const int32_t* scalars, int64_t L, uint32_t sentinel, int32_t* d_status) {
  if (scalars[2] == (int32_t)L && scalars[3] == ws_stamp(sentinel)) return true;
  if (d_status && threadIdx.x == 0 && blockIdx.x == 0) atomicOr(d_status, SS_DEV_BAD_WORKSPACE);
  return false;
}

// ---- (4) windowed segment reduction ---------------------------------------------------------
// A lane group owns a window of kWin consecutive sorted positions and adds the gradient rows of each
// run of equal keys in position order.  A run that lies inside the window is complete: its sum goes
// to gsum[u].  A run that crosses a window edge leaves a partial sum in the window's slot 0 (run
// covers the window's first position) or slot 1.  This kernel serves rows wider than 256 floats, and of more than
// 128 where windows are few or rows popular; the others take window_apply_kernel, which also updates the rows.
template <int G, int NV>
__global__ void __launch_bounds__(256)
window_reduce_kernel(const uint32_t* __restrict__ keys, const int32_t* __restrict__ sbag,
                     const int32_t* __restrict__ uidx, int64_t L,
                     uint32_t sentinel, int64_t N, int D, int B, const float* __restrict__ grad, int64_t ld_grad,
                     int col0, float* __restrict__ gsum, float* __restrict__ partial, int32_t* __restrict__ long_list,
                     int32_t* __restrict__ scalars, int nwin, int64_t umax, int32_t* __restrict__ d_status) {
  wait_for_previous_kernel();
  constexpr int kGroups = 256 / G;
  __shared__ uint32_t s_key[kGroups][kWin + 2];            // [0] = key before the window, [kWin+1] = key after
  __shared__ int32_t s_row[kGroups][kWin];                 // float4 index of the lookup's gradient row
  __shared__ int32_t s_u[kGroups][kWin];
  const int grp = threadIdx.x / G, lane = threadIdx.x % G;
  const int64_t win = (int64_t)blockIdx.x * kGroups + grp;
  const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << ((threadIdx.x & 31) / G * G));
  if (!ws_matches(scalars, L, sentinel, d_status)) return;
  if (win >= nwin) return;
  const int64_t w0 = win * kWin;
  const int nvec = D >> 2;
  const int64_t ld4 = ld_grad >> 2;
  // keys (one before and one after the window included), bag and segment of every position: one round of loads
  for (int i = lane; i < kWin + 2; i += G) {
    const int64_t j = w0 - 1 + i;
    const bool in_range = j >= 0 && j < L;
    const bool body = i >= 1 && i <= kWin;
    uint32_t key = in_range ? keys[j] : sentinel;
    const int sb = (body && in_range) ? sbag[j] : 0;
    const int u = (body && in_range) ? uidx[j] : 0;
    int32_t row = -1;
    if (body && key < sentinel) {
      const int t = (int)((uint32_t)sb / (uint32_t)B);     // bags are table-major: bag = t*B + b (32-bit division)
      const int b = sb - t * B;
      // a consistent workspace never fails these; an inconsistent one must not turn into a wild access
      if (sb >= 0 && (int64_t)key >= (int64_t)t * N && (int64_t)key < (int64_t)(t + 1) * N && u >= 0 && u < umax)
        row = (int32_t)((int64_t)b * ld4 + (int64_t)t * nvec);   // B * ld_grad / 4 < 2^31 is checked on the host
      else
        key = sentinel;
    }
    s_key[grp][i] = key;
    if (body) { s_row[grp][i - 1] = row; s_u[grp][i - 1] = u; }
  }
  __syncwarp(gmask);
  const float4* grad4 = reinterpret_cast<const float4*>(grad + col0);  // col0 is a multiple of 4

  float4 acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
  int run_start = 0;
  constexpr int kBatch = NV >= 8 ? 1 : (NV >= 4 ? 2 : (NV >= 2 ? 4 : 8));   // gradient rows in flight per lane
  for (int i0 = 0; i0 < kWin; i0 += kBatch) {
    float4 gv[kBatch][NV];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int32_t row = s_row[grp][i0 + u];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int c = lane + v * G;
        gv[u][v] = (row >= 0 && c < nvec) ? __ldg(grad4 + row + c) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int i = i0 + u;
      const uint32_t key = s_key[grp][1 + i];
      if (key >= sentinel) continue;                       // skipped lookups sort last; nothing follows them
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = add4(acc[v], gv[u][v]);
      const uint32_t next = s_key[grp][2 + i];
      if (next != key || i == kWin - 1) {
        const bool head_open = (run_start == 0) && (s_key[grp][0] == key);
        const bool tail_open = (next == key);              // only possible at the window's last position
        const bool complete = !head_open && !tail_open;
        float4* dst = complete ? reinterpret_cast<float4*>(gsum + (int64_t)s_u[grp][i] * D)
                               : reinterpret_cast<float4*>(partial + ((int64_t)win * 2 + (run_start == 0 ? 0 : 1)) * D);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int c = lane + v * G;
          if (c < nvec) dst[c] = acc[v];
          acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        // the window in which a multi-window run starts enters the row in the list of rows to combine
        if (!head_open && tail_open && lane == 0) {
          const int slot = atomicAdd(&scalars[1], 1);
          if (slot < nwin) long_list[slot] = s_u[grp][i];   // at most one such run per window
        }
        run_start = i + 1;
      }
    }
  }
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// ---- (4b) fused window kernel for rows of at most 256 floats --------------------------------------
// Same windows and same order of additions as window_reduce_kernel.  A block stages keys and gradient rows of its windows
// together (32 consecutive positions per warp and round) and requests the table rows of the runs into L2; ballots give the run
// structure of a window as 16-bit masks.  A batch of positions requests its gradient rows and, for the runs that end in it, the
// table rows and states at once; then it adds, and updates a row where a run ends.  A run of up to kShortSpan windows of one
// block is finished by the group it starts in, so only runs that leave the block, and long ones, are left to the combine kernel.
// What bounds it is latency: 40 % of the issue slots, 41 of the warp slots, 40 of DRAM (26 skewed tables of 21 500 lookups of 64
// floats; 128 floats 43, 44 and 44; 32 floats 41, 41 and 27; 256 floats 35, 42 and 44).  Rows one after the other as their runs end, and a thread's keys by
// itself, took 46 us for those tables (with the combine kernel 58; now 42 and 50), 100 us for 40 tables of 32 900 of 16 floats (now
// 84), 16 for 11 of 10 700 of 48 (the same; with the combine kernel 21, now 19).  Additions and steps take two floats an
// instruction.
constexpr int kShortSpan = 8;                              // most windows whose parts one lane group adds
constexpr int kWaThreads = 128;

// 16 bytes of a row: two packed pairs of floats.  Pairs are added and multiplied two floats an instruction, each rounded as by
// itself.
struct Quad { uint64_t a, b; };
__device__ __forceinline__ uint64_t add_pair(uint64_t x, uint64_t y) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(x), "l"(y));
  return d;
}
__device__ __forceinline__ uint64_t fma_pair(uint64_t x, uint64_t y, uint64_t z) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(x), "l"(y), "l"(z));
  return d;
}
__device__ __forceinline__ Quad add_quad(Quad x, Quad y) { return Quad{add_pair(x.a, y.a), add_pair(x.b, y.b)}; }
__device__ __forceinline__ float4 floats_of(Quad q) {
  return make_float4(__uint_as_float((uint32_t)q.a), __uint_as_float((uint32_t)(q.a >> 32)), __uint_as_float((uint32_t)q.b),
                     __uint_as_float((uint32_t)(q.b >> 32)));
}
__device__ __forceinline__ Quad quad_nc(const char* p) {
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(p));
  return Quad{v.x, v.y};
}
__device__ __forceinline__ Quad quad_at(const char* p) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
  return Quad{v.x, v.y};
}

// The columns of a lane in a group of G, NV float4 each G float4 apart: byte offsets inside a row.  Exact: the row is
// G * NV float4 wide.  Otherwise a lane whose column lies beyond the row reads another one in its place and stores nothing.
template <int G, int NV, bool Exact>
struct LaneColumns {
  int nvec, lane;
  __device__ __forceinline__ LaneColumns(int nvec_, int lane_) : nvec(nvec_), lane(lane_) {}
  __device__ __forceinline__ bool inside(int v) const { return Exact || lane + v * G < nvec; }
  __device__ __forceinline__ uint32_t first() const { return 16u * (uint32_t)(Exact || lane < nvec ? lane : 0); }
  __device__ __forceinline__ uint32_t next(int v) const { return inside(v) ? 16u * v * G : 0u; }   // beyond first()
};

// Sum over the group of g^2, the same in every lane: a lane's own columns first, then a tree over the lanes.
template <int G, int NV>
__device__ __forceinline__ float square_sum(const float4 (&g)[NV], unsigned mask) {
  float ss = 0.f;
#pragma unroll
  for (int v = 0; v < NV; ++v)
    ss += __fmaf_rn(g[v].w, g[v].w, __fmaf_rn(g[v].z, g[v].z, __fmaf_rn(g[v].x, g[v].x, __fmul_rn(g[v].y, g[v].y))));
#pragma unroll
  for (int off = G / 2; off >= 1; off >>= 1) ss += __shfl_xor_sync(mask, ss, off, G);
  return ss;
}

// The row's new state and the factor of its gradient.  Wide: rows of more than 128 floats, whose quotients are rounded exactly;
// for the others the reciprocal of D is loop-invariant and the quotient is within 2 ulp.
template <bool Wide>
__device__ __forceinline__ float next_state(float st, float ss, int D) {
  return Wide ? st + ss / (float)D : __fmaf_rn(ss, 1.0f / (float)D, st);
}
template <bool Wide>
__device__ __forceinline__ float step_scale(float lr, float sn, float eps) {
  return Wide ? lr / (sqrtf(sn) + eps) : __fdividef(lr, sqrtf(sn) + eps);
}

// Row-wise Adagrad on one row whose gradient is in the lanes' registers, NV float4 per lane (column lane + v*G).
template <int G, int NV, bool Wide>
__device__ __forceinline__ void adagrad_row_nv(const float4 (&g)[NV], uint32_t key, int lane, int nvec, int D,
                                               unsigned gmask, float* __restrict__ tables,
                                               float* __restrict__ row_state, float lr, float eps) {
  float4* row = reinterpret_cast<float4*>(tables + (int64_t)key * D);
  float4 r[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) r[v] = (lane + v * G < nvec) ? row[lane + v * G] : make_float4(0.f, 0.f, 0.f, 0.f);
  const float st = row_state[key];
  const float ss = square_sum<G, NV>(g, gmask);
  const float sn = next_state<Wide>(st, ss, D), scale = step_scale<Wide>(lr, sn, eps);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    if (lane + v * G < nvec) {
      float4 o = r[v];
      o.x -= scale * g[v].x; o.y -= scale * g[v].y; o.z -= scale * g[v].z; o.w -= scale * g[v].w;
      row[lane + v * G] = o;
    }
  }
  __syncwarp(gmask);
  if (lane == 0) row_state[key] = sn;
}

template <int G, int NV, int KB, int kMinBlocks, int KR, bool Exact, bool Wide>
__global__ void __launch_bounds__(kWaThreads, kMinBlocks)
window_apply_kernel(const uint32_t* __restrict__ keys, const int32_t* __restrict__ sbag,
                    const int32_t* __restrict__ uidx, int L, uint32_t sentinel, int T, uint32_t N, int D, int B,
                    const float* __restrict__ grad, int64_t ld_grad, int col0, float* __restrict__ partial,
                    int32_t* __restrict__ long_list, int32_t* __restrict__ scalars, int nwin,
                    int32_t* __restrict__ d_status, float* __restrict__ tables, float* __restrict__ row_state,
                    float lr, float eps) {
  wait_for_previous_kernel();
  constexpr int kGroups = kWaThreads / G, kPos = kGroups * kWin;
  constexpr unsigned kAll = 0xffffffffu;
  __shared__ __align__(16) uint32_t s_key[kPos];
  __shared__ __align__(16) int32_t s_row[kPos];            // float4 index of the lookup's gradient row
  __shared__ uint32_t s_valid[kPos / 32], s_head[kPos / 32];
  static_assert(kPos % 32 == 0, "whole warps stage positions");
  const int grp = threadIdx.x / G, lane = threadIdx.x % G;
  if (!ws_matches(scalars, L, sentinel, d_status)) return;
  const LaneColumns<G, NV, Exact> col(D >> 2, lane);
  const uint32_t row_bytes = (uint32_t)D * 4u;
  const int p0 = (int)blockIdx.x * kPos;                   // the block's first position (below L < 2^31)
  // ---- keys, gradient rows and run structure of the block's positions, 32 consecutive ones per warp and round
  {
    const int nvec = D >> 2, ld4 = (int)(ld_grad >> 2);    // B * ld_grad / 4 < 2^31 is checked on the host
    int t = (int)((uint32_t)sbag[p0] / (uint32_t)B);       // table of the block's first position
#pragma unroll
    for (int e0 = 0; e0 < kPos; e0 += kWaThreads) {
      const int e = e0 + threadIdx.x, j = p0 + e;
      if (kPos % kWaThreads != 0 && e >= kPos) break;      // (whole warps)
      uint32_t key = sentinel, before = sentinel;
      int32_t row = -1;
      if (j < L) {
        key = keys[j];
        const int sb = sbag[j];
        if (j > 0) before = keys[j - 1];
        if (key < sentinel) {
          int b = sb - t * B;                              // bags are table-major: bag = t*B + b
          if ((uint32_t)b >= (uint32_t)B) { t = (int)((uint32_t)sb / (uint32_t)B); b = sb - t * B; }
          // a consistent workspace never fails these; an inconsistent one must not turn into a wild access
          if (sb >= 0 && t < T && key - (uint32_t)t * N < N) row = b * ld4 + t * nvec;
          else key = sentinel;
        }
      }
      const bool valid = row >= 0, head = valid && (before != key || (e & (kWin - 1)) == 0);
      if (head) {                                          // request the run's row into L2
        const char* trow = reinterpret_cast<const char*>(tables) + (uint64_t)key * row_bytes;
        if (Exact) {
#pragma unroll
          for (int o = 0; o < G * NV * 16; o += 128) prefetch_l2(trow + o);
        } else {
          for (uint32_t o = 0; o < row_bytes; o += 128) prefetch_l2(trow + o);
        }
        prefetch_l2(row_state + key);
      }
      s_key[e] = key;
      s_row[e] = max(row, 0);                              // skipped lookups follow every run: what is added for them goes nowhere
      const uint32_t vb = __ballot_sync(kAll, valid), hb = __ballot_sync(kAll, head);
      if ((threadIdx.x & 31) == 0) { s_valid[e >> 5] = vb; s_head[e >> 5] = hb; }
    }
  }
  __syncthreads();
  const int w0 = grp * kWin, win = p0 / kWin + grp;        // the group's window: first position inside the block, number
  const uint32_t vm = (s_valid[w0 >> 5] >> (w0 & 16)) & 0xffffu, hm = (s_head[w0 >> 5] >> (w0 & 16)) & 0xffffu;
  // a run ends where the next position starts another run, is a skipped lookup, or lies outside the window
  const uint32_t tm = vm & ((hm >> 1) | (~vm >> 1) | 0x8000u), first_tail = tm & (0u - tm);
  bool first_open = false, last_open = false;              // the first / last run goes on in a neighbouring window
  if (vm & 1u) first_open = p0 + w0 > 0 && (w0 > 0 ? s_key[w0 - 1] : keys[p0 - 1]) == s_key[w0];
  if (vm >> (kWin - 1)) {
    const int j = p0 + w0 + kWin;
    last_open = j < L && (w0 + kWin < kPos ? s_key[w0 + kWin] : keys[j]) == s_key[w0 + kWin - 1];
  }
  // runs that end here and are complete; the others leave a partial sum
  const uint32_t um = tm & ~(first_open ? first_tail : 0u) & ~(last_open ? 0x8000u : 0u);
  const char* const gl = reinterpret_cast<const char*>(grad + col0) + col.first();   // col0 is a multiple of 4
  char* const tl = reinterpret_cast<char*>(tables) + col.first();
  float* const pl = partial + (int64_t)win * 2 * D + (col.first() >> 2);

  // a row's step from the sum of its gradients
  auto step = [&](const Quad (&g)[NV], const Quad (&r)[NV], float st, uint32_t key, bool store) {
    float4 f[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) f[v] = col.inside(v) ? floats_of(g[v]) : make_float4(0.f, 0.f, 0.f, 0.f);
    const float ss = square_sum<G, NV>(f, kAll);
    const float sn = next_state<Wide>(st, ss, D), scale = -step_scale<Wide>(lr, sn, eps);
    const uint64_t s2 = (uint64_t)__float_as_uint(scale) << 32 | __float_as_uint(scale);
    __syncwarp();                                          // every lane has read the state
    if (store) {
      char* const p = tl + (uint64_t)key * row_bytes;
#pragma unroll
      for (int v = 0; v < NV; ++v)
        if (col.inside(v))
          *reinterpret_cast<ulonglong2*>(p + 16 * v * G) = make_ulonglong2(fma_pair(s2, g[v].a, r[v].a), fma_pair(s2, g[v].b, r[v].b));
      if (lane == 0) row_state[key] = sn;
    }
  };

  Quad acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = Quad{0ull, 0ull};
#pragma unroll 1
  for (int i0 = 0; i0 < kWin;) {
    if constexpr (KR > 0) {
      // no run of the warp's windows ends in the next KR positions: no row is needed, and there is room for more gradients
      if (i0 + KR <= kWin && !__any_sync(kAll, tm >> i0 & ((1u << KR) - 1u))) {
        Quad gv[KR][NV];
#pragma unroll
        for (int u = 0; u < KR; ++u) {
          const char* const p = gl + (int64_t)s_row[w0 + i0 + u] * 16;
#pragma unroll
          for (int v = 0; v < NV; ++v) gv[u][v] = quad_nc(p + col.next(v));
        }
#pragma unroll
        for (int u = 0; u < KR; ++u)
#pragma unroll
          for (int v = 0; v < NV; ++v) acc[v] = add_quad(acc[v], gv[u][v]);
        i0 += KR;
        continue;
      }
    }
    Quad gv[KB][NV], rv[KB][NV];
    float st[KB];
    uint32_t key[KB];
    const uint32_t tails = tm >> i0, upds = um >> i0;
#pragma unroll
    for (int u = 0; u < KB; ++u) {
      const char* const p = gl + (int64_t)s_row[w0 + i0 + u] * 16;
#pragma unroll
      for (int v = 0; v < NV; ++v) gv[u][v] = quad_nc(p + col.next(v));
    }
#pragma unroll
    for (int u = 0; u < KB; ++u) {
      key[u] = s_key[w0 + i0 + u];
      st[u] = 0.f;
#pragma unroll
      for (int v = 0; v < NV; ++v) rv[u][v] = Quad{0ull, 0ull};
      if ((upds >> u) & 1u) {
        const char* const p = tl + (uint64_t)key[u] * row_bytes;
        st[u] = row_state[key[u]];
#pragma unroll
        for (int v = 0; v < NV; ++v) rv[u][v] = quad_at(p + col.next(v));
      }
    }
#pragma unroll
    for (int u = 0; u < KB; ++u) {
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = add_quad(acc[v], gv[u][v]);
      const bool tail = (tails >> u) & 1u, upd = (upds >> u) & 1u;
      if (__any_sync(kAll, tail)) {
        step(acc, rv[u], st[u], key[u], upd);
        if (tail && !upd) {
          // the run goes on in a neighbouring window: its part goes to the window's partial slot
          // (slot 0 when the run holds the window's first position)
          float* const dst = pl + ((first_tail >> (i0 + u)) & 1u ? 0 : D);
#pragma unroll
          for (int v = 0; v < NV; ++v)
            if (col.inside(v)) *reinterpret_cast<ulonglong2*>(dst + 4 * v * G) = make_ulonglong2(acc[v].a, acc[v].b);
        }
        if (tail) {
#pragma unroll
          for (int v = 0; v < NV; ++v) acc[v] = Quad{0ull, 0ull};
        }
      }
    }
    i0 += KB;
  }
  // ---- a run that starts in this window and goes on: its parts are added here, in window order, if they are all of this
  // block and no more than kShortSpan; otherwise the row enters the combine kernel's list
  __syncthreads();                                         // the block's parts are in memory
  const bool starts = last_open && !(first_open && first_tail == 0x8000u);
  const uint32_t key = s_key[w0 + kWin - 1];
  int span = 0;                                            // windows the run covers, 0: too many or not all of them here
  if (starts) {
    int e = grp + 1;
    while (e < kGroups && e - grp < kShortSpan - 1 && s_key[e * kWin + kWin - 1] == key &&
           (e + 1 == kGroups || s_key[e * kWin + kWin] == key)) ++e;
    bool ends = e < kGroups;
    if (ends && s_key[e * kWin + kWin - 1] == key) {       // up to the window's end: does the next one begin with another row?
      const int j = p0 + (e + 1) * kWin;
      ends = j >= L || (e + 1 < kGroups ? s_key[e * kWin + kWin] : keys[j]) != key;
    }
    if (ends) {
      span = e - grp + 1;
    } else if (lane == 0) {
      const int u_at = uidx[p0 + w0 + kWin - 1];
      const int slot = atomicAdd(&scalars[1], 1);
      if (slot < nwin) long_list[slot] = u_at;             // at most one such run per window
    }
  }
  if (!__any_sync(kAll, span > 0)) return;
  Quad rv[NV];
  float st = 0.f;
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = rv[v] = Quad{0ull, 0ull};
  if (span > 0) {
    st = row_state[key];
#pragma unroll
    for (int v = 0; v < NV; ++v) rv[v] = quad_at(tl + (uint64_t)key * row_bytes + col.next(v));
  }
  for (int k0 = 0; k0 < span; k0 += KB) {
    Quad pv[KB][NV];
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      // the run's part is in slot 0 of a window whose first position it holds: of all but perhaps the first
      const float* const src = pl + (int64_t)(k0 + k) * 2 * D + (k0 + k > 0 || first_tail == 0x8000u ? 0 : D);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        pv[k][v] = Quad{0ull, 0ull};
        if (k0 + k < span) pv[k][v] = quad_at(reinterpret_cast<const char*>(src) + col.next(v));
      }
    }
#pragma unroll
    for (int k = 0; k < KB; ++k)
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = add_quad(acc[v], pv[k][v]);
  }
  step(acc, rv, st, key, span > 0);
}

// ---- (5) rows whose run crosses window edges: add their window partials ---------------------------
// Rows spanning up to kShort windows: one lane group adds the partials in window order.  Longer rows: one
// block per row, lane group j adds the partials of windows k0+j, k0+j+groups, ... in ascending order and
// the group sums are then added in group order.  The association is fixed by the
// segment's position alone (the order of the list does not matter).
// FUSE (behind window_apply_kernel): the combined sum is not stored; the row is updated here.
template <int G, int NV, bool FUSE, bool Wide>
__global__ void __launch_bounds__(256)
combine_rows_kernel(const int32_t* __restrict__ seg, int32_t* scalars,
                    const int32_t* __restrict__ long_list, int nwin, int nb_long, int D, const float* __restrict__ partial,
                    float* __restrict__ gsum, int64_t L, uint32_t sentinel, int64_t umax,
                    const int32_t* __restrict__ uniq, float* __restrict__ tables, float* __restrict__ row_state,
                    float lr, float eps) {
  wait_for_previous_kernel();
  constexpr int kGroups = 256 / G;
  const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << ((threadIdx.x & 31) / G * G));
  extern __shared__ float4 s_part[];                       // [kGroups][D/4]
  const int grp = threadIdx.x / G, lane = threadIdx.x % G;
  const int nvec = D >> 2;
  if (!ws_matches(scalars, L, sentinel, nullptr)) return;
  const int n = min(scalars[1], nwin);
  // The block that finds all others past this point empties the list in the end, so that the apply half can be repeated on
  // one sort without a memset.
  __syncthreads();                                         // every thread of the block has read the list's length
  int ticket = 0;
  if (threadIdx.x == 0) ticket = atomicAdd(scalars + kListTicket, 1);
  // Spans of up to kShort windows: one lane group per row, which requests kBatch partials at a time and adds them in
  // window order.  Only the rows with longer spans (the hottest of a skewed table) take a whole block each: a
  // block works through its rows one after the other, so that path must stay short -- but a lane group walking a
  // long span is a chain of dependent rounds at the kernel's tail: of 2 / 4 / 8 / 32 / 128 windows, 8 was the
  // fastest (the call 66.7 us against 69.5 with 32 and 89.8 with 128).
  constexpr int kShort = kShortSpan;
  constexpr int kBatch = NV <= 1 ? 8 : (NV <= 2 ? 4 : 2);
  const bool do_short = nb_long == 0 || (int)blockIdx.x >= nb_long;
  const bool do_long = nb_long == 0 || (int)blockIdx.x < nb_long;
  const int a_blk = nb_long == 0 ? (int)blockIdx.x : (int)blockIdx.x - nb_long;
  const int a_blocks = nb_long == 0 ? (int)gridDim.x : (int)gridDim.x - nb_long;
  const int b_blocks = nb_long == 0 ? (int)gridDim.x : nb_long;
  // phase A
  for (int i = a_blk * kGroups + grp; do_short && i < n; i += a_blocks * kGroups) {
    const int u = long_list[i];
    if (u < 0 || u >= umax) continue;
    const int s0 = seg[u], s1 = seg[u + 1];
    if (s0 < 0 || s1 <= s0 || s1 > L) continue;
    const int k0 = s0 / kWin, k1 = (s1 - 1) / kWin;
    if (k1 - k0 + 1 > kShort) continue;
    float4 t[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) t[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int kb = k0; kb <= k1; kb += kBatch) {
      float4 pv[kBatch][NV];
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int k = kb + j;
        const int slot = (s0 <= k * kWin) ? 0 : 1;         // the run covers the window's first position -> slot 0
        const float4* p = reinterpret_cast<const float4*>(partial + ((int64_t)k * 2 + slot) * D);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int c = lane + v * G;
          pv[j][v] = (k <= k1 && c < nvec) ? p[c] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
#pragma unroll
      for (int j = 0; j < kBatch; ++j)
#pragma unroll
        for (int v = 0; v < NV; ++v) t[v] = add4(t[v], pv[j][v]);   // adding zeros for absent windows changes nothing
    }
    if (!FUSE) {
      float4* dst = reinterpret_cast<float4*>(gsum + (int64_t)u * D);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int c = lane + v * G;
        if (c < nvec) dst[c] = t[v];
      }
    }
    if (FUSE) {
      const uint32_t key = (uint32_t)uniq[u];
      if (key < sentinel) adagrad_row_nv<G, NV, Wide>(t, key, lane, nvec, D, gmask, tables, row_state, lr, eps);
    }
  }
  // phase B: long spans, the whole block per row.  The block owns the list entries blockIdx.x + k*gridDim.x;
  // its threads look at 256 of them at a time (one round of loads) and queue the long ones.
  __shared__ int s_long[256];
  __shared__ int s_nlong;
  for (int64_t base = 0; do_long && (int64_t)blockIdx.x + base * b_blocks < n; base += 256) {
    if (threadIdx.x == 0) s_nlong = 0;
    __syncthreads();
    {
      const int64_t i = (int64_t)blockIdx.x + (base + threadIdx.x) * b_blocks;
      if (i < n) {
        const int u = long_list[i];
        if (u >= 0 && u < umax) {
          const int s0 = seg[u], s1 = seg[u + 1];
          if (s0 >= 0 && s1 > s0 && s1 <= L && (s1 - 1) / kWin - s0 / kWin + 1 > kShort) s_long[atomicAdd(&s_nlong, 1)] = u;
        }
      }
    }
    __syncthreads();
    const int nlong = s_nlong;
  for (int q = 0; q < nlong; ++q) {
    const int u = s_long[q];                               // checked above; uniform over the block
    const int s0 = seg[u], s1 = seg[u + 1];
    const int k0 = s0 / kWin, k1 = (s1 - 1) / kWin;
    float4 acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    // (four windows of a group in flight by hand instead of the compiler's unrolling: 22.5 -> 28.7 us for 26 skewed tables)
    for (int k = k0 + grp; k <= k1; k += kGroups) {
      const int slot = (s0 <= k * kWin) ? 0 : 1;
      const float4* p = reinterpret_cast<const float4*>(partial + ((int64_t)k * 2 + slot) * D);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int c = lane + v * G;
        if (c < nvec) acc[v] = add4(acc[v], p[c]);
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int c = lane + v * G;
      if (c < nvec) s_part[grp * nvec + c] = acc[v];
    }
    __syncthreads();
    if (grp == 0) {
      const int used = min(kGroups, k1 - k0 + 1);
      float4* dst = reinterpret_cast<float4*>(gsum + (int64_t)u * D);
      float4 tt[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int c = lane + v * G;
        tt[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c < nvec) {
          float4 t = s_part[c];
          for (int j = 1; j < used; ++j) t = add4(t, s_part[j * nvec + c]);
          if (!FUSE) dst[c] = t;
          tt[v] = t;
        }
      }
      if (FUSE) {
        const uint32_t key = (uint32_t)uniq[u];
        if (key < sentinel) adagrad_row_nv<G, NV, Wide>(tt, key, lane, nvec, D, gmask, tables, row_state, lr, eps);
      }
    }
    __syncthreads();
  }
  }
  if (threadIdx.x == 0 && ticket == (int)gridDim.x - 1) { scalars[1] = 0; scalars[kListTicket] = 0; }
}

// ---- (6) row-wise Adagrad, one lane group per distinct row (what window_reduce_kernel summed) ----------------------------------
//   g = gsum[u];  s = state + mean_d g^2;  row -= lr * g / (sqrt(s) + eps)
template <int G, int NV>
__global__ void __launch_bounds__(256)
apply_rows_kernel(const int32_t* __restrict__ uniq, const int32_t* __restrict__ scalars, int D,
                  const float* __restrict__ gsum, float* __restrict__ tables, float* __restrict__ row_state,
                  float lr, float eps, int64_t L, uint32_t sentinel, int64_t umax) {
  wait_for_previous_kernel();
  constexpr int kGroups = 256 / G;
  const int grp = threadIdx.x / G, lane = threadIdx.x % G;
  const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << ((threadIdx.x & 31) / G * G));
  if (!ws_matches(scalars, L, sentinel, nullptr)) return;
  const int64_t u = (int64_t)blockIdx.x * kGroups + grp;
  if (u >= min((int64_t)scalars[0], umax)) return;
  const uint32_t key = (uint32_t)uniq[u];
  const int nvec = D >> 2;
  const float4* p = reinterpret_cast<const float4*>(gsum + u * D);   // on its way beside the key
  float4 g[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) g[v] = lane + v * G < nvec ? p[lane + v * G] : make_float4(0.f, 0.f, 0.f, 0.f);
  if (key >= sentinel) return;                             // never true for a consistent workspace
  adagrad_row_nv<G, NV, true>(g, key, lane, nvec, D, gmask, tables, row_state, lr, eps);
}

// Lanes a window, float4 a lane, positions a batch, blocks per SM (of 128 threads: 8 leave a thread 64 registers, 10 leave 48),
// positions at once where no run ends (0: as any others).  A request should cover 128 bytes of a row: groups of 4 lanes with 4
// float4 each move rows of 256 bytes at half the rate (random rows of 7 GB: 8.7 G a second, groups of 8 or 16 15.9 G).  More warps
// beat more requests a warp: 16 float4 in flight a lane, at 120 registers, took 62 us where 8, at 64, take 51.
template <int G_, int NV_, int KB_, int kMinBlocks_, int KR_> struct WindowShape {
  static constexpr int G = G_, NV = NV_, KB = KB_, kMinBlocks = kMinBlocks_, KR = KR_;
};
// By the float4 a row has, rounded up to a power of two.  `few` is for up to kFew windows per SM, fewer than its blocks hold at
// once: then a window's own rounds are all the time there is, and larger batches or more lanes for them are what counts.  Where
// that takes 128 registers a thread, it is for one block per SM, two of the wider rows: with four, three replicas of an odd-sized
// model (48 floats, 50 windows per SM) take 109 us a round instead of 102, though the call alone is a tenth faster up to there.
// us of the update half, 26 tables (of 256 floats 10), with one shape for any number of windows (rows of 128 floats: one position a
// batch at 48 registers, which spilled) -> now, for 20 000 lookups a table hit once / 66 / 200 times a row, and Zipf 1.2;
// then 8 windows per SM, uniform ids and 16 lookups a row:
template <int kQuads> struct WindowShapeFor;
template <> struct WindowShapeFor<4> {                     // 16 floats 19 / 14 / 20 / 32 (8 blocks 19 / 14 / 20 / 33); 12 floats 9.9, 7.6 -> 9.4, 7.4
  static constexpr int kFew = 32;
  using many = WindowShape<4, 1, 4, 7, 0>;
  using few = WindowShape<4, 1, 8, 4, 0>;
};
template <> struct WindowShapeFor<8> {                     // 32 floats 29 / 20 / 27 / 39 -> 24 / 17 / 22 / 38, 17 to 31 floats alike;
  static constexpr int kFew = 120;                         // 4000 lookups a table `few` 15, `many` 17
  using many = WindowShape<4, 2, 2, 8, 4>;
  using few = WindowShape<8, 1, 2, 10, 0>;
};
template <> struct WindowShapeFor<16> {                    // 64 floats 47 / 22 / 29 / 55 -> 47 / 22 / 28 / 54, 48 floats 47 / 25 / 31 / 60 ->
  static constexpr int kFew = 16;                          // 48 / 24 / 30 / 61; 48 floats 14.8, 11.5 -> 12.1, 10.4
  using many = WindowShape<8, 2, 2, 8, 8>;
  using few = WindowShape<8, 2, 4, 4, 0>;
};
template <> struct WindowShapeFor<32> {                    // 128 floats 87 / 37 / 39 / 89 -> 85 / 36 / 37 / 85, 100 floats
  static constexpr int kFew = 16;                          // 92 / 40 / 41 / 101 -> 87 / 37 / 38 / 94; 100 floats 18.7, 12.2 -> 12.2, 9.8
  using many = WindowShape<16, 2, 2, 8, 4>;
  using few = WindowShape<16, 2, 4, 4, 0>;
};
template <> struct WindowShapeFor<64> {                    // 256 floats 67 / - / - / 77 -> 65 / - / - / 72, 160 floats 63 / - / - / 73 ->
  static constexpr int kFew = 28;                          // 57 / - / - / 65; 20 windows an SM `few` 17 to 20, `many` 18 to 22
  using many = WindowShape<32, 2, 2, 8, 4>;
  using few = WindowShape<32, 2, 2, 6, 0>;
};

template <int G, int NV, bool kFuse>
static void launch_reduce_as(const BwdPlan& p, char* ws, const uint32_t* keys, int T, int64_t N,
                          int D, int B, const float* grad, int64_t ld_grad, int col0, float* tables,
                          float* row_state, float lr, float eps, int32_t* d_status, cudaStream_t st) {
  constexpr int kGroups = 256 / G;
  const uint64_t maxkey = (uint64_t)T * (uint64_t)N;
  const uint64_t umax = (uint64_t)p.L < maxkey ? (uint64_t)p.L : maxkey;
  const uint32_t sentinel = (uint32_t)((uint64_t)T * (uint64_t)N);
  float* partial = reinterpret_cast<float*>(ws + p.off_partial);
  float* gsum = reinterpret_cast<float*>(ws + p.off_gsum);
  const unsigned blocks = (unsigned)((p.nwin + kGroups - 1) / kGroups);
  int32_t* scalars = reinterpret_cast<int32_t*>(ws + p.off_scalars);
  int32_t* long_list = reinterpret_cast<int32_t*>(ws + p.off_long);
  int32_t* seg = reinterpret_cast<int32_t*>(ws + p.off_seg);
  int32_t* uniq = reinterpret_cast<int32_t*>(ws + p.off_uniq);
  constexpr bool kWide = NV == 2;                          // (32 lanes hold up to 128 floats with one float4 each)
  if constexpr (kFuse) {
    auto window = [&](auto shape) {
      using S = decltype(shape);
      constexpr int kPos = kWaThreads / S::G * kWin;
      SS_TIMED("window_apply_kernel", st);
      auto go = [&](auto kernel) {
        launch_dependent(kernel, (unsigned)((p.L + kPos - 1) / kPos), kWaThreads, 0, st, keys, reinterpret_cast<int32_t*>(ws + p.off_sbag),
                         reinterpret_cast<int32_t*>(ws + p.off_uidx), (int)p.L, sentinel, T, (uint32_t)N, D, B, grad, ld_grad, col0,
                         partial, long_list, scalars, p.nwin, d_status, tables, row_state, lr, eps);
      };
      if (D == S::G * S::NV * 4) go(window_apply_kernel<S::G, S::NV, S::KB, S::kMinBlocks, S::KR, true, kWide>);
      else go(window_apply_kernel<S::G, S::NV, S::KB, S::kMinBlocks, S::KR, false, kWide>);
    };
    using Shapes = WindowShapeFor<G * NV>;
    if (p.nwin > Shapes::kFew * num_sms()) window(typename Shapes::many());
    else if constexpr (Shapes::kFew > 0) window(typename Shapes::few());
  } else {
    SS_TIMED("window_reduce_kernel", st);
    launch_dependent(window_reduce_kernel<G, NV>, blocks, 256, 0, st, 
        keys, reinterpret_cast<int32_t*>(ws + p.off_sbag), reinterpret_cast<int32_t*>(ws + p.off_uidx), p.L, sentinel, N, D,
        B, grad, ld_grad, col0, gsum, partial, long_list, scalars, p.nwin, (int64_t)umax, d_status);
  }
  {
    SS_TIMED("combine_rows_kernel", st);
    // The long spans and the short ones are two chains of dependent loads: with enough blocks the first part of the grid takes the
    // long ones and the rest the short ones, so that the chains run side by side.  Half of 8 blocks per SM for each where the
    // window kernel leaves all crossing runs, or leaves its block at every fourth window (wide rows; with a quarter of 5 per SM for
    // the short spans 16 us instead of 14 where rows are looked up 66 times).  Behind the others few short spans are left, and most
    // of 8 per SM only took other kernels' places: with 5, a quarter of them for the short spans, four replicas of the ordinary
    // model take 452 us a round instead of 455, three of an odd-sized one 104 instead of 106 (the call alone 51 and 51, 93 and 93
    // for 128 floats; 3 per SM: 449 and 103, but 54 and 100).
    const bool few_short = kFuse && (!kWide || p.nwin <= WindowShapeFor<64>::kFew * num_sms());
    const int per_sm = few_short ? 5 : 8, cblocks = p.nwin < num_sms() * per_sm ? p.nwin : num_sms() * per_sm;
    const int long_blocks = cblocks < 4 ? 0 : few_short ? cblocks * 3 / 4 : cblocks / 2;   // 0: every block does both
    // fused rows of at least eight float4: two float4 per lane, half as many lanes per row, twice as many rows in flight
    constexpr int CG = (kFuse && !kWide && G >= 8) ? G / 2 : G, CNV = (kFuse && G >= 8) ? 2 : NV;
    launch_dependent(combine_rows_kernel<CG, CNV, kFuse, kWide>, cblocks, 256, (size_t)(256 / CG) * D * 4, st, 
        seg, scalars, long_list, p.nwin, long_blocks, D, partial, gsum, p.L, sentinel, (int64_t)umax, uniq, tables, row_state, lr, eps);
  }
  if constexpr (!kFuse) {
    // every distinct row is updated from its sum in gsum
    const uint64_t per_block = (uint64_t)kGroups;
    const unsigned ublocks = (unsigned)((umax + per_block - 1) / per_block);
    SS_TIMED("apply_rows_kernel", st);
    launch_dependent(apply_rows_kernel<G, NV>, ublocks, 256, 0, st, uniq, scalars, D, gsum, tables, row_state, lr, eps, p.L, sentinel,
                                                      (int64_t)umax);
  }
}

// Rows of up to 128 floats are updated from the window kernel, wider ones than 256 from their sums in memory.  In between the sums'
// way through memory and back is what the fused kernel saves, a chain of dependent rounds for the 16 positions of a window what it
// costs; so it needs windows enough to fill the SMs and rows that are not all popular (lookups per row of the tables: at least that
// many a row on average, whichever rows they are).  us of the update half, fused / not:
//   windows per SM      uniform ids, 132 / 192 / 256 floats        Zipf 1.05
//   8                   17 / 15, 17 / 16, 16 / 16                  18 / 13, 18 / 13, 17 / 14
//   16                  18 / 18, 20 / 20, 18 / 25                  19 / 16, 20 / 17, 18 / 18
//   20                  18 / 21, 19 / 25, 18 / 34                  19 / 18, 18 / 18, 17 / 20
//   32                  25 / 32, 26 / 40, 25 / 49                  26 / 24, 25 / 25, 22 / 27
//   64                  42 / 61, 50 / 75, 54 / 84                  33 / 37, 36 / 43, 37 / 50
//   lookups per row     (135 windows per SM for 132 floats, 90 for 160 to 256; 132 / 160 / 256 floats)
//   25                  29 / 27, 27 / 28, 28 / 30
//   66                  30 / 24, 29 / 24, 30 / 26
//   200                 26 / 24, 24 / 23, 25 / 25
//   4000                29 / 28, 28 / 29, 27 / 28
constexpr int kFuseWindows = 16, kFuseHits = 32;           // per SM; per row
template <int G, int NV>
static void launch_reduce(const BwdPlan& p, char* ws, const uint32_t* keys, int T, int64_t N,
                          int D, int B, const float* grad, int64_t ld_grad, int col0, float* tables,
                          float* row_state, float lr, float eps, int32_t* d_status, cudaStream_t st) {
  auto as = [&](auto fuse) {
    launch_reduce_as<G, NV, decltype(fuse)::value>(p, ws, keys, T, N, D, B, grad, ld_grad, col0, tables, row_state, lr, eps, d_status, st);
  };
  if constexpr (NV == 1) as(std::true_type());
  else if constexpr (NV > 2) as(std::false_type());
  else if (p.nwin >= kFuseWindows * num_sms() && p.L <= (int64_t)kFuseHits * T * N) as(std::true_type());
  else as(std::false_type());
}

#define SS_DISPATCH_GNV(D_, CALL)                                                 \
  do {                                                                            \
    const int nvec__ = (D_) / 4;                                                  \
    if (nvec__ <= 4) { CALL(4, 1); }                                              \
    else if (nvec__ <= 8) { CALL(8, 1); }                                         \
    else if (nvec__ <= 16) { CALL(16, 1); }                                       \
    else if (nvec__ <= 32) { CALL(32, 1); }                                       \
    else if (nvec__ <= 64) { CALL(32, 2); }                                       \
    else if (nvec__ <= 128) { CALL(32, 4); }                                      \
    else { CALL(32, 8); }                                                         \
  } while (0)

// Closes an empty sort.
__global__ void unique_finish_kernel(const __grid_constant__ SortOut o) { wait_for_previous_kernel(); finish_unique(o, 0u); }

// Whether the bucket sort takes a problem, how many lookups it gives a range, and the most ranges there can be, whatever the
// tables' lengths: a block for each.  Every further range reads the index list once more and holds an SM, so a table gets as
// few ranges as hold its lookups (four replicas of the ordinary model 478 us a round with two ranges a table, 494 with three).
// Few tables are cut finer: down to 5500 lookups a range, while that takes no more than a quarter of the SMs, where the sort is
// a call by itself, which runs beside other work (three replicas of 11 tables of 10 700 lookups 104 us a round; 107 with 2750 a
// range, 121 with 1400 and half of the SMs); down to 1400, up to six ranges on a third of them, where the update waits for the sort
// in the same call.  One such call alone would take half of the SMs (12 tables of 10 200 lookups: by the rule above 50 us, half 41,
// a third 41), but several at a time lose more than that: three of 12 tables 62 / 61 / 54, four 72 / 80 / 68, four of 11
// 64 / 73 / 63, four of 16 of 20 500 116 / 126 / 116.  Up to three ranges a table are worth half of the SMs all the same (22 of
// 25 900, Zipf 1.2: 177 us with two ranges, 147 with three; 26 of 5100 42 with one, 37 with two); four calls at a time lose there
// (132 -> 143 for 22 of 25 900).  With eight ranges a table's list is walked too often (3 of 32 800, Zipf 1.2: 71 us, six 66).
// Blocks without a range cost nothing that could be measured.
static bool plan_bucket_sort(int T, int64_t N, int B, int64_t L, bool waited_for, BucketSort* a, int64_t* blocks, int* nb) {
  const int64_t avg = (L + T - 1) / T;
  if (B > 65535 || avg > 44000) return false;              // bag numbers, plus one, take 16 bits
  int64_t C = (avg + kBsRange - 1) / kBsRange;
  const int64_t least = waited_for ? 1400 : 5500, fine = (avg + least - 1) / least, most = waited_for ? 6 : kBsMaxBuckets;
  int64_t room = num_sms() / (waited_for ? 3 : 4) / T;
  if (waited_for && room < 3) room = num_sms() / 2 / T < 3 ? num_sms() / 2 / T : 3;
  a->per_range = kBsRange;
  if (C < fine && C < room) {
    C = fine < room ? fine : room;
    if (C > most) C = most;
    a->per_range = (int)(avg * 115 / 100 / C);             // tables a little longer than the average get no further range
  }
  if (C < 1) C = 1;
  a->T = T; a->B = B; a->N = N;
  a->ranges = T > kBsThreads ? (int)C : 0;
  int bits = 1;
  while (((uint64_t)((N + C - 1) / C - 1) >> bits) != 0) ++bits;   // of a slice of the rows; a longer range takes another pass
  const int passes = (bits + kBsDigit - 1) / kBsDigit;
  *nb = (bits + passes - 1) / passes;
  if (*nb < 5) *nb = 5;                                    // the in-block scan wants at least 32 bins
  a->cap = L < kBsCap ? (int)((L + 31) & ~(int64_t)31) : kBsCap;   // small problems leave shared memory to others
  *blocks = a->ranges > 0 ? T * C : T + L / a->per_range;
  return true;
}

template <int NB>
static ss_status launch_bucket_sort_nb(const BucketSort& a, const TiledSort& t, int64_t blocks, cudaStream_t st) {
  static bool attr_set[64];
  int dev = 0;
  SS_CUDA(current_device(&dev));
  if (dev >= 0 && dev < 64 && !attr_set[dev]) {
    SS_CUDA(cudaFuncSetAttribute(bucket_sort_kernel<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bs_smem(kBsCap, NB)));
    attr_set[dev] = true;
  }
  SS_TIMED("bucket_sort_kernel", st);
  launch_dependent(bucket_sort_kernel<NB>, (unsigned)blocks, kBsThreads, bs_smem(a.cap, NB), st, a, t);
  SS_LAUNCH_OK();
  return SS_OK;
}
static ss_status launch_bucket_sort(const BucketSort& a, const TiledSort& t, int64_t blocks, int nb, cudaStream_t st) {
  switch (nb) {
    case 5: return launch_bucket_sort_nb<5>(a, t, blocks, st);
    case 6: return launch_bucket_sort_nb<6>(a, t, blocks, st);
    case 7: return launch_bucket_sort_nb<7>(a, t, blocks, st);
    case 8: return launch_bucket_sort_nb<8>(a, t, blocks, st);
    case 9: return launch_bucket_sort_nb<9>(a, t, blocks, st);
    default: return launch_bucket_sort_nb<10>(a, t, blocks, st);
  }
}

}  // namespace ss

extern "C" {

ss_status ss_embbag_fwd(const float* tables, int T, int64_t N, int D, const int32_t* indices,
                        const int32_t* offsets, int B, float* out_f32, int64_t ld_f32, void* out_bf16,
                        int64_t ld_bf16, int col0, int32_t* d_status, ss_stream stream) {
  if (!tables || !indices || !offsets) return SS_ERR_NULL;
  if (!out_f32 && !out_bf16) return SS_ERR_NULL;
  if (T < 0 || B < 0 || N <= 0 || D <= 0 || D > 1024 || (D & 3) || col0 < 0) return SS_ERR_SHAPE;
  if ((uint64_t)T * (uint64_t)N >= (1ull << 31) || T > 65535 || (uint64_t)N * (uint64_t)(D / 4) >= (1ull << 32)) return SS_ERR_SHAPE;
  if (!ss::aligned16(tables) || (col0 & 3)) return SS_ERR_ALIGN;
  if (out_f32 && (!ss::aligned16(out_f32) || (ld_f32 & 3) || ld_f32 < col0 + (int64_t)T * D)) return SS_ERR_ALIGN;
  if (out_bf16 && ((reinterpret_cast<uintptr_t>(out_bf16) & 7u) || (ld_bf16 & 3) || ld_bf16 < col0 + (int64_t)T * D))
    return SS_ERR_ALIGN;
  ss_status st = ss::check_arch();
  if (st != SS_OK) return st;
  if ((int64_t)T * B == 0) return SS_OK;
  cudaStream_t cs = ss::as_stream(stream);
#define SS_FWD(G_, NV_)                                                                                     \
  ss::launch_fwd<G_, NV_>(tables, T, N, D, indices, offsets, B, out_f32, ld_f32, (__nv_bfloat16*)out_bf16, \
                          ld_bf16, col0, d_status, cs)
  SS_DISPATCH_GNV(D, SS_FWD);
#undef SS_FWD
  SS_LAUNCH_OK();
  return SS_OK;
}

size_t ss_embbag_bwd_workspace_bytes(int T, int64_t N, int D, int B, int64_t L) {
  (void)B;
  if (T < 0 || N <= 0 || D <= 0 || L < 0) return 0;
  return ss::make_plan(T, N, D, L).total;
}

static ss_status bwd_impl(bool do_sort, bool do_apply, float* tables, float* row_state, int T, int64_t N, int D,
                          const int32_t* indices, const int32_t* offsets, int B, int64_t L, const float* grad,
                          int64_t ld_grad, int col0, float lr, float eps, void* workspace, size_t workspace_bytes,
                          int32_t* uniq_keys, int32_t* seg_off, int32_t* perm, int32_t* d_num_unique,
                          int32_t* d_status, ss_stream stream) {
  using namespace ss;
  if (!workspace) return SS_ERR_NULL;
  if (do_sort && ((!indices && L > 0) || !offsets)) return SS_ERR_NULL;
  if (do_apply && (!tables || !row_state || !grad)) return SS_ERR_NULL;
  if (T < 0 || B < 0 || N <= 0 || D <= 0 || D > 1024 || (D & 3) || col0 < 0 || L < 0) return SS_ERR_SHAPE;
  if ((uint64_t)T * (uint64_t)N >= (1ull << 31) || L >= (1ll << 31) - kSortTile) return SS_ERR_SHAPE;
  if (!aligned16(workspace)) return SS_ERR_ALIGN;
  if (do_apply) {
    if (!aligned16(tables) || !aligned16(grad) || (ld_grad & 3) || (col0 & 3)) return SS_ERR_ALIGN;
    if (ld_grad < col0 + (int64_t)T * D || (int64_t)B * ld_grad / 4 >= (1ll << 31)) return SS_ERR_SHAPE;
  }
  const BwdPlan p = make_plan(T, N, D, L);
  if (workspace_bytes < p.total) return SS_ERR_WORKSPACE;
  ss_status stt = check_arch();
  if (stt != SS_OK) return stt;
  cudaStream_t cs = as_stream(stream);
  char* ws = reinterpret_cast<char*>(workspace);
  uint32_t* keys_a = reinterpret_cast<uint32_t*>(ws + p.off_keys_a);
  uint32_t* keys_b = reinterpret_cast<uint32_t*>(ws + p.off_keys_b);
  int32_t* pos_a = reinterpret_cast<int32_t*>(ws + p.off_pos_a);
  int32_t* pos_b = reinterpret_cast<int32_t*>(ws + p.off_pos_b);
  int32_t* bag_of = reinterpret_cast<int32_t*>(ws + p.off_bag);
  const uint32_t sentinel = (uint32_t)((uint64_t)T * (uint64_t)N);

  SortOut out{};
  out.uidx = reinterpret_cast<int32_t*>(ws + p.off_uidx); out.sbag = reinterpret_cast<int32_t*>(ws + p.off_sbag);
  out.uniq = reinterpret_cast<int32_t*>(ws + p.off_uniq); out.seg = reinterpret_cast<int32_t*>(ws + p.off_seg);
  out.perm_out = perm; out.uniq_out = uniq_keys; out.seg_out = seg_off; out.d_num_unique = d_num_unique;
  out.scalars = reinterpret_cast<int32_t*>(ws + p.off_scalars); out.d_status = d_status;
  out.L = L; out.sentinel = sentinel;
  if (L == 0 || (int64_t)T * B == 0) {
    if (do_sort) {
      SS_TIMED("unique_finish_kernel", cs);
      launch_dependent(unique_finish_kernel, 1, 1, 0, cs, out);
      SS_LAUNCH_OK();
    }
    return SS_OK;
  }
  // the sorted arrays end up in the buffers the last pass wrote
  const uint32_t* keys_sorted = (p.passes & 1) ? keys_b : keys_a;
  const int32_t* perm_sorted = (p.passes & 1) ? pos_b : pos_a;
  if (do_sort) {
    out.keys = const_cast<uint32_t*>(keys_sorted); out.perm = const_cast<int32_t*>(perm_sorted);
    int* ctl = reinterpret_cast<int*>(ws + p.off_ctl);
    TiledSort ts{};
    ts.indices = indices; ts.offsets = offsets; ts.T = T; ts.B = B; ts.N = N;
    ts.keys_a = keys_a; ts.keys_b = keys_b; ts.pos_a = pos_a; ts.pos_b = pos_b; ts.bag_of = bag_of;
    ts.hist = reinterpret_cast<uint32_t*>(ws + p.off_hist); ts.bintot = reinterpret_cast<uint32_t*>(ws + p.off_bintot);
    ts.tile_heads = reinterpret_cast<uint32_t*>(ws + p.off_heads);
    ts.ctl = ctl + kCtlTiled; ts.passes = p.passes; ts.digit_bits = p.digit_bits; ts.bins = p.bins; ts.out = out;
    BucketSort bs{};
    int64_t blocks = 0;
    int nb = 0;
    const bool bucket = plan_bucket_sort(T, N, B, L, do_apply, &bs, &blocks, &nb);
    stt = clear_words(ctl, kCtlCounts + (bucket ? T * kBsMaxBuckets : 0), cs);
    if (stt != SS_OK) return stt;
    if (bucket) {
      bs.indices = indices; bs.offsets = offsets;
      bs.fallback = ctl + kCtlFallback; bs.ticket = ctl + kCtlTicket; bs.counts = reinterpret_cast<uint32_t*>(ctl + kCtlCounts);
      bs.serial_fallback = L <= bs.cap;                    // no range can be too full: only malformed input takes the fallback
      stt = launch_bucket_sort(bs, ts, blocks, nb, cs);
      if (stt != SS_OK) return stt;
      ts.run_if = bs.fallback;
    }
    if (!bucket || !bs.serial_fallback) {
      const int64_t key_items = ((int64_t)T * B + kSortThreads - 1) / kSortThreads;
      int64_t grid = key_items > p.nblk ? key_items : p.nblk;
      if (grid > 4 * num_sms()) grid = 4 * num_sms();
      SS_TIMED("tiled_sort_kernel", cs);
      launch_dependent(tiled_sort_kernel, (unsigned)grid, kSortThreads, 0, cs, ts);
      SS_LAUNCH_OK();
    }
  }

  // (4) windowed segment reduction, (5) combine, (6) row-wise Adagrad
  if (do_apply) {
#define SS_RED(G_, NV_) \
  launch_reduce<G_, NV_>(p, ws, keys_sorted, T, N, D, B, grad, ld_grad, col0, tables, row_state, lr, eps, d_status, cs)
    SS_DISPATCH_GNV(D, SS_RED);
#undef SS_RED
    SS_LAUNCH_OK();
  }
  return SS_OK;
}

ss_status ss_embbag_bwd_adagrad(float* tables, float* row_state, int T, int64_t N, int D, const int32_t* indices,
                                const int32_t* offsets, int B, int64_t L, const float* grad, int64_t ld_grad,
                                int col0, float lr, float eps, void* workspace, size_t workspace_bytes,
                                int32_t* uniq_keys, int32_t* seg_off, int32_t* perm, int32_t* d_num_unique,
                                int32_t* d_status, ss_stream stream) {
  return bwd_impl(true, true, tables, row_state, T, N, D, indices, offsets, B, L, grad, ld_grad, col0, lr, eps, workspace,
                  workspace_bytes, uniq_keys, seg_off, perm, d_num_unique, d_status, stream);
}

ss_status ss_embbag_bwd_sort(int T, int64_t N, int D, const int32_t* indices, const int32_t* offsets, int B, int64_t L,
                             void* workspace, size_t workspace_bytes, int32_t* uniq_keys, int32_t* seg_off,
                             int32_t* perm, int32_t* d_num_unique, int32_t* d_status, ss_stream stream) {
  return bwd_impl(true, false, nullptr, nullptr, T, N, D, indices, offsets, B, L, nullptr, 0, 0, 0.f, 0.f, workspace,
                  workspace_bytes, uniq_keys, seg_off, perm, d_num_unique, d_status, stream);
}

ss_status ss_embbag_bwd_apply(float* tables, float* row_state, int T, int64_t N, int D, int B, int64_t L,
                              const float* grad, int64_t ld_grad, int col0, float lr, float eps, void* workspace,
                              size_t workspace_bytes, int32_t* d_status, ss_stream stream) {
  return bwd_impl(false, true, tables, row_state, T, N, D, nullptr, nullptr, B, L, grad, ld_grad, col0, lr, eps, workspace,
                  workspace_bytes, nullptr, nullptr, nullptr, nullptr, d_status, stream);
}

// ------------------------------------------------------------------------------------------------
// Sort / unique without any caller-provided or allocated scratch.
//
// Some callers of this library may not allocate device memory at the moment they need the sort: a
// host process whose memory pool has already handed every byte of the GPU to other owners, a plug-in
// that runs inside somebody else's serving loop where cudaMalloc's implicit device-wide
// synchronisation would stall unrelated streams, or start-up code that runs before the application's
// allocator exists.  For them the scratch of the sort lives in the array below, which is part of the
// library image: every GPU that loads the library holds these bytes until the process exits.
// ------------------------------------------------------------------------------------------------
constexpr int64_t kNoAllocMaxL = 65536;                       // most lookups one call may sort
constexpr size_t kNoAllocScratchBytes = 2162688;              // 2112 KiB, enough for kNoAllocMaxL lookups
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

// Device address of the array for the current device.  The array's name is only a handle on the
// host: the address a kernel can use comes from cudaGetSymbolAddress, asked once per device.
static ss_status noalloc_scratch_ptr(unsigned char** out) {
  static unsigned char* ptr[64];
  int dev = 0;
  SS_CUDA(ss::current_device(&dev));
  if (dev < 0 || dev >= 64) return SS_ERR_SHAPE;
  if (!ptr[dev]) {
    void* p = nullptr;
    SS_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    ptr[dev] = reinterpret_cast<unsigned char*>(p);
  }
  *out = ptr[dev];
  return SS_OK;
}

ss_status ss_embbag_bwd_sort_noalloc(int T, int64_t N, const int32_t* indices, const int32_t* offsets, int B,
                                     int64_t L, int32_t* uniq_keys, int32_t* seg_off, int32_t* perm,
                                     int32_t* d_num_unique, int32_t* d_status, ss_stream stream) {
  using namespace ss;
  if (!offsets || (!indices && L > 0) || !uniq_keys || !seg_off || !perm || !d_num_unique) return SS_ERR_NULL;
  if (T < 0 || B < 0 || N <= 0 || L < 0) return SS_ERR_SHAPE;
  if (L > kNoAllocMaxL) return SS_ERR_SHAPE;                   // beyond the built-in scratch: use ss_embbag_bwd_sort
  if ((uint64_t)T * (uint64_t)N >= (1ull << 31)) return SS_ERR_SHAPE;
  ss_status stt = check_arch();
  if (stt != SS_OK) return stt;
  unsigned char* ws = nullptr;
  stt = noalloc_scratch_ptr(&ws);
  if (stt != SS_OK) return stt;
  cudaStream_t cs = as_stream(stream);

  // digit plan of the radix sort (same rule as the workspace variant)
  const uint64_t maxkey = (uint64_t)T * (uint64_t)N;
  int bits = 1;
  while ((maxkey >> bits) != 0) ++bits;
  const int passes = (bits + 8) / 9;
  const int digit_bits = (bits + passes - 1) / passes;

  // carve the array; every piece is rewritten in full by each call before it is read, so nothing
  // depends on what an earlier call left behind
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t r = o; o += align256(bytes); return r; };
  const size_t l4 = (size_t)kNoAllocMaxL * 4;
  uint32_t* keys_a = reinterpret_cast<uint32_t*>(ws + take(l4));
  uint32_t* keys_b = reinterpret_cast<uint32_t*>(ws + take(l4));
  int32_t* pos_a = reinterpret_cast<int32_t*>(ws + take(l4));
  int32_t* pos_b = reinterpret_cast<int32_t*>(ws + take(l4));
  int32_t* bag_of = reinterpret_cast<int32_t*>(ws + take(l4));
  int32_t* uidx = reinterpret_cast<int32_t*>(ws + take(l4));
  int32_t* uniq = reinterpret_cast<int32_t*>(ws + take(l4));
  int32_t* seg = reinterpret_cast<int32_t*>(ws + take(l4 + 4));
  uint32_t* hist = reinterpret_cast<uint32_t*>(ws + take((size_t)(kNoAllocMaxL / kSortTile) * kMaxBins * 4));
  uint32_t* bintot = reinterpret_cast<uint32_t*>(ws + take((size_t)kMaxBins * 4));
  uint32_t* heads = reinterpret_cast<uint32_t*>(ws + take((size_t)(kNoAllocMaxL / kSortTile) * 4));
  int32_t* scalars = reinterpret_cast<int32_t*>(ws + take(256));
  if (o > kNoAllocScratchBytes) return SS_ERR_WORKSPACE;
  const uint32_t sentinel = (uint32_t)maxkey;

  TiledSort ts{};
  SortOut& out = ts.out;
  out.keys = (passes & 1) ? keys_b : keys_a; out.perm = (passes & 1) ? pos_b : pos_a;
  out.uidx = uidx; out.uniq = uniq; out.seg = seg;
  out.perm_out = perm; out.uniq_out = uniq_keys; out.seg_out = seg_off; out.d_num_unique = d_num_unique;
  out.scalars = scalars; out.d_status = d_status; out.L = L; out.sentinel = sentinel;
  if (L == 0 || (int64_t)T * B == 0) {
    launch_dependent(unique_finish_kernel, 1, 1, 0, cs, out);
    SS_LAUNCH_OK();
    return SS_OK;
  }
  ts.indices = indices; ts.offsets = offsets; ts.T = T; ts.B = B; ts.N = N;
  ts.keys_a = keys_a; ts.keys_b = keys_b; ts.pos_a = pos_a; ts.pos_b = pos_b; ts.bag_of = bag_of;
  ts.hist = hist; ts.bintot = bintot; ts.tile_heads = heads; ts.ctl = scalars + 8;
  ts.passes = passes; ts.digit_bits = digit_bits; ts.bins = 1 << digit_bits;
  stt = clear_words(ts.ctl, 3, cs);
  if (stt != SS_OK) return stt;
  const int64_t key_items = ((int64_t)T * B + kSortThreads - 1) / kSortThreads;
  const int64_t tiles = (L + kSortTile - 1) / kSortTile;
  int64_t grid = key_items > tiles ? key_items : tiles;
  if (grid > 4 * num_sms()) grid = 4 * num_sms();
  launch_dependent(tiled_sort_kernel, (unsigned)grid, kSortThreads, 0, cs, ts);
  SS_LAUNCH_OK();
  return SS_OK;
}

}  // extern "C"
