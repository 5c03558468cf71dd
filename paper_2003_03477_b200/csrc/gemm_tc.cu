// bf16 x bf16 -> fp32 GEMM on the 5th-generation tensor cores (tcgen05) of sm_100a, as a persistent kernel.
//
//   C[m, n] = sum_k A(m, k) * B(n, k)
//
// One launch (a "flow") holds one or several products.  Its CTAs (at most one per SM) stay resident and draw
// 128 x kBN output tiles from a counter in device memory, in the order the products are listed.  Inside a CTA
// three roles run concurrently on their own warps:
//   warp 0 (one lane)  draws tiles and streams 128 x 64 / 64 x kBN operand tiles into a ring of shared-memory
//                      stages with TMA (128-byte swizzle), running ahead into the next tile;
//   warp 1 (one lane)  issues tcgen05.mma (M = 128, N = 16..kBN, K = 16) into one of TWO accumulators in tensor
//                      memory and releases stages with tcgen05.commit;
//   warps 2-5          read a finished accumulator with tcgen05.ld (one row per thread, 64 columns at a time) and apply
//                      the epilogue (bias, ReLU, ReLU-gradient mask, bf16 / fp32 stores), while the MMA warp already
//                      fills the other accumulator.
// Set-up (barriers, tensor memory, descriptor prefetch) is paid once per CTA, not once per tile.
//
// A product may read what an earlier product of the same flow writes (a layer reading the previous layer's
// activations, a weight gradient reading the gradient tensor an input-gradient product produces).  Finished tiles
// count up a per-(product, row block) word in device memory; the TMA role of a dependent tile waits for the words
// it needs before it loads the operand (release / acquire at device scope, plus a proxy fence because the data is
// written through the generic proxy and read by TMA).  A tile only ever waits for tiles drawn before it, by CTAs
// that are running, so the wait ends whatever else occupies the device.
//
// Either operand may be K-major (k contiguous in memory: the forward pass reads activations [B, in]
// and weights [out, in] this way) or MN-major (m or n contiguous: the backward pass reads the same
// buffers transposed, dW = dY^T X and dX = dY W), so no transposed copy of any matrix is ever made.
// K-major tiles are one TMA box of 128 rows x 64 k; MN-major tiles are boxes of 64 k x 64 m, the
// canonical 128-byte-swizzle layouts of the shared-memory matrix descriptor in both cases.
//
// Every wait (mbarrier or dependency word) is bounded: when it runs out the kernel raises a device error flag,
// every role stops, nothing more is stored, outstanding copies are awaited, tensor memory is freed and the kernel
// returns; the host reads the flag (ss_device_error).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <string.h>
#include <memory>
#include <mutex>
#include <vector>
#include "gemm.cuh"
#include "profile.cuh"

// Hook for a time-stamp trace of the roles (a development harness defines it before including this file); no code here.
#ifndef SS_TC_TRACE
#define SS_TC_TRACE(id, tile)
#endif

namespace ss {

constexpr int kBM = 128;             // tile rows; the tile width kBN (64 or 256) and the k depth of a stage kBK (64 or 128)
                                     // are template parameters
constexpr int kAtomK = 64;           // k depth of a 128-byte-swizzle atom of a K-major operand
__host__ __device__ constexpr int stage_bytes(int bn, int bk) { return (kBM + bn) * bk * 2; }
// Epilogue warps: one per tensor-memory lane quadrant.  Eight (two per quadrant) make a flow that has the device to itself
// faster (the forward chain of the ordinary model 38 -> 32 us on all SMs) but take threads
// from the other streams' kernels: two replicas of the large model 913 -> 990 us a round.
constexpr int kEpiWarps = 4;
constexpr int kTcThreads = 64 + 32 * kEpiWarps;
constexpr int kQueue = 4;                                 // tiles a CTA may have drawn and not yet finished
// Stages of the ring.  The thread that fills them takes about 450 cycles for one, whatever its size: 64-wide tiles,
// whose MMAs are over sooner, take 128 k at a time (3 x 48 KiB); 256-wide tiles and CTA pairs take 64 (3 x 48, 5 x 32 KiB).
// One CTA per SM in every case.
constexpr int kStagesSmall = 3, kStagesWide = 3, kStagesPair = 5;
constexpr int kCtlBytes = 512;                            // barriers, tile queue, tensor-memory address, abort flag
// Per epilogue warp: two 4 KiB slabs (32 rows x 128 bytes, 128-byte swizzle) from which TMA stores pieces of the
// output (one is filled while the other is being read), and the bias values of its columns of the tile.
constexpr int kSlabBytes = 32 * 128;
constexpr int kChunk = 64;                                // columns an epilogue warp takes at a time
constexpr int kBiasFloats = 256;                          // the widest tile
constexpr int kEpiWarpBytes = 2 * kSlabBytes;
constexpr size_t tc_smem_bytes(int stages, int load_n, int bk, size_t meta_bytes) {
  return (size_t)stages * stage_bytes(load_n, bk) + kEpiWarps * (kEpiWarpBytes + kBiasFloats * 4) + 1024 /*alignment slack*/ +
         kCtlBytes + meta_bytes;
}
constexpr long long kWaitCycles = 400ll * 1000 * 1000;    // ~0.2 s: far beyond any legitimate wait

__device__ int g_device_error = 0;   // 0 ok; otherwise the code of the first wait that ran out

// How the operand part of a stage is fetched:
//   FORM_K_ATOMS   K-major, K a multiple of 64: one 3-d box, 64 k x up to 256 rows x (kBK / 64)
//   FORM_K_BOXES   K-major, any K: one box of 64 k x up to 256 rows per 64 k
//   FORM_MN_ATOMS  MN-major, width a multiple of 64: one 3-d box, 64 columns x kBK k x atoms
//   FORM_MN_BOXES  MN-major, any width: one box of 64 columns x kBK k per atom
enum { FORM_K_ATOMS = 0, FORM_K_BOXES = 1, FORM_MN_ATOMS = 2, FORM_MN_BOXES = 3 };

struct TcParams {
  int M, N, K;
  int a_mn, b_mn;          // 1 = MN-major operand
  int a_form, b_form;      // how a stage of it is fetched
  int a_box_bytes, b_box_bytes;   // what one TMA load of it brings
  int a_k_atom, b_k_atom;  // K-major: bytes from one 64-k atom of a stage to the next
  int k_splits;            // the K range is cut into this many slices; slice z writes out_lo + z*split_stride
  int64_t split_stride;    // in floats
  int dep, dep_mode, dep_k, dep_need;   // see TcJob; dep_need = arrivals that complete a row block of `dep`
  int dep_need_all;        // arrivals that complete all of `dep`
  int signals;             // 1: another product of the flow waits for this one
  int tma_out, pad;        // tma_out = 1: outputs leave through shared memory and TMA stores
  Epilogue ep;
};

// One product of a flow: its tensor maps, its parameters and its share of the tile sequence.
// Tile `tile_begin + (z * grid_y + y) * grid_x + x` is (row block y, column block x) of K slice z.
// Everything but the tensor maps is copied into shared memory when a CTA starts and from there into registers when a
// role takes up a tile: the parameter block is indexed by a run-time product number, and reading it field by field
// inside the loops would put a constant-bank load in front of every use.
struct TcMeta {
  TcParams p;
  int tile_begin, grid_x, grid_y, pad;
};
struct TcProblem {
  CUtensorMap map_a, map_b;
  CUtensorMap map_lo;                     // out_lo (3-d for float: column, row, K slice); used when tma_out
  TcMeta meta;
};
template <int NP>
struct TcFlow {
  TcProblem prob[NP];
  int n, total_tiles;
  int* ctrl;               // [0] tile counter, [1] exit ticket, [2 + j * rb_stride + rb] completions; nullptr: round-robin
  int rb_stride;
  int* err;
};

// ---------------------------------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// One thread of the (converged) warp.  Unlike a test of the lane number this tells the compiler that a single thread is
// active behind it, so operands of TMA and MMA instructions move to uniform registers directly.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok));
  return ok != 0;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One try: the hardware may park the thread for up to the given time while the phase is incomplete (it is woken
// when the phase completes), so a waiting role leaves the issue slots to the other warps of the SM.
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(20000u) : "memory");
  return ok;
}
// The same for a barrier that threads of the other CTA of a cluster arrive on: what they wrote before is visible.
__device__ __forceinline__ uint32_t mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(20000u) : "memory");
  return ok;
}
// Bounded wait.  Returns false when the limit is reached (records `code`) or another role has given up.
template <bool kCluster = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* aborted, int* err, int code) {
  auto try_wait = [&] { return kCluster ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity); };
  if (try_wait()) return true;
  const long long t0 = clock64();
  while (!try_wait()) {
    if (*aborted) return false;
    if (clock64() - t0 > kWaitCycles) {
      *aborted = 1;
      atomicCAS(err, 0, code);
      return false;
    }
  }
  return true;
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Counts one completion; everything this thread did (or was ordered after) is visible to whoever acquires the count.
__device__ __forceinline__ void red_release(int* p) {
  asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p) : "memory");
}
// Bounded wait for a completion word of the flow to reach `need`.
__device__ __forceinline__ bool wait_count(const int* word, int need, volatile int* aborted, int* err) {
  if (ld_acquire(word) < need) {
    const long long t0 = clock64();
    while (ld_acquire(word) < need) {
      if (*aborted) return false;
      if (clock64() - t0 > kWaitCycles) {
        *aborted = 1;
        atomicCAS(err, 0, 4);
        return false;
      }
      __nanosleep(32);
    }
  }
  // what the other CTAs stored through the generic proxy is read by TMA (async proxy) from here on
  asm volatile("fence.proxy.async;" ::: "memory");
  return true;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int x, int y, int z) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// ---- CTA pairs (cta_group::2): two CTAs of a cluster share one 256-row MMA
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t smem_addr, uint32_t rank) {   // the same offset in another CTA of the cluster
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t cluster_addr, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
// TMA load of one CTA of a pair; the bytes are counted on a barrier that may live in the other CTA (no multicast:
// each CTA fetches its own tiles)
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar_cluster, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar_cluster, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {          // arrives on the barrier at this offset in both CTAs
  const uint16_t mask = 3;
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask) : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle, descriptor version 1 (sm_100).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;
  d |= 2ull << 61;
  return d;
}

// Bits of 32 consecutive columns: perfect shuffle between "bit j = column j" and "bit i = column 2i, bit 16 + i =
// column 2i + 1" (the order in which packed bf16 pairs yield them).
__device__ __forceinline__ uint32_t swap_bits(uint32_t x, uint32_t mask, int by) {
  const uint32_t t = (x ^ (x >> by)) & mask;
  return x ^ t ^ (t << by);
}
__device__ __forceinline__ uint32_t pairs_to_columns(uint32_t x) {
  x = swap_bits(x, 0x0000FF00u, 8);
  x = swap_bits(x, 0x00F000F0u, 4);
  x = swap_bits(x, 0x0C0C0C0Cu, 2);
  return swap_bits(x, 0x22222222u, 1);
}
__device__ __forceinline__ uint32_t columns_to_pairs(uint32_t x) {
  x = swap_bits(x, 0x22222222u, 1);
  x = swap_bits(x, 0x0C0C0C0Cu, 2);
  x = swap_bits(x, 0x00F000F0u, 4);
  return swap_bits(x, 0x0000FF00u, 8);
}
// 0xFFFF in each half of a packed bf16 pair that is positive
__device__ __forceinline__ uint32_t positive_halves(uint32_t packed) {
  const uint32_t zero = 0u;
  return __hgt2_mask(*reinterpret_cast<const __nv_bfloat162*>(&packed), *reinterpret_cast<const __nv_bfloat162*>(&zero));
}
__device__ __forceinline__ uint32_t relu_pair(uint32_t packed) {
  const uint32_t zero = 0u;
  const __nv_bfloat162 h = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&packed), *reinterpret_cast<const __nv_bfloat162*>(&zero));
  return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// Columns of the MMA of a tile with `left` columns of the product at or beyond its first: rounded up to the
// instruction's granule (a pair: whole 64-column atoms for each half).
__device__ __forceinline__ int tile_columns(int left, int bn, bool pair) {
  const int granule = pair ? 128 : 16;
  return left >= bn ? bn : (left + granule - 1) & ~(granule - 1);
}

// A tile of the flow: which product, which block, which K range.
struct TileAt {
  int j, x, y, z, kb_begin, nk;     // kb_begin, nk in atoms of 64 k
};
// Atoms [0, nd) of a tile's range wait for the producing product and are taken last, the others do not; a stage takes up
// to kBK / 64 atoms of one of the two parts.  So the order of the sums, and with it every bit of the result, is the same for
// every tile shape.
__device__ __forceinline__ int atoms_that_wait(const TcParams& p, int nk) {
  if (p.dep < 0 || p.dep_mode != 1) return 0;
  const int nd = p.k_splits == 1 ? (p.dep_k + kAtomK - 1) / kAtomK : 0;
  return nd > 0 && nd < nk ? nd : nk;
}
__device__ __forceinline__ TileAt locate_tile(const TcMeta* meta, int n, int t) {
  int j = 0;
  for (int end = n; end - j > 1;) {                        // the last product that begins at or before tile t
    const int mid = (j + end) >> 1;
    if (t >= meta[mid].tile_begin) j = mid; else end = mid;
  }
  const int gx = meta[j].grid_x, gy = meta[j].grid_y, K = meta[j].p.K, ks = meta[j].p.k_splits;
  const int local = t - meta[j].tile_begin;
  TileAt a;
  a.j = j;
  a.x = local % gx;
  a.y = (local / gx) % gy;
  a.z = local / (gx * gy);
  const int atoms = (K + kAtomK - 1) / kAtomK;
  a.kb_begin = (int)((int64_t)atoms * a.z / ks);
  a.nk = (int)((int64_t)atoms * (a.z + 1) / ks) - a.kb_begin;   // >= 1: k_splits <= atoms
  return a;
}

// ---------------------------------------------------------------------------------------- kernel
// kPair: the CTAs come in pairs (clusters of two).  A pair computes a 256 x kBN tile with one tcgen05.mma.cta_group::2
// per k step, issued by the pair's first CTA: each CTA holds its 128 rows of A, HALF of the B tile (the tensor cores of
// both SMs read both halves) and the accumulator of its own 128 rows.  Per flop a CTA loads and reads a third less
// shared memory than with 128 x 256 tiles of its own, which is what bounds those.  The first CTA's producer draws the
// pair's tiles and hands each to the second CTA; every CTA loads, waits for and reports its own 128-row blocks, so the
// dependencies between products are the same in both forms.
// 112 registers a thread (the epilogue would take 144; capped, it recomputes a few addresses and spills nothing): a
// CTA of this kernel sits beside the blocks of other streams' kernels, which get the registers it leaves.
template <int kStages, int kBN, int kBK, int NP, bool kPair>
__global__ void __maxnreg__(112)
gemm_tc_kernel(const __grid_constant__ TcFlow<NP> flow) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int kLoadN = kPair ? kBN / 2 : kBN;            // columns of B this CTA loads
  constexpr int kTileM = kPair ? 2 * kBM : kBM;            // rows of a tile
  constexpr int kStageBytes = stage_bytes(kLoadN, kBK), kABytes = kBM * kBK * 2;
  constexpr int kKAtoms = kBK / kAtomK;                    // 64-k atoms of a stage
  constexpr int kTmemCols = 2 * kBN;                       // two accumulators of kBN fp32 columns
  const uint32_t rank = kPair ? cluster_rank() : 0u;       // 0: the CTA that issues the pair's MMAs
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;                 // 1024-byte aligned swizzle atoms
  uint8_t* gen = smem_raw + (tiles - raw);
  const uint32_t epi0 = tiles + kStages * kStageBytes;            // 1024-byte aligned: stages are multiples of 1 KiB
  uint8_t* epi_gen = gen + (size_t)kStages * kStageBytes;
  constexpr int kEpiBytes = kEpiWarps * (kEpiWarpBytes + kBiasFloats * 4);
  uint8_t* ctl = epi_gen + kEpiBytes;
  const uint32_t bar0 = epi0 + kEpiBytes;
  // barriers: [0,S) full, [S,2S) empty, then accumulator full[2], empty[2], queue full[kQueue], empty[kQueue]
  constexpr int kNumBars = 2 * kStages + 4 + 2 * kQueue;
  int* tile_q = reinterpret_cast<int*>(ctl + 8 * kNumBars);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tile_q + kQueue);
  volatile int* aborted = reinterpret_cast<volatile int*>(tmem_slot + 1);
  TcMeta* meta = reinterpret_cast<TcMeta*>(ctl + kCtlBytes);
  static_assert(8 * kNumBars + 4 * kQueue + 8 <= kCtlBytes, "control region");
  static_assert(sizeof(TcMeta) % 4 == 0, "copied word by word");
  const int n_prob = flow.n;
  for (int j = 0; j < n_prob; ++j) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(&flow.prob[j].meta);
    uint32_t* dst = reinterpret_cast<uint32_t*>(meta + j);
    for (int i = threadIdx.x; i < (int)(sizeof(TcMeta) / 4); i += kTcThreads) dst[i] = src[i];
  }
  auto full = [&](int s) { return bar0 + 8u * s; };
  auto empty = [&](int s) { return bar0 + 8u * (kStages + s); };
  auto acc_full = [&](int b) { return bar0 + 8u * (2 * kStages + b); };
  auto acc_empty = [&](int b) { return bar0 + 8u * (2 * kStages + 2 + b); };
  auto q_full = [&](int s) { return bar0 + 8u * (2 * kStages + 4 + s); };
  auto q_empty = [&](int s) { return bar0 + 8u * (2 * kStages + 4 + kQueue + s); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int j = 0; j < flow.n; ++j) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&flow.prob[j].map_a)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&flow.prob[j].map_b)) : "memory");
    }
    for (int s = 0; s < kStages; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), kPair ? 2 * kEpiWarps : kEpiWarps); }
    for (int s = 0; s < kQueue; ++s) { mbar_init(q_full(s), 1); mbar_init(q_empty(s), (kPair ? 2 : 1) * (1 + kEpiWarps)); }
    *aborted = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    if (kPair) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (kPair) cluster_sync_all();                           // the other CTA's barriers exist before anything arrives on them
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  wait_for_previous_kernel();                              // set-up above touches nothing in device memory
  int* const done0 = flow.ctrl ? flow.ctrl + 2 : nullptr;
  if (threadIdx.x == 0) SS_TC_TRACE(1, -1);

  if (warp == 0) {
    // ------------------------------------------------------------------ tile scheduler + TMA producer
    // One thread feeds the tensor cores: a k block costs it as many cycles as the instructions of the loop below, one
    // after the other, so the loop holds what changes per k block and nothing else (590 cycles a k block before, with
    // every operand behind a lane test, every address recomputed and up to six boxes; the MMAs of a 128 x 256 x 64 block
    // take 512, of a narrower one less).
    if (elect_one()) {
      uint32_t s = 0, parity = 1;                          // stage to fill next, and the phase of its `empty` barrier to wait for
      uint32_t filled = 0;                                 // stages filled so far (over all tiles)
      const bool draws = !(kPair && rank != 0);            // a pair's tiles are drawn by its first CTA
      // The ticket of the next tile is drawn with the last k block of the current one: its round trip to L2 is over by the
      // time the ring has a free stage again, and not earlier, or a CTA would hold two tiles while another has none (with
      // about as many tiles as CTAs, as the layers of a small batch have, that doubled the time of a layer).  Tickets are
      // drawn in order by running CTAs and worked off in order, which is all the waiting needs.
      const int unit = kPair ? (int)(blockIdx.x >> 1) : (int)blockIdx.x, n_units = kPair ? (int)(gridDim.x >> 1) : (int)gridDim.x;
      int t_next = !draws ? 0 : (flow.ctrl ? atomicAdd(flow.ctrl, 1) : unit);
      for (uint32_t qi = 0;; ++qi) {
        const int qs = qi % kQueue;
        int t;
        if (!draws) {                                      // the tile the first CTA drew
          if (!mbar_wait<true>(q_full(qs), (qi / kQueue) & 1, aborted, flow.err, 5)) break;
          t = tile_q[qs];
          mbar_arrive_cluster(map_to_cta(q_empty(qs), 0));
        } else {
          if (!mbar_wait<kPair>(q_empty(qs), ((qi / kQueue) & 1) ^ 1u, aborted, flow.err, 5)) break;
          t = t_next;
          if (t >= flow.total_tiles) t = -1;
          tile_q[qs] = t;
          if (kPair) {
            st_cluster(map_to_cta(smem_u32(tile_q + qs), 1), t);
            mbar_arrive_cluster(map_to_cta(q_full(qs), 1));
          }
          mbar_arrive(q_full(qs));
        }
        if (t < 0) break;
        SS_TC_TRACE(2, t);
        const TileAt a = locate_tile(meta, n_prob, t);
        const TcParams& p = meta[a.j].p;
        const CUtensorMap* const map_a = &flow.prob[a.j].map_a;
        const CUtensorMap* const map_b = &flow.prob[a.j].map_b;
        const int n_mma = tile_columns(p.N - a.x * kBN, kBN, kPair);
        const int n_load = kPair ? n_mma / 2 : n_mma;      // columns of B this CTA fetches
        const int m0 = a.y * kTileM + (int)rank * kBM, n0 = a.x * kBN + (int)rank * n_load;
        const int M = p.M, a_form = p.a_form, b_form = p.b_form;
        // Boxes of a stage: one per operand where the layout allows it.  Rows of A at or beyond M are not fetched when a
        // whole box lies there (their accumulators are not stored).
        auto boxes_of = [](int form, int first, int end, int most) {
          if (form != FORM_MN_BOXES) return first < end ? (form == FORM_K_BOXES ? kKAtoms : 1) : 0;
          const int left = (end - first + 63) >> 6;
          return left < 0 ? 0 : (left > most ? most : left);
        };
        const int na = boxes_of(a_form, m0, M, 2), nb = boxes_of(b_form, n0, n0 + n_load, kLoadN / 64);
        const uint32_t a_bytes = p.a_box_bytes, b_bytes = p.b_box_bytes;
        uint32_t tile_bytes = na * a_bytes + nb * b_bytes;
        if (kPair) tile_bytes += boxes_of(a_form, m0 + kBM, M, 2) * a_bytes + nb * b_bytes;   // of both CTAs; only the first counts
        const int* dep_words = p.dep >= 0 ? done0 + p.dep * flow.rb_stride : nullptr;
        const int dep_mode = p.dep >= 0 ? p.dep_mode : 0;
        // dep_mode 2 (the producer's row blocks are the k blocks): nothing from k_ready on may be read yet.
        const int nd = atoms_that_wait(p, a.nk);
        int k_ready = 0x7fffffff;
        if (dep_mode == 2) {
          if (ld_acquire(dep_words + flow.rb_stride - 1) >= p.dep_need_all) asm volatile("fence.proxy.async;" ::: "memory");
          else k_ready = a.kb_begin * kAtomK / kBM * kBM;
        }
        bool failed = false;
        int left = (a.nk - nd + kKAtoms - 1) / kKAtoms + (nd + kKAtoms - 1) / kKAtoms;
        for (int part = 0; part < 2 && !failed; ++part) {
          const int kb1 = part == 0 ? a.nk : nd;
          if (part == 1 && nd > 0 && na > 0 && !wait_count(dep_words + m0 / kBM, p.dep_need, aborted, flow.err)) { failed = true; break; }
          int k0 = (a.kb_begin + (part == 0 ? nd : 0)) * kAtomK;
          for (int kb = part == 0 ? nd : 0; kb < kb1; kb += kKAtoms, k0 += kBK) {
            if (--left == 0 && draws) t_next = flow.ctrl ? atomicAdd(flow.ctrl, 1) : (int)(unit + (qi + 1) * n_units);
            if (k0 + kBK > k_ready) {                      // (what a stage fetches beyond its part is not read)
              const int last = k0 + (kb + kKAtoms <= kb1 ? kBK : kAtomK) - 1;
              for (; k_ready <= last; k_ready += kBM)
                if (!wait_count(dep_words + k_ready / kBM, p.dep_need, aborted, flow.err)) { failed = true; break; }
              if (failed) break;
            }
            if (!mbar_wait(empty(s), parity, aborted, flow.err, 1)) { failed = true; break; }
            const uint32_t sa = tiles + s * kStageBytes, sb = sa + kABytes;
            // of a pair, both CTAs' tiles are counted on the first CTA's barrier, which its MMA thread waits on
            const uint32_t bar = kPair ? map_to_cta(full(s), 0) : full(s);
            if (draws) mbar_expect_tx(full(s), tile_bytes);
            auto load2 = [&](uint32_t dst, const CUtensorMap* map, int x, int y) {
              if (kPair) tma_load_2d_pair(dst, map, bar, x, y); else tma_load_2d(dst, map, bar, x, y);
            };
            auto load3 = [&](uint32_t dst, const CUtensorMap* map, int y, int z) {
              if (kPair) tma_load_3d_pair(dst, map, bar, 0, y, z); else tma_load_3d(dst, map, bar, 0, y, z);
            };
            auto load = [&](uint32_t dst, const CUtensorMap* map, int form, uint32_t bytes, int mn, int h) {
              if (form == FORM_K_ATOMS) load3(dst, map, mn, k0 >> 6);
              else if (form == FORM_MN_ATOMS) load3(dst, map, k0, mn >> 6);
              else if (form == FORM_K_BOXES) load2(dst + h * bytes, map, k0 + kAtomK * h, mn);
              else load2(dst + h * bytes, map, mn + 64 * h, k0);
            };
            if (na > 0) load(sa, map_a, a_form, a_bytes, m0, 0);
            if (na > 1) load(sa, map_a, a_form, a_bytes, m0, 1);
            load(sb, map_b, b_form, b_bytes, n0, 0);
            for (int h = 1; h < nb; ++h) load(sb, map_b, b_form, b_bytes, n0, h);
            ++filled;
            if (++s == kStages) { s = 0; parity ^= 1u; }
          }
        }
        if (failed) break;
        SS_TC_TRACE(4, t);
      }
      if (*aborted) {
        // the copies still in flight land in this CTA's shared memory: wait for them (bounded) before leaving
        const uint32_t first = filled > (uint32_t)kStages ? filled - kStages : 0u;
        for (uint32_t i = first; i < filled; ++i) {
          const long long t0 = clock64();
          while (!mbar_try_wait(full(i % kStages), (i / kStages) & 1) && clock64() - t0 < 4000000ll) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (rank == 0 && elect_one()) {                        // a pair's MMAs are issued by its first CTA
      uint32_t s = 0, parity = 0, at = 0;                  // stage to consume next and its phase, tiles accumulated
      for (uint32_t qi = 0;; ++qi) {
        const int qs = qi % kQueue;
        if (!mbar_wait(q_full(qs), (qi / kQueue) & 1, aborted, flow.err, 6)) break;
        const int t = tile_q[qs];
        mbar_arrive(q_empty(qs));
        if (t < 0) break;
        const TileAt a = locate_tile(meta, n_prob, t);
        const int a_mn = meta[a.j].p.a_mn, b_mn = meta[a.j].p.b_mn;
        const int n_mma = tile_columns(meta[a.j].p.N - a.x * kBN, kBN, kPair);
        // instruction descriptor: D = f32, A = B = bf16, majors, N >> 3, M >> 4
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
                               ((uint32_t)(n_mma >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
        // K-major: 8-row groups 1024 B apart (SBO), K step of 16 elements = 32 B inside the swizzle span, atoms of 64 k
        // a_k_atom apart.  MN-major: 64-wide m atoms kBK * 128 B apart (LBO), 8-k groups 1024 B apart (SBO), K step = 2048 B.
        // The descriptor of a stage and step is that of the ring's start plus its offset in 16-byte units (no carry: shared
        // memory addresses take 14 bits there).
        const uint64_t ad0 = smem_desc(tiles, a_mn ? kBK * 128u : 16u, 1024u), bd0 = smem_desc(tiles + kABytes, b_mn ? kBK * 128u : 16u, 1024u);
        const uint32_t a_step = (a_mn ? 2048u : 32u) >> 4, b_step = (b_mn ? 2048u : 32u) >> 4;
        const uint32_t a_atom = (a_mn ? 8192u : (uint32_t)meta[a.j].p.a_k_atom) >> 4, b_atom = (b_mn ? 8192u : (uint32_t)meta[a.j].p.b_k_atom) >> 4;
        const int buf = at & 1;
        if (!mbar_wait<kPair>(acc_empty(buf), ((at >> 1) & 1) ^ 1u, aborted, flow.err, 7)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem + (uint32_t)(buf * kBN);
        bool failed = false;
        const int nd = atoms_that_wait(meta[a.j].p, a.nk);
        uint32_t accumulate = 0;
        for (int part = 0; part < 2 && !failed; ++part) {
          const int kb1 = part == 0 ? a.nk : nd;
          for (int kb = part == 0 ? nd : 0; kb < kb1; kb += kKAtoms) {
            if (!mbar_wait(full(s), parity, aborted, flow.err, 2)) { failed = true; break; }
            if (!accumulate) SS_TC_TRACE(5, t);
            tc_fence_after();
            const uint32_t off = s * (uint32_t)(kStageBytes >> 4);
#pragma unroll
            for (int h = 0; h < kKAtoms; ++h) {
              if (h > 0 && kb + h >= kb1) break;
#pragma unroll
              for (int k = 0; k < kAtomK / 16; ++k) {
                const uint64_t ad = ad0 + (off + h * a_atom + k * a_step), bd = bd0 + (off + h * b_atom + k * b_step);
                if (kPair) tc_mma_pair(d_tmem, ad, bd, idesc, accumulate);
                else tc_mma(d_tmem, ad, bd, idesc, accumulate);
                accumulate = 1;
              }
            }
            if (kPair) tc_commit_pair(empty(s));   // frees the stage in both CTAs when these MMAs have read it
            else tc_commit(empty(s));
            if (++s == kStages) { s = 0; parity ^= 1u; }
          }
        }
        if (failed) break;
        if (kPair) tc_commit_pair(acc_full(buf));   // accumulator complete, in both CTAs
        else tc_commit(acc_full(buf));
        SS_TC_TRACE(6, t);
        ++at;
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue warps 2..5
    const int q = warp & 3;               // tensor-memory lane quadrant this warp may read
    uint8_t* const slab_gen = epi_gen + q * kEpiWarpBytes;
    const uint32_t slab_out = epi0 + q * kEpiWarpBytes;
    float* const s_bias = reinterpret_cast<float*>(epi_gen + kEpiWarps * kEpiWarpBytes) + q * kBiasFloats;
    constexpr int kChunks = kBN / kChunk;
    uint32_t n_stores = 0;                // slabs handed to TMA so far (they alternate)
    uint32_t at = 0;
    for (uint32_t qi = 0;; ++qi) {
      const int qs = qi % kQueue;
      if (!mbar_wait<kPair>(q_full(qs), (qi / kQueue) & 1, aborted, flow.err, 8)) break;
      const int t = tile_q[qs];
      __syncwarp();
      if (lane == 0) {
        if (kPair) mbar_arrive_cluster(map_to_cta(q_empty(qs), 0));
        else mbar_arrive(q_empty(qs));
      }
      if (t < 0) break;
      const TileAt a = locate_tile(meta, n_prob, t);
      const Epilogue ep = meta[a.j].p.ep;                  // by value: registers
      const int M = meta[a.j].p.M, N = meta[a.j].p.N;
      const int m0 = a.y * kTileM + (int)rank * kBM, n0 = a.x * kBN;
      const int buf = at & 1;
      const bool tma_out = meta[a.j].p.tma_out != 0;
      const TcProblem& pr = flow.prob[a.j];
      // Everything the epilogue needs from memory is requested as soon as the tile is known, so that it arrives while
      // the tensor cores still work on the tile: the bias values of the warp's columns (every thread needs all of them:
      // 8 bytes per lane and chunk into the warp's shared memory) and the thread's words of the ReLU-gradient mask.
      const int64_t mrow = (int64_t)m0 + 32 * q + lane;
      const bool use_bits = ep.mask_bits != nullptr;
      uint2 mq[kChunks];
#pragma unroll
      for (int i = 0; i < kChunks; ++i) {
        const int nb = n0 + kChunk * i;
        if (ep.bias) {
          float2 bv = make_float2(0.f, 0.f);
          if (nb + 2 * lane < N) bv = __ldg(reinterpret_cast<const float2*>(ep.bias + nb + 2 * lane));   // N is a multiple of 8
          *reinterpret_cast<float2*>(s_bias + kChunk * i + 2 * lane) = bv;
        }
        mq[i] = make_uint2(~0u, ~0u);
        if (use_bits && mrow < M && nb < ep.mask_cols)
          mq[i] = __ldg(reinterpret_cast<const uint2*>(ep.mask_bits + mrow * ep.ld_mask_bits + (nb >> 5)));
      }
      __syncwarp();                                        // the bias values are in shared memory
      if (!mbar_wait(acc_full(buf), (at >> 1) & 1, aborted, flow.err, 3)) break;
      if (threadIdx.x == 64) SS_TC_TRACE(7, t);
      tc_fence_after();
      const int sw = lane & 7;
      const uint32_t row_off = (uint32_t)lane * 128u;
#pragma unroll 1
      for (int i = 0; i < kChunks; ++i) {
        const int nb = n0 + kChunk * i;
        if (nb >= N || m0 + 32 * q >= M) break;            // no column, or none of the warp's rows, is inside the matrix
        // the thread's row of the chunk: 64 accumulator columns, both loads in flight together
        uint32_t r[2][32];
        const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * kBN + kChunk * i);
        tc_ld32(taddr, r[0]);
        tc_ld32(taddr + 32, r[1]);
        tc_ld_wait();
        uint2 mw = mq[0];
#pragma unroll
        for (int k = 1; k < kChunks; ++k)
          if (i == k) mw = mq[k];
        if (tma_out && ep.lo_bf16) {
          // bias, ReLU and mask in registers, the packed row into the warp's slab in the 128-byte-swizzle layout; one
          // lane hands the slab to TMA, which stores whole rows of it and clips what lies beyond the matrix
          uint8_t* const slab = slab_gen + (n_stores & 1) * kSlabBytes;
          if (lane == 0) tma_store_wait_read1();           // this slab's previous contents have been read (the other may be in flight)
          __syncwarp();
          uint32_t bits[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t o[16];
            if (ep.bias) {
#pragma unroll
              for (int j = 0; j < 32; j += 4) {
                const float4 bv = *reinterpret_cast<const float4*>(s_bias + kChunk * i + 32 * h + j);   // the same address in every lane
                o[j / 2] = pack2(__uint_as_float(r[h][j]) + bv.x, __uint_as_float(r[h][j + 1]) + bv.y);
                o[j / 2 + 1] = pack2(__uint_as_float(r[h][j + 2]) + bv.z, __uint_as_float(r[h][j + 3]) + bv.w);
              }
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j) o[j] = pack2(__uint_as_float(r[h][2 * j]), __uint_as_float(r[h][2 * j + 1]));
            }
            if (ep.relu) {                                 // rounding is monotonic: the same values as ReLU before it
#pragma unroll
              for (int j = 0; j < 16; ++j) o[j] = relu_pair(o[j]);
            }
            if (use_bits) {
              const uint32_t w = columns_to_pairs(h ? mw.y : mw.x);
#pragma unroll
              for (int j = 0; j < 16; ++j) o[j] &= ((w >> j) & 0x00010001u) * 0xFFFFu;
            }
            if (ep.bits_out) {
              uint32_t b = 0;
#pragma unroll
              for (int j = 0; j < 16; ++j) b |= positive_halves(o[j]) & (0x00010001u << j);
              bits[h] = pairs_to_columns(b);
            }
#pragma unroll
            for (int g = 0; g < 4; ++g)
              *reinterpret_cast<uint4*>(slab + row_off + ((uint32_t)((g + 4 * h) ^ sw) << 4)) =
                  make_uint4(o[4 * g], o[4 * g + 1], o[4 * g + 2], o[4 * g + 3]);
          }
          if (ep.bits_out && mrow < M && !*aborted)
            *reinterpret_cast<uint2*>(ep.bits_out + mrow * ep.ld_bits_out + (nb >> 5)) = make_uint2(bits[0], bits[1]);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0 && !*aborted) {
            tma_store_2d(&pr.map_lo, slab_out + (n_stores & 1) * kSlabBytes, nb, m0 + 32 * q);
            tma_store_commit();
          }
          ++n_stores;
        } else if (tma_out) {
          // float output: 32 columns per slab
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (nb + 32 * h >= N) break;
            uint8_t* const slab = slab_gen + (n_stores & 1) * kSlabBytes;
            if (lane == 0) tma_store_wait_read1();
            __syncwarp();
#pragma unroll
            for (int g = 0; g < 8; ++g)
              *reinterpret_cast<uint4*>(slab + row_off + ((uint32_t)(g ^ sw) << 4)) =
                  make_uint4(r[h][4 * g], r[h][4 * g + 1], r[h][4 * g + 2], r[h][4 * g + 3]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0 && !*aborted) {
              tma_store_3d(&pr.map_lo, slab_out + (n_stores & 1) * kSlabBytes, nb + 32 * h, m0 + 32 * q, a.z);
              tma_store_commit();
            }
            ++n_stores;
          }
        } else if (mrow < M && !*aborted) {
          // a mask given by values (the producing layer ran on the SIMT kernel): plain loads and stores, bf16 output
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            const int n = nb + 8 * g;
            if (n >= N) break;
            uint32_t* const x = &r[g >> 2][8 * (g & 3)];
            uint32_t o[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) o[j] = pack2(__uint_as_float(x[2 * j]), __uint_as_float(x[2 * j + 1]));
            if (ep.mask && n < ep.mask_cols) {             // bf16 activation of the producing layer
              const uint4 mk = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(ep.mask) + mrow * ep.ld_mask + n);
              o[0] &= positive_halves(mk.x); o[1] &= positive_halves(mk.y);
              o[2] &= positive_halves(mk.z); o[3] &= positive_halves(mk.w);
            }
            *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(ep.out_lo) + mrow * ep.ld_lo + n) = make_uint4(o[0], o[1], o[2], o[3]);
          }
        }
      }
      if (!tma_out) asm volatile("fence.proxy.async;" ::: "memory");   // plain stores that a TMA load may read
      // the accumulator may be overwritten: this warp's reads of it are complete
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (kPair) mbar_arrive_cluster(map_to_cta(acc_empty(buf), 0));   // the MMA thread of the pair's first CTA waits for both
        else mbar_arrive(acc_empty(buf));
      }
      if (threadIdx.x == 64) SS_TC_TRACE(8, t);
      // completion words of the row block and of the product, for the products that read this output: what the warp's
      // TMA stores wrote is complete in memory, what its lanes stored is ordered by the warp barrier above
      if (done0 && meta[a.j].p.signals && lane == 0 && m0 < M) {
        if (tma_out) tma_store_wait_all();
        asm volatile("fence.proxy.async;" ::: "memory");
        red_release(done0 + a.j * flow.rb_stride + m0 / kBM);
        red_release(done0 + a.j * flow.rb_stride + flow.rb_stride - 1);   // after the row block's own word
      }
      ++at;
    }
    if (lane == 0) tma_store_wait_all();                   // the slabs are read before the CTA gives up its shared memory
  }

  tc_fence_before();
  __syncthreads();
  if (kPair) cluster_sync_all();                           // neither CTA leaves while the other may still signal it
  if (warp == 1) {
    tc_fence_after();
    if (kPair) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
  // the last CTA to leave clears the control words for the next launch (every other CTA is past its last access)
  if (flow.ctrl && threadIdx.x == 0 && !*aborted) {
    __threadfence();
    if (atomicAdd(flow.ctrl + 1, 1) == (int)gridDim.x - 1) {
      const int words = 2 + flow.n * flow.rb_stride;
      for (int i = 0; i < words; ++i) flow.ctrl[i] = 0;
      __threadfence();
    }
  }
}

// ---------------------------------------------------------------------------------------- host side
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// Matrix with `inner` contiguous elements per row, `outer` rows, row pitch ld elements (and `planes` such matrices
// plane_stride elements apart when rank is 3); 128-byte swizzle, so box_inner * element size is at most 128 bytes.
static bool make_map_any(CUtensorMap* map, CUtensorMapDataType dt, int esize, const void* base, int64_t inner, int64_t outer,
                         int64_t ld, int box_inner, int box_outer, int rank = 2, int64_t planes = 1, int64_t plane_stride = 0) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)outer, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)ld * esize, (cuuint64_t)plane_stride * esize};
  cuuint32_t box[3] = {(cuuint32_t)box_inner, (cuuint32_t)box_outer, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(map, dt, rank, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}
static bool make_map(CUtensorMap* map, const void* base, int64_t inner, int64_t outer, int64_t ld, int box_inner,
                     int box_outer) {
  return make_map_any(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, inner, outer, ld, box_inner, box_outer);
}

// bf16 matrix (rows ld apart) as atoms of 64 contiguous elements: dimensions 64, rows, n_atoms; box 64 x box_rows x box_atoms.
static bool make_map_atoms(CUtensorMap* map, const void* base, int64_t rows, int64_t ld, int64_t n_atoms, int box_rows, int box_atoms) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {64, (cuuint64_t)rows, (cuuint64_t)n_atoms};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 2, 128};
  cuuint32_t box[3] = {64, (cuuint32_t)box_rows, (cuuint32_t)box_atoms};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static int* device_error_ptr() {
  static int* ptr[64];
  int dev = 0;
  if (current_device(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  if (!ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_device_error) != cudaSuccess) return nullptr;
    ptr[dev] = reinterpret_cast<int*>(p);
  }
  return ptr[dev];
}

bool gemm_tc_eligible(int M, int N, int K, const Operand& A, const Operand& B, const Epilogue& ep) {
  if (A.kind != OP_BF16 || B.kind != OP_BF16) return false;
  if (M < 1 || N < 8 || K < 16 || (N & 7)) return false;
  auto ok = [](const Operand& o) {
    const bool kmaj = o.s_k == 1, mnmaj = o.s_row == 1 && o.s_k != 1;
    if (!kmaj && !mnmaj) return false;
    const int64_t ld = kmaj ? o.s_row : o.s_k;
    return (ld & 7) == 0 && aligned16(o.p);
  };
  if (!ok(A) || !ok(B)) return false;
  if ((ep.lo_cols & 7) || (ep.mask && ((ep.mask_cols & 7) || !ep.mask_bf16 || (ep.ld_mask & 7) || !aligned16(ep.mask))))
    return false;
  if (ep.out_lo && (!aligned16(ep.out_lo) || (ep.ld_lo & (ep.lo_bf16 ? 7 : 3)))) return false;
  if (ep.lo_cols < N) return false;                        // one output matrix per product
  if (!ep.lo_bf16 && (ep.bias || ep.relu || ep.mask)) return false;   // float outputs are plain sums
  if (ep.mask && ep.bits_out) return false;
  return true;
}

template <int kStages, int kBN, int kBK, bool kPair>
static ss_status launch_flow(const TcFlow<kTcMaxFlow>& f, int ctas, cudaStream_t st) {
  static bool attr_set[64];
  int dev = 0;
  SS_CUDA(current_device(&dev));
  const size_t smem = tc_smem_bytes(kStages, kPair ? kBN / 2 : kBN, kBK, sizeof(TcMeta) * kTcMaxFlow);
  if (dev >= 0 && dev < 64 && !attr_set[dev]) {
    SS_CUDA(cudaFuncSetAttribute(gemm_tc_kernel<kStages, kBN, kBK, kTcMaxFlow, kPair>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
    attr_set[dev] = true;
  }
  { SS_TIMED("gemm_tc_kernel", st);
  SS_CUDA(launch_cluster_dependent(gemm_tc_kernel<kStages, kBN, kBK, kTcMaxFlow, kPair>, ctas, kTcThreads, smem, kPair ? 2 : 1, st, f));
  }
  SS_LAUNCH_OK();
  return SS_OK;
}

// Fills one problem of a flow for tile width bn; returns its tile count (0 on failure).
static int fill_problem(TcProblem* pr, const TcJob& j, int bn, int bk, int tile_begin, bool pair) {
  const int tile_m = pair ? 2 * kBM : kBM;
  TcParams& p = pr->meta.p;
  p.M = j.M; p.N = j.N; p.K = j.K;
  p.a_mn = (j.A.s_k != 1);
  p.b_mn = (j.B.s_k != 1);
  const int cuts = (j.K + kAtomK - 1) / kAtomK;
  int ks = j.k_splits < 1 ? 1 : j.k_splits;
  if (ks > cuts) ks = cuts;
  p.k_splits = ks;
  p.split_stride = j.split_stride;
  p.ep = j.ep;
  p.dep = -1; p.dep_mode = 0; p.dep_k = 0; p.dep_need = 0; p.dep_need_all = 0;
  // Operand fetches: as few boxes per stage as the layout allows, and no wider than the matrix.  (The 3-d view of an
  // MN-major matrix, [atom][k][64 columns], has to cover whole atoms, hence the multiple of 64; its rows are ld apart.)
  auto fetch = [&](CUtensorMap* map, const Operand& o, int rows, bool mn, int tile_rows, int* form, int* bytes, int* k_atom) {
    const int most = rows < tile_rows ? (rows + 7) & ~7 : tile_rows;
    *k_atom = most * kAtomK * 2;
    if (!mn) {
      const bool whole = (j.K & (kAtomK - 1)) == 0;
      *form = whole ? FORM_K_ATOMS : FORM_K_BOXES;
      *bytes = *k_atom * (whole ? bk / kAtomK : 1);
      return whole ? make_map_atoms(map, o.p, rows, o.s_row, j.K / kAtomK, most, bk / kAtomK)
                   : make_map(map, o.p, j.K, rows, o.s_row, kAtomK, most);
    }
    if (rows & 63) {
      *form = FORM_MN_BOXES;
      *bytes = 64 * bk * 2;
      return make_map(map, o.p, rows, j.K, o.s_k, 64, bk);
    }
    const int atoms = (most + 63) / 64;
    *form = FORM_MN_ATOMS;
    *bytes = atoms * 64 * bk * 2;
    return make_map_atoms(map, o.p, j.K, o.s_k, rows / 64, bk, atoms);
  };
  const int load_n = pair ? bn / 2 : bn;
  if (!fetch(&pr->map_a, j.A, j.M, p.a_mn, kBM, &p.a_form, &p.a_box_bytes, &p.a_k_atom) ||
      !fetch(&pr->map_b, j.B, j.N, p.b_mn, load_n, &p.b_form, &p.b_box_bytes, &p.b_k_atom))
    return 0;
  // Outputs through TMA stores; a mask must come as sign bits (a mask given by values only takes plain loads and stores).
  const Epilogue& ep = j.ep;
  p.tma_out = 0;
  pr->map_lo = pr->map_a;                                  // defined, unused unless tma_out
  if (!ep.mask || ep.mask_bits) {
    bool ok;
    if (ep.lo_bf16) {
      ok = make_map_any(&pr->map_lo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ep.out_lo, j.N, j.M, ep.ld_lo, kChunk, 32);
    } else {
      const int64_t plane = ks > 1 ? j.split_stride : (int64_t)ep.ld_lo * j.M;
      ok = (plane & 3) == 0 && make_map_any(&pr->map_lo, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, ep.out_lo, j.N, j.M, ep.ld_lo, 32,
                                            32, 3, ks, plane);
    }
    if (!ok) return 0;
    p.tma_out = 1;
  }
  pr->meta.tile_begin = tile_begin;
  pr->meta.grid_x = (j.N + bn - 1) / bn;
  pr->meta.grid_y = (j.M + tile_m - 1) / tile_m;
  pr->meta.pad = 0;
  p.signals = 0;
  return pr->meta.grid_x * pr->meta.grid_y * ks;
}

static bool splits_ok(const TcJob& j) {
  const Epilogue& ep = j.ep;                 // slices are plain fp32 sums
  return j.k_splits <= 1 || !ep.lo_bf16;
}

// How many CTAs a flow takes.  A CTA of a flow holds its SM's shared memory and a third of its registers whether it works
// or waits for a row block, and the kernels of other streams then lack them; a flow that has the device to itself is
// fastest with a CTA on every SM.  Measured, us per round at 32 / 48 / 64 / 148 CTAs: three independent replicas of the
// ordinary model, batch 2048, 134 / 126 / 130 / 141 a round each (one round by itself 253 / 229 / 225 / 204); four replicas
// of one model 480 / 469 / 488 / 551; two of a model ten times as large, batch 4096, 684 / 675 / 684 / 733; scoring 8191
// examples of that model, nothing beside it, 451 / 342 / 292 / 212.  Eight and sixteen replicas are fastest with 32.  So:
// every SM when no other stream launches flows, else 192 CTAs shared by those who do, 32 to 48 each.
// `sharers` is what the caller knows (replicas trained side by side, 0 = nothing); the streams of the last flows launched
// on the device count as well.  The number changes no result.
constexpr int kFlowCtasMin = 32, kFlowCtasMax = 48, kFlowCtasShared = 192;
static int g_flow_ctas = 0;     // 0: by the rule above
int set_flow_ctas(int ctas) {
  if (ctas >= 0) g_flow_ctas = ctas;
  return g_flow_ctas > 0 ? g_flow_ctas : kFlowCtasMin;
}

int flow_ctas(int sharers, cudaStream_t st) {
  constexpr int kRecent = 8;
  struct Recent { cudaStream_t stream[kRecent]; unsigned next, filled; };
  static Recent recent[64];
  static std::mutex lock;
  if (g_flow_ctas > 0) return g_flow_ctas;
  int dev = 0, streams = 0;
  if (current_device(&dev) == cudaSuccess && dev >= 0 && dev < 64) {
    std::lock_guard<std::mutex> guard(lock);
    Recent& r = recent[dev];
    r.stream[r.next++ % kRecent] = st;
    if (r.filled < kRecent) ++r.filled;
    for (unsigned i = 0; i < r.filled; ++i) {
      bool seen = false;
      for (unsigned k = 0; k < i && !seen; ++k) seen = r.stream[k] == r.stream[i];
      streams += !seen;
    }
  }
  const int n = sharers > streams ? sharers : streams;
  if (n <= 1) return num_sms();
  const int share = kFlowCtasShared / n;
  return share < kFlowCtasMin ? kFlowCtasMin : (share > kFlowCtasMax ? kFlowCtasMax : share);
}

// The parameter block of a flow: tensor maps, tile sequence, dependencies.  It is a function of the arguments alone
// (addresses, shapes, tile width), and a training loop launches the same few flows over and over, while encoding their
// 30 to 60 tensor maps costs 8-15 us of host time; so the blocks built last are kept, at most kFlowPlans of them
// (12 KiB each) for the process, looked up by all of their arguments.
static ss_status build_flow(const TcJob* jobs, int n, int* ctrl, int max_rows, int bn, int bk, bool pair, int* err, TcFlow<kTcMaxFlow>* out) {
  TcFlow<kTcMaxFlow>& f = *out;
  memset(out, 0, sizeof(*out));                            // padding too: launches are compared byte by byte (step.cu)
  f.n = n;
  int total = 0;
  for (int i = 0; i < n; ++i) {
    const int tiles = fill_problem(&f.prob[i], jobs[i], bn, bk, total, pair);
    if (tiles < 1) return SS_ERR_CUDA;
    total += tiles;
  }
  for (int i = 0; i < n; ++i) {
    const TcJob& j = jobs[i];
    if (j.dep < 0) continue;
    TcParams& p = f.prob[i].meta.p;
    p.dep = j.dep; p.dep_mode = j.dep_mode; p.dep_k = j.dep_k;
    p.dep_need = kEpiWarps * f.prob[j.dep].meta.grid_x;      // every epilogue warp reports per tile
    f.prob[j.dep].meta.p.signals = 1;
    p.dep_need_all = p.dep_need * ((jobs[j.dep].M + kBM - 1) / kBM);
  }
  for (int i = n; i < kTcMaxFlow; ++i) f.prob[i] = f.prob[n - 1];   // never selected; keeps the parameter block defined
  f.total_tiles = total;
  f.ctrl = ctrl;
  f.rb_stride = (max_rows + kBM - 1) / kBM + 1;    // per product: one word per row block, then their total
  f.err = err;
  return SS_OK;
}

static void flow_key(const TcJob* jobs, int n, int* ctrl, int max_rows, int bn, bool pair, int* err, std::vector<int64_t>* key) {
  auto put = [&](auto v) { key->push_back((int64_t)v); };
  auto ptr = [&](const void* v) { key->push_back((int64_t)reinterpret_cast<intptr_t>(v)); };
  put(n); ptr(ctrl); put(max_rows); put(bn); put(pair); ptr(err);
  for (int i = 0; i < n; ++i) {
    const TcJob& j = jobs[i];
    const Epilogue& e = j.ep;
    put(j.M); put(j.N); put(j.K); put(j.k_splits); put(j.split_stride); put(j.dep); put(j.dep_mode); put(j.dep_k);
    for (const Operand* o : {&j.A, &j.B}) { ptr(o->p); put(o->kind); put(o->s_row); put(o->s_k); }
    ptr(e.bias); put(e.relu); ptr(e.mask); put(e.mask_bf16); put(e.ld_mask); put(e.mask_cols);
    ptr(e.out_lo); put(e.lo_bf16); put(e.ld_lo); put(e.lo_cols); ptr(e.out_hi); put(e.ld_hi);
    ptr(e.bits_out); put(e.ld_bits_out); ptr(e.mask_bits); put(e.ld_mask_bits);
  }
}

static ss_status flow_plan(const TcJob* jobs, int n, int* ctrl, int max_rows, int bn, bool pair, int* err, TcFlow<kTcMaxFlow>* out) {
  constexpr int kFlowPlans = 64;
  struct Plan { std::vector<int64_t> key; TcFlow<kTcMaxFlow> flow; uint64_t used = 0; };
  static std::vector<std::unique_ptr<Plan>> plans;
  static std::mutex lock;
  static uint64_t clock = 0;
  static thread_local std::vector<int64_t> key;
  key.clear();
  flow_key(jobs, n, ctrl, max_rows, bn, pair, err, &key);
  {
    std::lock_guard<std::mutex> guard(lock);
    for (auto& p : plans)
      if (p->key == key) { p->used = ++clock; memcpy(out, &p->flow, sizeof(*out)); return SS_OK; }
  }
  const ss_status st = build_flow(jobs, n, ctrl, max_rows, bn, bn == 256 ? 64 : 128, pair, err, out);
  if (st != SS_OK) return st;
  std::lock_guard<std::mutex> guard(lock);
  Plan* slot = nullptr;
  if ((int)plans.size() < kFlowPlans) {
    plans.emplace_back(new Plan);
    slot = plans.back().get();
  } else {
    for (auto& p : plans)                                  // the one not used for longest
      if (!slot || p->used < slot->used) slot = p.get();
  }
  slot->key = key; memcpy(&slot->flow, out, sizeof(*out)); slot->used = ++clock;
  return SS_OK;
}

ss_status gemm_tc_flow(const TcJob* jobs, int n, int* ctrl, int max_rows, int sharers, cudaStream_t st) {
  if (n < 1 || n > kTcMaxFlow) return SS_ERR_SHAPE;
  double flops = 0.0;
  for (int i = 0; i < n; ++i) {
    const TcJob& j = jobs[i];
    if (!splits_ok(j)) return SS_ERR_SHAPE;
    if (j.dep >= i || (j.dep >= 0 && (!ctrl || j.dep_mode < 1 || j.dep_mode > 2 || jobs[j.dep].k_splits > 1))) return SS_ERR_SHAPE;
    if (j.dep >= 0 && jobs[j.dep].M > max_rows) return SS_ERR_SHAPE;
    flops += 2.0 * j.M * j.N * j.K;
  }
  int* err = device_error_ptr();
  if (!err) return SS_ERR_CUDA;
  int ctas = num_sms();
  if (ctrl) {
    const int share = flow_ctas(sharers, st);
    if (g_step_sink) g_step_sink->ctas(share);
    if (share < ctas) ctas = share;
  }
  // Tile width.  128 x 256 tiles where the flow has three of them for two CTAs; with fewer, a layer takes as long as the k
  // loop of one tile on few SMs, and 64-wide tiles spread it (all SMs: forward chain of the ordinary model 43 us with
  // wide tiles, 29 with 64-wide ones; backward flow of a batch of 1337 47 and 34 us).  256 x 256 tiles on CTA pairs (a third less operand traffic per flop) where each pair gets four of
  // them and they are deep: with few k blocks a tile is bound by its epilogue and its dependencies, which the larger tiles
  // make coarser (four replicas of the ordinary model 493 -> 523 us a round on pairs, two of the large one 945 -> 860).
  long long t256 = 0, t_pair = 0, kb_pair = 0;
  for (int i = 0; i < n; ++i) {
    const long long ks = jobs[i].k_splits < 1 ? 1 : jobs[i].k_splits, gx = (jobs[i].N + 255) / 256;
    t256 += gx * ((jobs[i].M + kBM - 1) / kBM) * ks;
    const long long tiles = gx * ((jobs[i].M + 2 * kBM - 1) / (2 * kBM));
    t_pair += tiles * ks;
    kb_pair += tiles * ((jobs[i].K + 63) / 64);
  }
  const bool wide = 2 * t256 >= 3 * ctas;
  const bool pair = wide && ctas >= 2 && (ctrl ? t_pair >= 2 * ctas && kb_pair >= 12 * t_pair : t_pair >= ctas / 2);
  const int bn = wide ? 256 : 64;
  alignas(64) TcFlow<kTcMaxFlow> f;
  ss_status built;
  try {
    built = flow_plan(jobs, n, ctrl, max_rows, bn, pair, err, &f);
  } catch (...) {                                          // no host memory to keep the block: do without
    built = build_flow(jobs, n, ctrl, max_rows, bn, bn == 256 ? 64 : 128, pair, err, &f);
  }
  if (built != SS_OK) return built;
  const int total = f.total_tiles;
  if (pair) {
    ctas &= ~1;                                            // whole pairs
    if (2 * total < ctas) ctas = 2 * total;
    return launch_flow<kStagesPair, 256, 64, true>(f, ctas, st);
  }
  if (total < ctas) ctas = total;
  if (wide) return launch_flow<kStagesWide, 256, 64, false>(f, ctas, st);
  return launch_flow<kStagesSmall, 64, 128, false>(f, ctas, st);
}

ss_status gemm_tc(int M, int N, int K, const Operand& A, const Operand& B, const Epilogue& ep, cudaStream_t st,
                  int k_splits, int64_t split_stride) {
  TcJob j;
  j.M = M; j.N = N; j.K = K; j.A = A; j.B = B; j.ep = ep; j.k_splits = k_splits; j.split_stride = split_stride;
  return gemm_tc_flow(&j, 1, nullptr, 0, 0, st);
}

int read_device_error(bool clear) {
  int* d = device_error_ptr();
  if (!d) return -1;
  int v = 0;
  if (cudaMemcpy(&v, d, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
  if (clear && v != 0) {
    int z = 0;
    cudaMemcpy(d, &z, sizeof(int), cudaMemcpyHostToDevice);
  }
  return v;
}

}  // namespace ss

extern "C" {

int ss_device_error(int clear) { return ss::read_device_error(clear != 0); }

int ss_mlp_set_flow_ctas(int ctas) { return ss::set_flow_ctas(ctas); }

ss_status ss_gemm_bf16(const void* a, int a_mn_major, int64_t lda, const void* b, int b_mn_major, int64_t ldb,
                       float* c, int64_t ldc, int M, int N, int K, int force_simt, ss_stream stream) {
  using namespace ss;
  if (!a || !b || !c) return SS_ERR_NULL;
  if (M < 1 || N < 1 || K < 1 || lda < 1 || ldb < 1 || ldc < N) return SS_ERR_SHAPE;
  ss_status stt = check_arch();
  if (stt != SS_OK) return stt;
  Operand A{a, OP_BF16, a_mn_major ? 1 : lda, a_mn_major ? lda : 1};
  Operand B{b, OP_BF16, b_mn_major ? 1 : ldb, b_mn_major ? ldb : 1};
  Epilogue ep;
  ep.out_lo = c; ep.lo_bf16 = 0; ep.ld_lo = ldc; ep.lo_cols = N;
  if (force_simt) return gemm_simt(M, N, K, A, B, ep, as_stream(stream));
  if (!gemm_tc_eligible(M, N, K, A, B, ep)) return SS_ERR_ALIGN;
  return gemm_tc(M, N, K, A, B, ep, as_stream(stream), 1, 0);
}

}  // extern "C"
