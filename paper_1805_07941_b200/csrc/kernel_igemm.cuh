// Implicit-GEMM int8 convolution on the sm_100a tensor cores (Eq. 6 as a dense
// contraction): tcgen05.mma kind::i8 with int32 accumulators in tensor memory, operands
// staged in shared memory by TMA (NHWC activation boxes and K-major packed weights, both in
// the swizzled K-major canonical layout), and the requantization epilogue in registers.
//
// A tile is up to 128 output pixels x BN output channels.  The pixels of
// a tile are a box tq x tp x tn of the output (columns x rows x images), so that for filter
// tap (r, s) the activation operand is ONE TMA box of the input, shifted by the tap offset;
// taps that fall outside the image are zero-filled by the TMA unit, which is exact because
// the scheme is symmetric (zero is the integer 0).
//
// The kernel is persistent: a CTA walks a strided list of tiles, the operand ring keeps
// running across tiles, and two accumulator buffers in tensor memory let the epilogue of
// one tile overlap the loads and MMAs of the next.
//
// Warp roles (320 threads): warp 0 issues TMA loads, warp 1 owns tensor memory and issues
// the MMAs, warps 2-9 run the epilogue (each reads the TMEM lane quadrant warp_id % 4 and one
// half of the tile's columns).
// All waits on mbarriers are bounded; on expiry the CTA raises a status flag and leaves.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>
#include "epilogue.cuh"

namespace qc {

constexpr int kEpilogueWarps = 8;
constexpr int kGroupsPerWarp = 4;     // 16-column groups per epilogue warp: BN <= 2 * 4 * 16 = 128
constexpr int kGroupsPerWarpWide = 8; // the instantiations for 256-wide tiles (one CTA per SM)
constexpr int kIgemmThreads = 64 + 32 * kEpilogueWarps;
constexpr int kMaxStages = 12;
constexpr int kNpMaxProducts = 6;     // digit products of two operands of up to three digits
constexpr int kTileM = 128;

// Division of a non-negative 31-bit integer by a divisor fixed for the launch: q = umulhi(n, mul) >> shr with
// mul = ceil(2^(32 + shr) / d), shr = ceil(log2 d) - 1 (Granlund & Montgomery's round-up method; exact for
// n < 2^31), d == 1 passed through.  The set-up of a CTA decomposes its block index, its rows and its first ring
// positions into mixed-radix digits: about fifteen divisions by run-time values, some twenty dependent
// instructions each, at the head of every launch.
struct FastDiv {
  uint32_t mul, shr, d;
  __device__ __forceinline__ int div(int n) const {
    return d == 1u ? n : static_cast<int>(__umulhi(static_cast<uint32_t>(n), mul) >> shr);
  }
  __device__ __forceinline__ int divmod(int n, int* rem) const {
    const int q = div(n);
    *rem = n - q * static_cast<int>(d);
    return q;
  }
};

struct IgemmParams {
  int tq, tp, tn;                  // tile box, in output pixels (tq * tp * tn <= 128)
  int pool_bit;                    // 0, or the lane bit of a pixel's vertical neighbour (= tq, a power of two <= 16) when a
                                   //    2 x 2 max-pool is taken in the epilogue (tile rows q fastest: lane ^ 1 is the horizontal
                                   //    neighbour, lane ^ tq the vertical one)
  int q_step;                      // pixels from one box to the next along q, and the box's columns that are outputs:
                                   //    tq, except in the halo form (tq - (S - 1): the accumulator columns of the halo are dropped)
                                   //    and in the patch form (up to 14 of the box's 16)
  int tiles_q, tiles_p, tiles_n;   // number of boxes along each output axis
  int tiles_k;                     // number of output-channel tiles
  int BN;                          // channels per tile = MMA N (multiple of 16, <= 256)
  int BKC;                         // bytes of the contraction axis per pipeline stage (32/64/128)
  int nchunks;                     // channel chunks per filter tap
  int R, S;                        // taps seen by the kernel (1 x 1 for flattened / packed inputs)
  int pad_h, pad_w, stride_h, stride_w;
  int stages;
  int Q, P, Nimg;                  // output extent in the kernel's pixel space
  int K;                           // real output channels
  int out_c_offset, out_c_pitch;
  int tmem_cols;                   // power of two >= max(32, BN)
  int vec_store;                   // 1: 16-byte stores/loads of int8 rows are aligned
  int gen_simple;                  // general int8 epilogue: the accumulator bound leaves room for the single-pass rounding
  int gen_down, gen_away;          // EPI_GEN: round down (the table's bias then holds the mode's half), half away from zero by sign
  int gen_vec_y, gen_vec_res;      // general epilogues: 16 or 8 if every row piece of the output / the residual is aligned to
                                   //    so many bytes, else 0 (set per run from the pointers)
  uint32_t gen_stage_bytes;        // general epilogues: shared memory of the warps' staging rows (0 for the fast ones)
  int fast_epilogue;               // 1: int8 out, nearest-even, K % 16 == 0, aligned rows, and the
                                   //    accumulator bound leaves room for the rounding constant
  uint32_t a_stage_bytes, b_stage_bytes;   // shared-memory footprint per stage (1024-aligned)
  uint32_t out_stage_bytes;        // fast int8 epilogues: one staged output tile (128 rows of BN bytes, 1024-aligned); 0: direct stores
  uint32_t out_swz_mask;           // 16-byte-chunk XOR mask of the staged tile's swizzle (7 / 3 / 1 / 0 for BN = 128 / 64 / 32 / other)
  int out_stage_bufs;              // staged tiles: 2, or 3 when the residual tile is fetched into them by TMA one tile ahead; 0 with
                                   //    out_stage_bytes set: every CTA has one tile, and stages it in the ring, which is idle by then
  uint32_t res_tx_bytes;           // bytes one residual box delivers (BN * tq * tp * tn)
  uint32_t tx_bytes;               // bytes the TMA boxes of one ring stage deliver (activations + weights, or activations alone)
  int halo_s;                      // 0, or S: one activation stage is a box with a horizontal halo (tq = W + S - 1 pixels
                                   //    per image row) that serves the S horizontal taps of a filter row -- the same rows of
                                   //    shared memory, the operand's start advanced by one pixel per tap; the stage then
                                   //    carries S weight chunks, and the kernel sees R x 1 taps
  int halo_w;                      // taps of a stage that share a row of the box: halo_s, or 3 of 9 in the patch form, where the
                                   //    box also has tp + 2 rows and serves all taps of a 3 x 3 filter
  int store_rows;                  // patch form, staged tiles: image rows of a tile, each stored as a box of its own (the halo's
                                   //    columns stay behind); 0 otherwise
  uint32_t b_chunk_bytes;          // halo form: footprint of one of those weight chunks
  int tap_boxes;                   // 1: the halo_s taps of a stage are separate activation boxes, a_tap_bytes apart
                                   //    (grouped taps: no halo, no shifted reads; only the stage is shared)
  uint32_t a_tap_bytes;            // footprint of one activation box (= a_stage_bytes unless taps are grouped)
  FastDiv fd_tiles_k, fd_tiles_q, fd_tiles_p;   // by the tile counts (block index -> tile digits)
  FastDiv fd_tq, fd_tp;                         // by the box extents (accumulator row -> pixel of the box)
  FastDiv fd_nchunks, fd_S, fd_grid;            // ring position -> (chunk, tap); tiles of this CTA
  int walk_dk, walk_dq, walk_dp, walk_dn;       // digits of the grid size: the step from one tile of a CTA to its next
  int b_resident;                  // 1: the CTA's weight tile (all chunks) is loaded once and stays in shared memory;
                                   //    the ring then carries activations only and the CTA keeps one channel tile
  uint32_t b_res_tx_bytes;         // bytes of that weight tile
  int ksplit;                      // split contraction: CTAs of a cluster that share a tile (gen_stage_bytes is then their exchange area)
  int acc_bufs;                    // accumulator buffers in tensor memory: 2, or 1 when the products of EPI_NP leave no room
  // EPI_NP, floating-point operands: the chunks of a tap are those of np_products digit products one after the other, each
  // accumulated in BN columns of its own (np_cpp chunks per product)
  int np_products, np_cpp;
  FastDiv fd_np_cpp;
  int np_a[kNpMaxProducts];        // plane of the activations that product m multiplies
  int np_coef[kNpMaxProducts];     // weight of its accumulator in the 64-bit sum
  int np_n, np_p;                  // output type
  float np_top;                    // its beta_max
  int np_low;                      // EPI_NP3: low bits of the sum that the conversion keeps as one sticky bit, minus 7
};

// Error codes written to the status word.
constexpr int kStatusTimeout = -8;
// Polls granted to a wait for copies that were already issued (they always land): independent of the
// caller's wait limit, so that a CTA that gives up never retires with bulk copies still in flight
// into its shared memory.
constexpr unsigned int kDrainPolls = 1u << 22;

namespace ptx {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}
// The same probe with a time hint (nanoseconds): the hardware may suspend the thread until the phase completes
// or the hint runs out, whichever comes first.  A waiting role then issues next to no instructions and still
// wakes when the barrier flips.  Measured: it pays in the kernels that run one CTA per SM on long stages
// (SM-pair tiles: VGG conv4_2 92 -> 82 us) and costs 1-2 % in the two-CTA kernels of the short layers.
constexpr uint32_t kWaitHintNs = 2000;
__device__ __forceinline__ uint32_t mbar_try_wait_hint(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(kWaitHintNs)
      : "memory");
  return ok;
}
// Non-blocking probe of a barrier phase.
__device__ __forceinline__ uint32_t mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0,
                                            int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0,
                                            int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
// Shared-memory tile -> global tensor (clipped to the tensor's extent), tracked by the thread's bulk group.
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
      ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// All of this thread's bulk stores have finished READING shared memory (the source may be rewritten).
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// ... all but the most recent one.
__device__ __forceinline__ void bulk_wait_read_but_one() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
// Generic-proxy writes to shared memory become visible to the async proxy (TMA).
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void sts_uint4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
// True in exactly one lane of a fully converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile(
      "{\n\t.reg .b32 rx;\n\t.reg .pred px;\n\t"
      "elect.sync rx|px, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, px;\n\t}"
      : "=r"(pred));
  return pred != 0;
}
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// D[tmem] (+)= A[smem] * B[smem], int8 x int8 -> int32, issued by one thread.
__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// mbarrier arrives once every MMA issued so far by this thread has finished.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp receives lane (row) i.
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
// 32 lanes x 16 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster_uint4(uint32_t cluster_addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void grid_dependency_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void grid_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

}  // namespace ptx

// Shared-memory matrix descriptor of a K-major operand tile in the swizzled canonical
// layout: rows of `row_bytes` (= the swizzle span: 32, 64 or 128), groups of 8 rows
// contiguous, groups 8 * row_bytes apart.
__device__ __forceinline__ uint64_t make_kmajor_desc(uint32_t smem_addr, int row_bytes) {
  const uint64_t layout = row_bytes == 128 ? 2ull : (row_bytes == 64 ? 4ull : 6ull);
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr >> 4) & 0x3FFFu);            // start address / 16
  d |= 1ull << 16;                                                   // leading offset (unused here)
  d |= static_cast<uint64_t>((8u * row_bytes) >> 4) << 32;           // stride between 8-row groups / 16
  d |= 1ull << 46;                                                   // descriptor version for sm_100
  d |= layout << 61;
  return d;
}

// Instruction descriptor: int8 x int8 -> int32, both operands K-major, M = 128, N = bn.
__device__ __forceinline__ uint32_t make_idesc_i8(int bn) {
  uint32_t d = 0;
  d |= 2u << 4;                                  // accumulator format: signed 32-bit
  d |= 1u << 7;                                  // A: signed 8-bit
  d |= 1u << 10;                                 // B: signed 8-bit
  d |= static_cast<uint32_t>(bn >> 3) << 17;     // N / 8
  d |= static_cast<uint32_t>(kTileM >> 4) << 24; // M / 16
  return d;
}

// Per-channel epilogue constants, one 16-byte entry per output channel, prepared on the host:
//   x = bias, y = right shift s, and
//   int8 output:  z = 2^(s-1) - 1 (0 when s = 0), w = (s > 0) | 2^t << 1 with t the residual left shift;
//                 they serve the single-pass nearest-even rounding  (v + z + ((v >> s) & w & 1)) >> s
//                 (other rounding modes: see general_round);
//   general int8: y = s | t << 8;  wide output: y = t, with the bit pattern of the float 2^(e_x + e_w[k]) for float output.

struct IgemmShared {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint64_t res_full[3];           // residual tile landed in staged buffer i
  uint64_t b_full;                // resident weight tile landed
  uint32_t tmem_base;
  volatile int abort_flag;
  // Epilogue constants.  When they fit, those of ALL output channels are staged once per CTA; otherwise the current
  // and next tile's channels (at most 256 each) alternate.
  alignas(16) int32_t cst[2048];
};

constexpr uint32_t kCstBytes = sizeof(int32_t) * 2048;

// Bounded wait.  Returns false (and raises the CTA abort flag and the global status) if the
// barrier did not flip within `limit` polls, or if another role already gave up.
// HINT: probe with the hardware's suspend hint instead of sleeping between probes.
template <unsigned int SLEEP_NS = 0, bool HINT = false>
__device__ __forceinline__ bool wait_bounded(uint32_t bar, uint32_t parity, unsigned int limit,
                                             IgemmShared* sh, int* status) {
  for (unsigned int it = 0; it < limit; ++it) {
    if (HINT ? ptx::mbar_try_wait_hint(bar, parity) : ptx::mbar_try_wait(bar, parity)) return true;
    if (sh->abort_flag) return false;
    if (SLEEP_NS && !HINT) __nanosleep(SLEEP_NS);      // waiters that can afford it leave the issue slots alone
  }
  sh->abort_flag = 1;
  atomicExch(status, kStatusTimeout);
  return false;
}

// Barrier of the eight epilogue warps (named barrier 1) that also carries a vote: true in every
// thread if any thread passed `failed`.
__device__ __forceinline__ bool epilogue_vote(bool failed) {
  uint32_t any_failed;
  asm volatile(
      "{\n\t.reg .pred pin, pout;\n\t"
      "setp.ne.u32 pin, %1, 0;\n\t"
      "bar.red.or.pred pout, 1, %2, pin;\n\t"
      "selp.u32 %0, 1, 0, pout;\n\t}"
      : "=r"(any_failed)
      : "r"(failed ? 1u : 0u), "n"(kEpilogueWarps * 32)
      : "memory");
  return any_failed != 0;
}

struct TileCoord {
  int q0, p0, n0, k0;
};

// The tiles a CTA visits (blockIdx.x, + gridDim.x, ...) as mixed-radix digits advanced by addition
// with carries: integer divisions only once per kernel, not once per tile.
struct TileWalker {
  int kt, qt, pt, nt;          // digits of the current tile: channel tile fastest, then q, p, image
  int dk, dq, dp, dn;          // digits of the stride
  // first: the CTA's block index; the stride is the grid size, whose digits the host has worked out
  __device__ __forceinline__ void init(const IgemmParams& prm, int first) {
    int m = prm.fd_tiles_k.divmod(first, &kt);
    m = prm.fd_tiles_q.divmod(m, &qt);
    nt = prm.fd_tiles_p.divmod(m, &pt);
    dk = prm.walk_dk; dq = prm.walk_dq; dp = prm.walk_dp; dn = prm.walk_dn;
  }
  __device__ __forceinline__ void next(const IgemmParams& prm) {
    kt += dk; int c = kt >= prm.tiles_k; kt -= c ? prm.tiles_k : 0;
    qt += dq + c; c = qt >= prm.tiles_q; qt -= c ? prm.tiles_q : 0;
    pt += dp + c; c = pt >= prm.tiles_p; pt -= c ? prm.tiles_p : 0;
    nt += dn + c;
  }
  __device__ __forceinline__ TileCoord coord(const IgemmParams& prm) const {
    TileCoord t;
    t.q0 = qt * prm.q_step; t.p0 = pt * prm.tp; t.n0 = nt * prm.tn; t.k0 = kt * prm.BN;
    return t;
  }
};

// Epilogue variants, one kernel instantiation each so that a launch carries only the code it runs
// (these kernels are short; instruction fetch of unused paths is measurable):
//   FAST_I8 / FAST_I8_RES: int8 output, nearest-even, 8-bit saturation, K % 16 == 0, aligned rows,
//                          accumulator bound leaves room for the rounding constant; without / with residual
//   I8: any rounding mode, bit width, alignment;  I32, F32: wide or float output;  MAX: the largest |float output|
//                          alone, nothing is stored
//   GEN, GEN_RES: I8 where the wide value stays below 2^22 as well (see FLT below): any rounding mode by the rounding of the
//                          fused multiply-add; GEN_RES also serves the mode that needs the sign (half away, no ReLU)
//   NP: digit products of floating-point operands recombined in 64 bits and converted to the (n, p) output type
//   NP3: the three products of two-digit operands, recombined and converted in 32 bits (np3_encode)
//   FAST_I8_U / FAST_I8_RES_U: the same with one shift for all channels (per-layer scales): only the
//                          bias is per channel, everything else sits in kernel parameters
//   FLT_I8*:               the four fast variants again for layers whose wide value provably stays below
//                          2^22 in magnitude (bound computed from the actual weights at create time).
//                          There the integer ALU, the epilogue's bottleneck, is relieved by the FMA pipe:
//                          adding bias + 0x4B400000 yields the bit pattern of the float M + v, M = 1.5 * 2^23;
//                          (M + v) * 2^-s + M * (1 - 2^-s) is one FMA (product and addend exact) whose
//                          single rounding is nearest-even at integer granularity, i.e. the requantized
//                          value sits in the low mantissa byte; ReLU and the clamps are integer min/max
//                          on the bit patterns (positive floats order like integers).
enum : int { EPI_FAST_I8 = 0, EPI_FAST_I8_RES = 1, EPI_I8 = 2, EPI_I32 = 3, EPI_F32 = 4, EPI_FAST_I8_U = 5,
             EPI_FAST_I8_RES_U = 6, EPI_FLT_I8 = 7, EPI_FLT_I8_RES = 8, EPI_FLT_I8_U = 9, EPI_FLT_I8_RES_U = 10,
             EPI_MAX = 11, EPI_NP = 12, EPI_GEN = 13, EPI_GEN_RES = 14, EPI_NP3 = 15 };

template <int EPI> struct EpiTraits {
  static constexpr bool flt = EPI >= EPI_FLT_I8 && EPI <= EPI_FLT_I8_RES_U;
  static constexpr bool fast = EPI == EPI_FAST_I8 || EPI == EPI_FAST_I8_RES || EPI == EPI_FAST_I8_U ||
                               EPI == EPI_FAST_I8_RES_U || flt;
  static constexpr bool res = EPI == EPI_FAST_I8_RES || EPI == EPI_FAST_I8_RES_U || EPI == EPI_FLT_I8_RES ||
                              EPI == EPI_FLT_I8_RES_U;
  static constexpr bool uni = EPI == EPI_FAST_I8_U || EPI == EPI_FAST_I8_RES_U || EPI == EPI_FLT_I8_U ||
                              EPI == EPI_FLT_I8_RES_U;
  // shared-memory form of the channel constants: 4 bytes a channel when only the biases differ; for the float rounding
  // without residual 8, two channels side by side as {bias, bias, 2^-s, 2^-s}; else the table's 16
  static constexpr bool paired = EPI == EPI_FLT_I8 || EPI == EPI_GEN || EPI == EPI_I8 || EPI == EPI_I32 || EPI == EPI_F32 || EPI == EPI_MAX || EPI == EPI_NP3;
  static constexpr bool np = EPI == EPI_NP || EPI == EPI_NP3;
  static constexpr bool gen = EPI == EPI_GEN || EPI == EPI_GEN_RES, bytes = EPI == EPI_I8 || gen;   // general int8
  static constexpr uint32_t cst_bytes = uni ? 4u : paired ? 8u : 16u;
};

// Channel constant i of the table to its place in shared memory.
template <int EPI>
__device__ __forceinline__ void stage_constant(int32_t* cst, int i, const int4* __restrict__ entry) {
  if (EpiTraits<EPI>::uni) cst[i] = __ldg(&entry->x);
  else if (EpiTraits<EPI>::paired) {
    const int2 v = __ldg(reinterpret_cast<const int2*>(entry));
    cst[4 * (i >> 1) + (i & 1)] = v.x;
    cst[4 * (i >> 1) + 2 + (i & 1)] = v.y;
  } else reinterpret_cast<int4*>(cst)[i] = __ldg(entry);
}

constexpr int kMagicBits = 0x4B400000;        // bit pattern of 1.5 * 2^23 = 12582912.0f

// Two int32 -> two saturated int8 in the low half of the result, upper half taken from c's low half.
__device__ __forceinline__ uint32_t pack_sat_s8(int32_t hi_byte, int32_t lo_byte, uint32_t c) {
  uint32_t d;
  asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(hi_byte), "r"(lo_byte), "r"(c));
  return d;
}

// Byte B of a word, sign-extended to 32 bits in one permute (selector nibble 8 | B replicates the
// sign bit of byte B).
template <int B>
__device__ __forceinline__ int32_t sign_extend_byte(uint32_t w) {
  uint32_t d;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(d) : "r"(w), "n"(B | ((8 | B) << 4) | ((8 | B) << 8) | ((8 | B) << 12)));
  return static_cast<int32_t>(d);
}

// 16 bytes from a shared-memory address (the channel constants live there; an explicit shared load
// keeps the compiler from falling back to generic addressing).
__device__ __forceinline__ int4 lds_int4(uint32_t addr) {
  int4 v;
  asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}

// 16 accumulator columns of one row -> 16 output channels, stored by the thread (epilogue_16).  cst: shared-memory
// address of the tile's first channel constant.
// RELU: 0 / 1 fixed at compile time (the float-rounding variants: one predicated instruction less per
// output), 2 = taken from the parameters at run time.
// RSTG in the kernel's template list: 1 when the residual tile has been brought into the staged tile by TMA (read there,
// overwritten in place by the result), 2 the pooled epilogue, 4 the split contraction, 5 depthwise.
// The fast conversion of 16 accumulator columns to 16 int8 codes (four packed words): bias, residual << t, ReLU,
// shift with nearest-even rounding, saturation.  cst_g: shared-memory address of the first column's constant;
// rw: the 16 residual bytes (ignored without).
//
// The epilogue's warps are bound by their own latency (two CTAs of eight warps per SM, nine cycles from one instruction of
// a warp to its next), so what counts is instructions and exposed waits.  The constants of the first four columns come in
// from the caller, who loads them before it waits for the accumulators, and those of the next four are loaded before the
// current four's arithmetic.  Float rounding, per four outputs: four additions with the ReLU's maximum, two fused
// multiply-adds on pairs, and the clamp on pairs of 16-bit halves (the host sees to it that |result| < 2^15 before the
// clamp), which the byte packing needs anyway.
template <int EPI> struct CstAhead { int4 v[EpiTraits<EPI>::paired ? 2 : 1]; };
template <int EPI>
__device__ __forceinline__ CstAhead<EPI> load_ahead(uint32_t cst_g, int g) {
  CstAhead<EPI> a;
  if (EpiTraits<EPI>::uni) a.v[0] = lds_int4(cst_g + static_cast<uint32_t>(g * 16));
  if constexpr (EpiTraits<EPI>::paired) {
    a.v[0] = lds_int4(cst_g + static_cast<uint32_t>(g * 32));
    a.v[1] = lds_int4(cst_g + static_cast<uint32_t>(g * 32 + 16));
  }
  return a;
}

// (a.x * b.x + c.x, a.y * b.y + c.y), (a.x + b.x, a.y + b.y): one instruction each.
__device__ __forceinline__ float2 fma_pair(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 add_pair(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

// Four wide values + magic (as float bits, ReLU already applied) -> four codes.  scale: 2^-s per value; the addend is
// M (1 - 2^-s), or is made from M where only 2^-s is at hand: (M + v) - M is exact, and M + v 2^-s rounds once.
template <bool OWN_SCALE>
__device__ __forceinline__ uint32_t round_pack_4(const int32_t (&fb)[4], float2 s01, float2 s23, float2 add, bool relu, int lo) {
  constexpr float kM = 12582912.0f;
  float2 a = make_float2(__int_as_float(fb[0]), __int_as_float(fb[1])), b = make_float2(__int_as_float(fb[2]), __int_as_float(fb[3]));
  if (OWN_SCALE) {
    a = add_pair(a, make_float2(-kM, -kM));
    b = add_pair(b, make_float2(-kM, -kM));
  }
  const float2 r = fma_pair(a, s01, add), q = fma_pair(b, s23, add);
  uint32_t h0 = __byte_perm(__float_as_uint(r.x), __float_as_uint(r.y), 0x5410), h1 = __byte_perm(__float_as_uint(q.x), __float_as_uint(q.y), 0x5410);
  h0 = __vmins2(h0, 0x007F007Fu);
  h1 = __vmins2(h1, 0x007F007Fu);
  if (!relu) {
    const uint32_t lo2 = static_cast<uint32_t>(lo) * 0x10001u + (lo < 0 ? 0x10000u : 0u);   // lo in both halves
    h0 = __vmaxs2(h0, lo2);
    h1 = __vmaxs2(h1, lo2);
  }
  return __byte_perm(h0, h1, 0x6420);
}

template <int EPI, int RELU>
__device__ __forceinline__ void convert_16(const uint32_t* acc, uint32_t cst_g, CstAhead<EPI> ahead, const uint32_t (&rw)[4],
                                           const EpilogueParams& ep, uint32_t (&wds)[4]) {
  const bool relu = RELU == 2 ? ep.relu != 0 : RELU == 1;
  const float2 uni_c1 = make_float2(ep.uni_c1, ep.uni_c1), uni_c2 = make_float2(ep.uni_c2, ep.uni_c2);
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    int32_t q[4];
    int32_t rv[4] = {0, 0, 0, 0};
    if (EpiTraits<EPI>::res) {
      rv[0] = sign_extend_byte<0>(rw[g]); rv[1] = sign_extend_byte<1>(rw[g]);
      rv[2] = sign_extend_byte<2>(rw[g]); rv[3] = sign_extend_byte<3>(rw[g]);
    }
    const CstAhead<EPI> now = ahead;
    if (g < 3) ahead = load_ahead<EPI>(cst_g, g + 1);
    if constexpr (EpiTraits<EPI>::flt) {
      // x = bias + magic bits; y = bits of 2^-s; z = bits of M * (1 - 2^-s); w >> 1 = 2^t
      int32_t bias[4], mult[4];
      float2 s01 = uni_c1, s23 = uni_c1, add = uni_c2;
      if constexpr (EpiTraits<EPI>::uni) {
        bias[0] = now.v[0].x; bias[1] = now.v[0].y; bias[2] = now.v[0].z; bias[3] = now.v[0].w;
        mult[0] = mult[1] = mult[2] = mult[3] = ep.uni_w >> 1;
      } else if constexpr (EpiTraits<EPI>::paired) {
        bias[0] = now.v[0].x; bias[1] = now.v[0].y; bias[2] = now.v[1].x; bias[3] = now.v[1].y;
        s01 = make_float2(__int_as_float(now.v[0].z), __int_as_float(now.v[0].w));
        s23 = make_float2(__int_as_float(now.v[1].z), __int_as_float(now.v[1].w));
        add = make_float2(12582912.0f, 12582912.0f);
      } else {
        int4 c[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          c[b] = lds_int4(cst_g + static_cast<uint32_t>((g * 4 + b) * 16));
          bias[b] = c[b].x;
          mult[b] = c[b].w >> 1;
        }
        s01 = make_float2(__int_as_float(c[0].y), __int_as_float(c[1].y));
        s23 = make_float2(__int_as_float(c[2].y), __int_as_float(c[3].y));
        add = make_float2(12582912.0f, 12582912.0f);
      }
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        int32_t v = static_cast<int32_t>(acc[g * 4 + b]);
        if (EpiTraits<EPI>::res) v += rv[b] * mult[b];
        q[b] = relu ? __viaddmax_s32(v, bias[b], kMagicBits) : v + bias[b];
      }
      wds[g] = round_pack_4<!EpiTraits<EPI>::uni>(q, s01, s23, add, relu, ep.lo);
    } else {
      const int32_t bias4[4] = {now.v[0].x, now.v[0].y, now.v[0].z, now.v[0].w};
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int j = g * 4 + b;
        // per-channel constants from shared memory, or only the bias when the shift is per layer
        const int4 c = EpiTraits<EPI>::uni ? make_int4(bias4[b], ep.uni_shift, ep.uni_z, ep.uni_w)
                                           : lds_int4(cst_g + static_cast<uint32_t>(j * 16));
        int32_t v = static_cast<int32_t>(acc[j]);
        if (EpiTraits<EPI>::res) v += rv[b] * (c.w >> 1);         // residual scaled by 2^t
        v = relu ? __viaddmax_s32(v, c.x, 0) : v + c.x;
        // nearest-even:  (v + 2^(s-1) - 1 + lsb of the truncated quotient) >> s
        v = (v + c.z + ((v >> c.y) & c.w & 1)) >> c.y;
        q[b] = relu ? v : max(v, ep.lo);            // the upper bound is the 8-bit saturation below
      }
      wds[g] = pack_sat_s8(q[1], q[0], pack_sat_s8(q[3], q[2], 0u));
    }
  }
}

template <int EPI, int RELU>
__device__ __forceinline__ void epilogue_16(const uint32_t (&acc)[16], uint32_t cst, int col, int k, size_t pix,
                                            const IgemmParams& prm, const EpilogueParams& ep, const uint4& res16,
                                            void* __restrict__ y) {
  static_assert(EpiTraits<EPI>::fast, "16-byte-store variants; the others go through general_tile");
  const uint32_t rw[4] = {res16.x, res16.y, res16.z, res16.w};     // residual bytes, fetched ahead
  uint32_t wds[4];
  const uint32_t cst_g = cst + static_cast<uint32_t>(col) * EpiTraits<EPI>::cst_bytes;
  convert_16<EPI, RELU>(acc, cst_g, load_ahead<EPI>(cst_g, 0), rw, ep, wds);
  *reinterpret_cast<uint4*>(static_cast<int8_t*>(y) + pix * prm.out_c_pitch + prm.out_c_offset + k) =
      make_uint4(wds[0], wds[1], wds[2], wds[3]);
}

// ------------------------------------------------------------------------------------------------------------
// General epilogue: any rounding mode, bit width and alignment, K not a multiple of 16, int32 / float output, and
// the maximum of the float output.
//
// A thread holds one pixel's 16 channels at a time, but 32 lanes storing pieces of 32 different rows touch 32 sectors per
// instruction, and rows of K bytes may start at any address.  So every warp turns its part of the tile (32 rows x up to
// 64 bytes) around in its own rows of shared memory: conversion writes 16 bytes per thread, then consecutive lanes store
// consecutive pieces of a row; the residual comes in the same way.  Only the warp itself is involved (no block barrier).
// kGenPitch = 64 bytes of data + 16: 16-byte accesses of 8 consecutive rows fall into different banks.
//  - rows aligned to 16 or 8 bytes: pieces of that size (gen_copy_rows);
//  - any other alignment: the 4-byte words of global memory that the rows cover, shifted into place by a funnel shift,
//    a row's first and last partial word byte by byte (gen_copy_words).
// 13 x 35 x 27 x 96 -> 200, 3x3, residual, round-half-away: 58 -> 13 us with the byte stores gone.
constexpr int kGenPitch = 80;
constexpr int kGenWarpBytes = 32 * kGenPitch;

template <int V> struct GenVec;
template <> struct GenVec<8> { using T = uint2; };
template <> struct GenVec<16> { using T = uint4; };

// Moves a warp's rows between its staging rows and global memory: row r's `bytes` first bytes, at
// base + row_off(lane r) in global memory; rows whose lane passes ok == false are left out.
template <int V, bool STORE>
__device__ __forceinline__ void gen_copy_rows(uint8_t* stage, int8_t* base, long long row_off, bool ok, int bytes, int lane) {
  using T = typename GenVec<V>::T;
  constexpr int kLanes = 64 / V;                            // lanes side by side on a row
  const unsigned okmask = __ballot_sync(0xffffffffu, ok);
  const int c = (lane % kLanes) * V;
#pragma unroll
  for (int r0 = 0; r0 < 32; r0 += 32 / kLanes) {
    const int r = r0 + lane / kLanes;
    const long long off = __shfl_sync(0xffffffffu, row_off, r);
    if (((okmask >> r) & 1u) && c < bytes) {
      T* sp = reinterpret_cast<T*>(stage + r * kGenPitch + c);
      T* gp = reinterpret_cast<T*>(base + off + c);
      if (STORE) *gp = *sp; else *sp = __ldg(gp);
    }
  }
}

// The same for any alignment: the aligned words that hold the rows.  A loaded row stays where its words were: its first
// byte sits at its address modulo 4 (gen_row_words reads it).
template <bool STORE>
__device__ __forceinline__ void gen_copy_words(uint8_t* stage, int8_t* base, long long row_off, bool ok, int bytes, int lane) {
  const unsigned okmask = __ballot_sync(0xffffffffu, ok);
  const int words = (bytes + 6) >> 2;                       // at most, wherever the row starts (<= 17)
  const uint32_t inv = 65536u / static_cast<uint32_t>(words) + 1u;   // idx / words = (idx * inv) >> 16 for idx < 32 * 17
#pragma unroll 4
  for (int it = 0; it < words; ++it) {
    const int idx = it * 32 + lane;
    const int r = static_cast<int>((static_cast<uint32_t>(idx) * inv) >> 16), w = idx - r * words;
    int8_t* row = base + __shfl_sync(0xffffffffu, row_off, r);
    const int m = static_cast<int>(reinterpret_cast<uintptr_t>(row) & 3u), first = 4 * w - m;   // the word's first byte in the row
    if (!((okmask >> r) & 1u) || first >= bytes) continue;
    uint32_t* sp = reinterpret_cast<uint32_t*>(stage + r * kGenPitch) + w;
    const bool whole = first >= 0 && first + 4 <= bytes;
    if (STORE) {
      const uint32_t lo = w ? sp[-1] : 0u;                  // (w <= 16: the row's 17th word is inside its pitch)
      const uint32_t v = __funnelshift_l(lo, sp[0], 8 * m);
      if (whole) *reinterpret_cast<uint32_t*>(row + first) = v;
      else
        for (int j = 0; j < 4; ++j)
          if (first + j >= 0 && first + j < bytes) row[first + j] = static_cast<int8_t>(v >> (8 * j));
    } else {
      uint32_t v = 0u;
      if (whole) v = __ldg(reinterpret_cast<const uint32_t*>(row + first));
      else
        for (int j = 0; j < 4; ++j)
          if (first + j >= 0 && first + j < bytes) v |= static_cast<uint32_t>(static_cast<uint8_t>(__ldg(row + first + j))) << (8 * j);
      *sp = v;
    }
  }
}

// Rows at any alignment to global memory: their whole aligned 8-byte units by eight lanes a row, shifted into place, then
// every lane its own row's ends in pieces of 4, 2 and 1 bytes.  At least 16 bytes a row.  (With the ends among the units
// every step ran all three paths: 55 x 25 x 23 x 96 -> 746, 1 x 1, 32 us.)
__device__ __forceinline__ void gen_store_units(const uint8_t* stage, int8_t* base, long long row_off, bool ok, int bytes, int lane) {
  const unsigned okmask = __ballot_sync(0xffffffffu, ok);
#pragma unroll
  for (int r0 = 0; r0 < 32; r0 += 4) {
    const int r = r0 + (lane >> 3);
    int8_t* row = base + __shfl_sync(0xffffffffu, row_off, r);
    const int head = static_cast<int>(-reinterpret_cast<uintptr_t>(row) & 7u), at = head + 8 * (lane & 7);
    if (((okmask >> r) & 1u) && at + 8 <= bytes) {
      const uint32_t* sp = reinterpret_cast<const uint32_t*>(stage + r * kGenPitch + (at & ~3));
      const uint32_t w0 = sp[0], w1 = sp[1], w2 = sp[2];    // (inside the row's pitch)
      *reinterpret_cast<uint2*>(row + at) = make_uint2(__funnelshift_r(w0, w1, 8 * (at & 3)), __funnelshift_r(w1, w2, 8 * (at & 3)));
    }
  }
  if (!ok) return;
  int8_t* row = base + row_off;
  const uint8_t* src = stage + lane * kGenPitch;
  const int head = static_cast<int>(-reinterpret_cast<uintptr_t>(row) & 7u);
  if (head) {
    const uint2 w = *reinterpret_cast<const uint2*>(src);
    int pos = 0;
    if (head & 1) { row[0] = static_cast<int8_t>(w.x); pos = 1; }
    if (head & 2) {
      *reinterpret_cast<uint16_t*>(row + pos) = static_cast<uint16_t>(w.x >> (8 * pos));
      pos += 2;
    }
    if (head & 4) *reinterpret_cast<uint32_t*>(row + pos) = __funnelshift_r(w.x, w.y, 8 * pos);
  }
  const int tail = (bytes - head) & 7, start = bytes - tail;
  if (tail) {
    const uint32_t* sp = reinterpret_cast<const uint32_t*>(src + (start & ~3));
    const uint32_t lo = __funnelshift_r(sp[0], sp[1], 8 * (start & 3)), hi = __funnelshift_r(sp[1], sp[2], 8 * (start & 3));
    int8_t* dst = row + start;
    if (tail & 4) *reinterpret_cast<uint32_t*>(dst) = lo;
    const uint32_t w = tail & 4 ? hi : lo;
    dst += tail & 4;
    if (tail & 2) *reinterpret_cast<uint16_t*>(dst) = static_cast<uint16_t>(w);
    if (tail & 1) dst[tail & 2] = static_cast<int8_t>(tail & 2 ? w >> 16 : w);
  }
}

// The same way in.  A loaded row keeps its place relative to the words of memory: its first byte at its address modulo 4.
__device__ __forceinline__ void gen_load_units(uint8_t* stage, const int8_t* base, long long row_off, bool ok, int bytes, int lane) {
  const unsigned okmask = __ballot_sync(0xffffffffu, ok);
#pragma unroll
  for (int r0 = 0; r0 < 32; r0 += 4) {
    const int r = r0 + (lane >> 3);
    const int8_t* row = base + __shfl_sync(0xffffffffu, row_off, r);
    const int head = static_cast<int>(-reinterpret_cast<uintptr_t>(row) & 7u), at = head + 8 * (lane & 7);
    if (((okmask >> r) & 1u) && at + 8 <= bytes) {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(row + at));
      uint32_t* sp = reinterpret_cast<uint32_t*>(stage + r * kGenPitch + at + (reinterpret_cast<uintptr_t>(row) & 3u));
      sp[0] = v.x;
      sp[1] = v.y;
    }
  }
  if (!ok) return;
  const int8_t* row = base + row_off;
  uint8_t* dst = stage + lane * kGenPitch + (reinterpret_cast<uintptr_t>(row) & 3u);
  const int head = static_cast<int>(-reinterpret_cast<uintptr_t>(row) & 7u), tail = (bytes - head) & 7;
  int pos = 0;
  if (head & 1) { dst[0] = static_cast<uint8_t>(__ldg(row)); pos = 1; }
  if (head & 2) {
    *reinterpret_cast<uint16_t*>(dst + pos) = __ldg(reinterpret_cast<const uint16_t*>(row + pos));
    pos += 2;
  }
  if (head & 4) *reinterpret_cast<uint32_t*>(dst + pos) = __ldg(reinterpret_cast<const uint32_t*>(row + pos));
  pos = bytes - tail;
  if (tail & 4) {
    *reinterpret_cast<uint32_t*>(dst + pos) = __ldg(reinterpret_cast<const uint32_t*>(row + pos));
    pos += 4;
  }
  if (tail & 2) {
    *reinterpret_cast<uint16_t*>(dst + pos) = __ldg(reinterpret_cast<const uint16_t*>(row + pos));
    pos += 2;
  }
  if (tail & 1) dst[pos] = static_cast<uint8_t>(__ldg(row + pos));
}

template <bool STORE>
__device__ __forceinline__ void gen_copy(int vec, uint8_t* stage, int8_t* base, long long row_off, bool ok, int bytes, int lane) {
  if (bytes <= 0) return;
  if (vec == 16) gen_copy_rows<16, STORE>(stage, base, row_off, ok, bytes, lane);
  else if (vec == 8) gen_copy_rows<8, STORE>(stage, base, row_off, ok, bytes, lane);
  else if (STORE && bytes >= 16) gen_store_units(stage, base, row_off, ok, bytes, lane);
  else if (bytes >= 16) gen_load_units(stage, base, row_off, ok, bytes, lane);
  else gen_copy_words<STORE>(stage, base, row_off, ok, bytes, lane);
}

// Bytes 16 i ... of this lane's loaded row, which starts `m` bytes into its staging row.
__device__ __forceinline__ uint4 gen_row_words(const uint8_t* stage_row, int i, int m) {
  const uint4 a = *reinterpret_cast<const uint4*>(stage_row + 16 * i);
  const uint32_t next = *reinterpret_cast<const uint32_t*>(stage_row + 16 * i + 16);
  return make_uint4(__funnelshift_r(a.x, a.y, 8 * m), __funnelshift_r(a.y, a.z, 8 * m), __funnelshift_r(a.z, a.w, 8 * m),
                    __funnelshift_r(a.w, next, 8 * m));
}

// v / 2^s -> pattern of the nearest value of an (n, p) type; ties to the even pattern; saturation at beta_max;
// a zero magnitude is pattern 0.  The magnitude is first made a binary32 number with its last bit sticky (round to odd:
// 24 bits hold at least two more than any of these types, so rounding again is exact), then a float addition rounds it
// to the type's grid: see dynfloat_mag, whose constants these are.
struct NpEncode {
  uint32_t ke_min, ke_up, ke_off;
  int p, sign_bit;
  float top;
};
__device__ __forceinline__ uint32_t np_encode(long long v, int s, const NpEncode& f) {
  const unsigned long long mag = v < 0 ? 0ull - static_cast<unsigned long long>(v) : static_cast<unsigned long long>(v);
  const int lz = __clzll(static_cast<long long>(mag));
  const unsigned long long m = mag << (lz & 63);
  const uint32_t hi = static_cast<uint32_t>(m >> 32), lo = static_cast<uint32_t>(m);
  const uint32_t sig = (hi >> 8) | (((hi & 0xFFu) | lo) != 0u ? 1u : 0u);   // 24 bits, the first one set
  // value = sig * 2^(40 - lz - s); exponent field minus the implicit bit that sig carries
  const float exact = __uint_as_float((static_cast<uint32_t>(63 - lz - s + 126) << 23) + sig);
  const float a = fminf(mag ? exact : 0.0f, f.top);
  const uint32_t ke = max(__float_as_uint(a) & 0x7F800000u, f.ke_min);
  const float t = __uint_as_float(ke + f.ke_up) + a;
  uint32_t code = (ke >> (23 - f.p)) + __float_as_uint(t) - ke - f.ke_off;
  if (f.p == 0) {
    // bare powers of two: the tie at 1.5 * 2^k goes to the even exponent field, the one at 1/2 to 0
    const uint32_t fr = __float_as_uint(a) & 0x7FFFFFu, E = (__float_as_uint(a) >> 23) - 126u;
    code = a >= 1.0f ? E + (fr + (E & 1u) > 0x400000u ? 1u : 0u) : (a > 0.5f ? 1u : 0u);
  }
  return code | ((v < 0 && code) ? 1u << f.sign_bit : 0u);
}

// The same for the three products of two-digit operands, without 64-bit arithmetic.  The sum is
//   v = P0 + bias + 128 (P01 - P0 - P1) + 128^2 P1 = a + 128 h  with a = P0 + bias, h = P01 - P0 + 127 P1,
// both int32.  The shift s leaves every number that the conversion compares with (grid points and their midpoints) a multiple of
// 2^(s-1); so of v's low np_low + 7 <= s - 1 bits only whether they are zero matters: u = 2 floor(v / 2^(np_low+7)) + sticky, below
// 2^23 in magnitude (the host chose np_low so), is an exact binary32 number, and u 2^(np_low+6-s) lies between the same
// neighbours as v / 2^s.  scale: 2^(np_low+6-s).  23 instructions an output; with 64-bit sums 45.
struct Np3Encode {
  uint32_t ke_min, ke_up, ke_off, low_mask;
  int low, p, sign_bit;
  float top;
};
template <bool RELU>
__device__ __forceinline__ uint32_t np3_encode(int32_t p0, int32_t p1, int32_t p01, int32_t bias, float scale, const Np3Encode& f) {
  const int32_t a = p0 + bias;
  // (modulo 2^32: x itself is below 2^31)
  const int32_t x = static_cast<int32_t>(static_cast<uint32_t>(p01) - static_cast<uint32_t>(p0) + 127u * static_cast<uint32_t>(p1)) + (a >> 7);
  const uint32_t rest = (static_cast<uint32_t>(a) & 127u) | (static_cast<uint32_t>(x) & f.low_mask) << 7;
  int32_t u = 2 * (x >> f.low) + static_cast<int32_t>(min(rest, 1u));
  const bool negative = !RELU && u < 0;
  u = RELU ? max(u, 0) : abs(u);
  const float m = fminf((__int_as_float(0x4B000000 | u) - 8388608.0f) * scale, f.top);
  const uint32_t ke = max(__float_as_uint(m) & 0x7F800000u, f.ke_min);
  const float t = __uint_as_float(ke + f.ke_up) + m;
  uint32_t code = (ke >> (23 - f.p)) + __float_as_uint(t) - ke - f.ke_off;
  if (f.p == 0) {                                            // (as in np_encode)
    const uint32_t fr = __float_as_uint(m) & 0x7FFFFFu, E = (__float_as_uint(m) >> 23) - 126u;
    code = m >= 1.0f ? E + (fr + (E & 1u) > 0x400000u ? 1u : 0u) : (m > 0.5f ? 1u : 0u);
  }
  return code | (negative && code ? 1u << f.sign_bit : 0u);
}

// v / 2^s rounded in the descriptor's mode, in one pass: (v + z + cond) >> s, with m = 2^s - 1 (odd unless s = 0):
//   nearest-even: z = m / 2, cond = lowest bit of the truncated quotient;  half away: z = m / 2, cond = v > 0;
//   half up: z = (m + 1) / 2;  floor: z = 0;  no cond where s = 0.
template <bool EVEN>
__device__ __forceinline__ int32_t general_round(int32_t v, int s, int rounding) {
  const int32_t m = static_cast<int32_t>((1u << s) - 1u);
  if (EVEN) return (v + (m >> 1) + ((v >> s) & m & 1)) >> s;
  const int32_t z = rounding == 1 ? (m >> 1) + ((v > 0 ? 1 : 0) & m) : rounding == 2 ? static_cast<int32_t>((static_cast<uint32_t>(m) + 1u) >> 1) : 0;
  return (v + z) >> s;
}

// One group of 16 columns of the integer general int8 epilogue -> 16 codes in the staging row.  Channel constants: the bias
// and s | t << 8, 8 bytes a channel (with 16, reading them took as long as everything else).  A negative wide value never
// rounds above zero, so a ReLU is the lower clamp.
template <bool SIMPLE, bool EVEN>
__device__ __forceinline__ void general_int8_16(const uint32_t (&acc)[16], uint32_t cst_g, const uint4& res16, const EpilogueParams& ep, uint32_t stage) {
  const uint32_t rw[4] = {res16.x, res16.y, res16.z, res16.w};
  const int lo = ep.relu ? max(ep.lo, 0) : ep.lo;
  uint32_t wds[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const int4 a = lds_int4(cst_g + static_cast<uint32_t>(g * 32)), c = lds_int4(cst_g + static_cast<uint32_t>(g * 32 + 16));
    const int32_t bias[4] = {a.x, a.y, c.x, c.y}, pk[4] = {a.z, a.w, c.z, c.w};
    const int32_t rv[4] = {sign_extend_byte<0>(rw[g]), sign_extend_byte<1>(rw[g]), sign_extend_byte<2>(rw[g]), sign_extend_byte<3>(rw[g])};
    int32_t q[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int sft = pk[b] & 31;
      int32_t v = static_cast<int32_t>(acc[4 * g + b]) + bias[b] + static_cast<int32_t>(static_cast<uint32_t>(rv[b]) << (pk[b] >> 8));
      if (!SIMPLE && ep.relu) v = max(v, 0);
      q[b] = min(max(SIMPLE ? general_round<EVEN>(v, sft, ep.rounding) : round_shift(v, sft, ep.rounding), lo), ep.hi);
    }
    wds[g] = __byte_perm(__byte_perm(q[0], q[1], 0x0040), __byte_perm(q[2], q[3], 0x0040), 0x5410);
  }
  ptx::sts_uint4(stage, wds[0], wds[1], wds[2], wds[3]);
}

// One group of 16 columns with wide output.  res16: the residual bytes (zero without).  int32 / float: 16 words to the staging
// row; MAX: into *mx.
template <int EPI>
__device__ __forceinline__ void general_16(const uint32_t (&acc)[16], uint32_t cst_g, const uint4& res16, int ncols, bool row_ok,
                                           const IgemmParams& prm, const EpilogueParams& ep, uint32_t stage, float* mx) {
  const uint32_t rw[4] = {res16.x, res16.y, res16.z, res16.w};
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const int4 k01 = lds_int4(cst_g + static_cast<uint32_t>(g * 32)), k23 = lds_int4(cst_g + static_cast<uint32_t>(g * 32 + 16));
    const int32_t bias[4] = {k01.x, k01.y, k23.x, k23.y}, pk[4] = {k01.z, k01.w, k23.z, k23.w};
    uint32_t o[4];
    const int32_t rv[4] = {sign_extend_byte<0>(rw[g]), sign_extend_byte<1>(rw[g]), sign_extend_byte<2>(rw[g]), sign_extend_byte<3>(rw[g])};
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int j = g * 4 + b;
      int32_t v = static_cast<int32_t>(acc[j]) + bias[b] + static_cast<int32_t>(static_cast<uint32_t>(rv[b]) << (pk[b] & 31));
      if (ep.relu) v = max(v, 0);
      if (EPI == EPI_I32) {
        o[b] = static_cast<uint32_t>(v);
      } else {
        // beta -> float: the bits of 2^(e_x + e_w[k]); the product is exact (power of two)
        const float f = __int2float_rn(v) * __int_as_float(pk[b] & 0x7F800000);
        if (EPI == EPI_MAX) {
          if (row_ok && j < ncols) *mx = fmaxf(*mx, fabsf(f));
        } else {
          o[b] = __float_as_uint(f);
        }
      }
    }
    if (EPI != EPI_MAX) {
      ptx::sts_uint4(stage + g * 16u, o[0], o[1], o[2], o[3]);
    }
  }
}

// One group of 16 columns of the float-rounding general epilogues (EPI_GEN, EPI_GEN_RES) -> 16 codes in the staging row.
// q = magic + v + h, an integer below 2^22 in magnitude; with h = 2^(s-1) and the multiply-add rounding down that is round
// half up, with h = 0 floor, and rounding to nearest half to even.  Half away from zero is half up from zero on, and one
// less below: the table's z = h - 1, plus one where v >= 0 (bit 22 of the float's pattern); with a ReLU it is half up.
template <int EPI>
__device__ __forceinline__ void gen_flt_16(const uint32_t (&acc)[16], uint32_t cst_g, const uint4& res16, const IgemmParams& prm,
                                           const EpilogueParams& ep, uint32_t stage) {
  constexpr float kM = 12582912.0f;
  const uint32_t rw[4] = {res16.x, res16.y, res16.z, res16.w};
  const int lo = ep.relu ? 0 : ep.lo;
  const uint32_t lo2 = __byte_perm(static_cast<uint32_t>(lo), 0u, 0x1010), hi2 = __byte_perm(static_cast<uint32_t>(ep.hi), 0u, 0x1010);
  auto fma_down = [](float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "fma.rm.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
  };
  uint32_t wds[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    int32_t q[4];
    float2 s01, s23;
    if constexpr (EpiTraits<EPI>::paired) {
      const int4 a = lds_int4(cst_g + static_cast<uint32_t>(g * 32)), b = lds_int4(cst_g + static_cast<uint32_t>(g * 32 + 16));
      q[0] = static_cast<int32_t>(acc[4 * g]) + a.x; q[1] = static_cast<int32_t>(acc[4 * g + 1]) + a.y;
      q[2] = static_cast<int32_t>(acc[4 * g + 2]) + b.x; q[3] = static_cast<int32_t>(acc[4 * g + 3]) + b.y;
      s01 = make_float2(__int_as_float(a.z), __int_as_float(a.w));
      s23 = make_float2(__int_as_float(b.z), __int_as_float(b.w));
    } else {
      const int32_t rv[4] = {sign_extend_byte<0>(rw[g]), sign_extend_byte<1>(rw[g]), sign_extend_byte<2>(rw[g]), sign_extend_byte<3>(rw[g])};
      float sc[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int4 c = lds_int4(cst_g + static_cast<uint32_t>((g * 4 + b) * 16));
        q[b] = static_cast<int32_t>(acc[4 * g + b]) + c.x + rv[b] * (c.w >> 1);
        if (prm.gen_away) q[b] += c.z + ((q[b] >> 22) & 1);
        sc[b] = __int_as_float(c.y);
      }
      s01 = make_float2(sc[0], sc[1]);
      s23 = make_float2(sc[2], sc[3]);
    }
    const float2 m = make_float2(kM, kM);
    const float2 a = add_pair(make_float2(__int_as_float(q[0]), __int_as_float(q[1])), make_float2(-kM, -kM));
    const float2 b = add_pair(make_float2(__int_as_float(q[2]), __int_as_float(q[3])), make_float2(-kM, -kM));
    const float2 x = prm.gen_down ? fma_down(a, s01, m) : fma_pair(a, s01, m), y = prm.gen_down ? fma_down(b, s23, m) : fma_pair(b, s23, m);
    uint32_t h0 = __byte_perm(__float_as_uint(x.x), __float_as_uint(x.y), 0x5410), h1 = __byte_perm(__float_as_uint(y.x), __float_as_uint(y.y), 0x5410);
    h0 = __vmaxs2(__vmins2(h0, hi2), lo2);
    h1 = __vmaxs2(__vmins2(h1, hi2), lo2);
    wds[g] = __byte_perm(h0, h1, 0x6420);
  }
  ptx::sts_uint4(stage, wds[0], wds[1], wds[2], wds[3]);
}

// 16 accumulator columns of one row with a 2 x 2 / stride 2 max-pool over pixels taken on the way.  The conversion
// (bias, ReLU, shift with rounding, saturation) is non-decreasing in the accumulator, so the maximum over the four
// pixels of a window is taken on the raw accumulators and converted once.  The four pixels of a window sit in the
// lanes l, l ^ 1 (horizontal neighbour) and l ^ vbit, l ^ 1 ^ vbit (vertical neighbours) of one warp.  The
// maximum is a reduce-scatter: lanes l and l ^ 1 exchange one half of the 16 columns each and keep the other,
// then l and l ^ vbit exchange one half of those 8, so every lane ends up with the window's maxima of 4 of the 16
// columns, converts those and stores 4 bytes; the window's four lanes write 16 consecutive bytes of the pooled
// pixel.  All 32 lanes must call (shuffles); `store_ok` says whether this lane's pixel lies inside the image.
// Fast epilogues without residual only.
template <int EPI, int RELU>
__device__ __forceinline__ void epilogue_pool_16(const uint32_t (&acc)[16], uint32_t cst, int col, int k, size_t pooled_pix,
                                                 bool store_ok, int lane, int vbit, const IgemmParams& prm,
                                                 const EpilogueParams& ep, void* __restrict__ y) {
  static_assert(EpiTraits<EPI>::fast && !EpiTraits<EPI>::res, "pooled epilogue: fast variants without residual");
  const bool relu = RELU == 2 ? ep.relu != 0 : RELU == 1;
  const bool odd_q = (lane & 1) != 0, odd_p = (lane & vbit) != 0;
  int32_t r8[8], v4[4];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int32_t lo = static_cast<int32_t>(acc[i]), hi = static_cast<int32_t>(acc[i + 8]);
    const int32_t keep = odd_q ? hi : lo, send = odd_q ? lo : hi;
    r8[i] = max(keep, __shfl_xor_sync(0xffffffffu, send, 1));
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int32_t keep = odd_p ? r8[i + 4] : r8[i], send = odd_p ? r8[i] : r8[i + 4];
    v4[i] = max(keep, __shfl_xor_sync(0xffffffffu, send, vbit));
  }
  const int c0 = (odd_q ? 8 : 0) + (odd_p ? 4 : 0);              // this lane's 4 columns of the 16
  const uint32_t cst_g = cst + static_cast<uint32_t>(col + c0) * EpiTraits<EPI>::cst_bytes;
  uint32_t word;
  if constexpr (EpiTraits<EPI>::flt) {
    const CstAhead<EPI> k = load_ahead<EPI>(cst_g, 0);
    int32_t q[4];
    int32_t bias[4] = {k.v[0].x, k.v[0].y, k.v[0].z, k.v[0].w};
    float2 s01 = make_float2(ep.uni_c1, ep.uni_c1), s23 = s01, add = make_float2(ep.uni_c2, ep.uni_c2);
    if constexpr (EpiTraits<EPI>::paired) {
      bias[2] = k.v[1].x; bias[3] = k.v[1].y;
      s01 = make_float2(__int_as_float(k.v[0].z), __int_as_float(k.v[0].w));
      s23 = make_float2(__int_as_float(k.v[1].z), __int_as_float(k.v[1].w));
      add = make_float2(12582912.0f, 12582912.0f);
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) q[b] = relu ? __viaddmax_s32(v4[b], bias[b], kMagicBits) : v4[b] + bias[b];
    word = round_pack_4<!EpiTraits<EPI>::uni>(q, s01, s23, add, relu, ep.lo);
  } else {
    int4 bq = make_int4(0, 0, 0, 0);
    if (EpiTraits<EPI>::uni) bq = lds_int4(cst_g);
    const int32_t bias4[4] = {bq.x, bq.y, bq.z, bq.w};
    int32_t q[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int4 c = EpiTraits<EPI>::uni ? make_int4(bias4[b], ep.uni_shift, ep.uni_z, ep.uni_w)
                                         : lds_int4(cst_g + static_cast<uint32_t>(b) * 16u);
      int32_t v = relu ? __viaddmax_s32(v4[b], c.x, 0) : v4[b] + c.x;
      v = (v + c.z + ((v >> c.y) & c.w & 1)) >> c.y;
      q[b] = relu ? v : max(v, ep.lo);
    }
    word = pack_sat_s8(q[1], q[0], pack_sat_s8(q[3], q[2], 0u));
  }
  if (store_ok)
    *reinterpret_cast<uint32_t*>(static_cast<int8_t*>(y) + pooled_pix * prm.out_c_pitch + prm.out_c_offset + k + c0) = word;
}

// Split contraction (RSTG == 4).  A layer with few tiles and a long contraction (ResNet's 14 x 14 and 7 x 7 layers on one
// image: 8 to 32 tiles, up to 4608 bytes) leaves most SMs idle while each busy one walks its chain of stages.  A cluster
// of `ksplit` CTAs then shares a tile: each accumulates its part of the contraction in its own tensor memory, sends the
// 16-column groups it does not own to their owner's shared memory (group g belongs to CTA g % ksplit), and after one
// cluster barrier every CTA adds up, converts and stores its own groups.  Integer sums: the result does not depend on
// the split.  Exchange area: [own group][sender][4 columns][128 rows][16 bytes], so that a warp's 16-byte accesses are
// consecutive.  Per launch in a train: 7 x 7 x 512 3 x 3 6.9 -> 4.5 us, 7 x 7 x 2048 -> 512 6.2 -> 4.2, 14 x 14 x 256
// 3 x 3 4.6 -> 4.0; ResNet-50 on one image 212 -> 199 us.
//
// Depthwise 3 x 3 (RSTG == 5).  A tile's BN channels are its contraction chunk too (BKC = BN bytes of a pixel), and only
// the diagonal of a tap's matrix is not zero.  An MMA of N <= 96 takes 54 cycles whatever its width, so the chunk's MMAs
// (32 bytes along K each) multiply a 32 x 32 block, each into accumulator columns of its own: 9 taps x BN / 32 MMAs a
// tile, which leaves the CUDA cores the conversion alone (the tap-packed kernels spend 17 instructions an output).
// Weights: [channel][tap][32], the tap's weight at position channel % 32.  Per launch, batch 256: 112 x 112 x 64 stride 2
// 61 -> 49 us, 56 x 56 x 128 78 -> 71, stride 2 35 -> 28, 28 x 28 x 256 43 -> 37, stride 2 21 -> 14, 14 x 14 x 512
// 26 -> 22, 7 x 7 x 1024 16.7 -> 14.2; a single image 6.4 -> 4.6.
//
// Persistent kernel: each CTA walks tiles blockIdx.x, blockIdx.x + gridDim.x, ...  The shared-memory
// ring of operand stages runs on across tiles, and the accumulator is double-buffered in tensor
// memory so the epilogue of one tile overlaps the loads and MMAs of the next.
// GPW: 16-column groups an epilogue warp may own: 4 (tiles up to 128 channels wide, two CTAs per SM) or
// 8 (tiles up to 256 wide: an MMA of N = 256 lasts twice as long for the same A operand, so a stage
// carries twice the tensor work per byte fetched and per instruction of the issuing thread; both
// accumulator buffers together fill the tensor memory, hence one CTA per SM).
template <int EPI, int RELU = 2, int RSTG = 0, int GPW = kGroupsPerWarp>
__global__ void __launch_bounds__(kIgemmThreads, (GPW > kGroupsPerWarp || EpiTraits<EPI>::np) ? 1 : 2)
igemm_i8_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                const __grid_constant__ CUtensorMap tmap_y, const __grid_constant__ CUtensorMap tmap_r,
                const IgemmParams prm, const EpilogueParams ep, const int4* __restrict__ chan_table,
                const int8_t* __restrict__ res, void* __restrict__ y, int* status, unsigned int wait_limit) {
  extern __shared__ uint8_t smem_raw[];
  // operand stages need 1024-byte alignment (swizzle atom); the launch reserves the slack
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~static_cast<uintptr_t>(1023));
  // ring stages (activations + weights, or activations alone), then the resident weight tile if any
  const uint32_t stage_bytes = prm.a_stage_bytes + (prm.b_resident ? 0u : prm.b_stage_bytes);
  const int num_kb_all = prm.R * prm.S * prm.nchunks;
  const uint32_t b_res_off = static_cast<uint32_t>(prm.stages) * stage_bytes;
  uint8_t* out_stage = tiles + b_res_off + (prm.b_resident ? static_cast<uint32_t>(num_kb_all) * prm.b_stage_bytes : 0u);   // staged output tiles
  IgemmShared* sh = reinterpret_cast<IgemmShared*>(out_stage + static_cast<uint32_t>(prm.out_stage_bufs) * prm.out_stage_bytes +
                                                   prm.gen_stage_bytes);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  constexpr bool kPool = RSTG == 2;              // 2 x 2 max-pool taken in the epilogue
  constexpr bool kSplit = RSTG == 4;             // this CTA's cluster shares one tile's contraction
  constexpr bool kDw = RSTG == 5;                // depthwise
  const int b_row = kDw ? 32 : prm.BKC;          // bytes of a weight row per stage and tap
  constexpr bool kHint = GPW > kGroupsPerWarp;   // one CTA per SM on long stages: waits use the suspend hint
  const int num_kb = prm.R * prm.S * prm.nchunks;
  const int total_tiles = prm.tiles_q * prm.tiles_p * prm.tiles_n * prm.tiles_k;
  // this CTA's first tile, and its part of a tile's stages (a split kernel has one tile per cluster)
  const int ks_rank = kSplit ? static_cast<int>(ptx::cluster_ctarank()) : 0;
  const int first_tile = kSplit ? static_cast<int>(blockIdx.x) / prm.ksplit : static_cast<int>(blockIdx.x);
  const int kb_begin = kSplit ? num_kb * ks_rank / prm.ksplit : 0;
  const int kb_end = kSplit ? num_kb * (ks_rank + 1) / prm.ksplit : num_kb;

  if (threadIdx.x == 0) {
    for (int s = 0; s < prm.stages; ++s) {
      ptx::mbar_init(ptx::smem_u32(&sh->full[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&sh->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(ptx::smem_u32(&sh->acc_full[b]), 1);
      ptx::mbar_init(ptx::smem_u32(&sh->acc_empty[b]), kEpilogueWarps);   // one arrival per epilogue warp
    }
    for (int b = 0; b < 3; ++b) ptx::mbar_init(ptx::smem_u32(&sh->res_full[b]), 1);
    ptx::mbar_init(ptx::smem_u32(&sh->b_full), 1);
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tmap(&tmap_a);
    ptx::prefetch_tmap(&tmap_b);
    if (EpiTraits<EPI>::fast && prm.out_stage_bytes) ptx::prefetch_tmap(&tmap_y);
    if (EpiTraits<EPI>::res && RSTG == 1) ptx::prefetch_tmap(&tmap_r);
  }
  if (warp == 1) {
    ptx::tmem_alloc(ptx::smem_u32(&sh->tmem_base), static_cast<uint32_t>(prm.acc_bufs * prm.tmem_cols));
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  if (kSplit) ptx::cluster_sync_all();           // the cluster's CTAs all run from here on: their shared memory may be written
  const uint32_t tmem_base = sh->tmem_base;
  // Everything above touched no tensor of another kernel, so under programmatic dependent launch
  // it overlaps the tail of the previous kernel in the stream.  The next kernel may start its own
  // set-up right away; each role of this one waits for the previous kernel (griddepcontrol.wait)
  // immediately before its first access to a tensor that kernel may have written, with all the
  // arithmetic leading up to that access already done.
  ptx::grid_launch_dependents();

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    // The CTA's loads form one sequence of stages (tile, filter row r, tap sx, channel chunk ci); stage g
    // goes to ring slot g % stages.  The first pass over the ring is issued by `stages` lanes side by
    // side, lane l taking stage l: the address arithmetic of a stage costs one thread some hundred cycles
    // of dependent instructions, so a single thread would spend longer issuing the nine small stages of
    // a short layer than the tensor core spends on them, and after the wait on the previous kernel the
    // whole first pass goes out at once.  From the second pass on a stage can only follow the MMAs that
    // free its slot, in order: one lane walks the sequence (lanes polling different barriers in one warp
    // only slow each other down).
    const uint32_t tiles_addr = ptx::smem_u32(tiles);
    const bool has_tiles = first_tile < total_tiles;
    // (a resident weight tile is fetched by the MMA warp, which has nothing else to do at this point: the
    // activation loads below then go out without waiting behind a dozen weight copies)
    // One stage: arm the slot's barrier, load the weight chunk(s) unless resident, then the activation box.
    // `first` marks a lane's first activation load: the previous kernel's results are needed from there on
    // (not for the weights), so the wait on it sits right in front of that load.
    // `doit`: this thread issues (the arithmetic may run on all lanes with warp-uniform values, see below).
    auto issue = [&](int slot, const TileCoord& tc, int r, int sx, int ci, bool first, bool doit) {
      const uint32_t full = ptx::smem_u32(&sh->full[slot]);
      const uint32_t a_dst = tiles_addr + static_cast<uint32_t>(slot) * stage_bytes;
      const int w0 = tc.q0 * prm.stride_w - prm.pad_w + sx, h0 = tc.p0 * prm.stride_h - prm.pad_h + r;
      int a_ci = ci;                                         // channel chunk of the activations
      if (EpiTraits<EPI>::np) {
        int in_plane;
        const int product = prm.fd_np_cpp.divmod(ci, &in_plane);
        a_ci = prm.np_a[product] * prm.np_cpp + in_plane;
      }
      const int a_c = kDw ? tc.k0 : a_ci * prm.BKC;
      if (doit) {
        ptx::mbar_expect_tx(full, prm.tx_bytes);
        if (!prm.b_resident) {
          if (prm.halo_s) {
            for (int hs = 0; hs < prm.halo_s; ++hs)
              ptx::tma_load_2d(a_dst + prm.a_stage_bytes + static_cast<uint32_t>(hs) * prm.b_chunk_bytes, &tmap_b, full,
                               ((r * prm.halo_s + hs) * prm.nchunks + ci) * b_row, tc.k0);
          } else {
            ptx::tma_load_2d(a_dst + prm.a_stage_bytes, &tmap_b, full, ((r * prm.S + sx) * prm.nchunks + ci) * b_row, tc.k0);
          }
        }
        if (first) ptx::grid_dependency_wait();
        ptx::tma_load_4d(a_dst, &tmap_a, full, a_c, w0, h0, tc.n0);
        if (prm.tap_boxes)
          for (int hs = 1; hs < prm.halo_s; ++hs)           // the filter row's other taps, each a box of its own
            ptx::tma_load_4d(a_dst + static_cast<uint32_t>(hs) * prm.a_tap_bytes, &tmap_a, full, a_c, w0 + hs, h0, tc.n0);
      }
    };
    // stages this CTA issues in all, and how many of them make up the first pass
    const int my_tiles = kSplit ? 1 : has_tiles ? prm.fd_grid.div(total_tiles - first_tile + static_cast<int>(gridDim.x) - 1) : 0;
    const long long total_stages = kSplit ? kb_end - kb_begin : static_cast<long long>(my_tiles) * num_kb;
    const int first_pass = static_cast<int>(total_stages < prm.stages ? total_stages : prm.stages);
    {
      // position `lane` of the sequence (lane `first_pass` of lane 0's walk below): mixed-radix digits
      const int pos = lane < first_pass ? lane : first_pass;
      int ci, sx;
      int t0 = prm.fd_nchunks.divmod(kb_begin + pos, &ci);
      int r = prm.fd_S.divmod(t0, &sx);
      int tile = first_tile;
      TileWalker walk;
      walk.init(prm, first_tile);
      while (r >= prm.R && tile < total_tiles) { r -= prm.R; tile += gridDim.x; walk.next(prm); }
      issue(lane < first_pass ? lane : 0, walk.coord(prm), r, sx, ci, true, lane < first_pass);
      __syncwarp();
      {
        // The rest of the sequence, in order, from position first_pass.  The whole warp runs this loop with
        // warp-uniform values (addresses and coordinates then live in uniform registers, which is where the
        // copy instructions take their operands from); lane 0 alone issues.
        const bool leader = lane == 0;
        t0 = prm.fd_nchunks.divmod(kb_begin + first_pass, &ci);
        r = prm.fd_S.divmod(t0, &sx);
        tile = first_tile;
        walk.init(prm, first_tile);
        while (r >= prm.R && tile < total_tiles) { r -= prm.R; tile += gridDim.x; walk.next(prm); }
        int stage = 0;
        uint32_t phase = 1;                                  // second pass over the ring
        long long issued = first_pass;
        bool ok = true;
        TileCoord tc = walk.coord(prm);
        while (tile < total_tiles && (!kSplit || issued < total_stages)) {
          if (!(kHint ? ptx::mbar_try_wait_hint : ptx::mbar_try_wait)(ptx::smem_u32(&sh->empty[stage]), phase ^ 1u)) {
            ok = wait_bounded<32, kHint>(ptx::smem_u32(&sh->empty[stage]), phase ^ 1u, wait_limit, sh, status);
            if (!ok) break;
          }
          issue(stage, tc, r, sx, ci, false, leader);
          ++issued;
          if (++ci == prm.nchunks) {
            ci = 0;
            if (++sx == prm.S) {
              sx = 0;
              if (++r == prm.R) { r = 0; tile += gridDim.x; walk.next(prm); tc = walk.coord(prm); }
            }
          }
          if (++stage == prm.stages) { stage = 0; phase ^= 1u; }
        }
        __syncwarp();
        if (!leader) issued = 0;                             // (lane 0 alone waits below)
        // Whatever happened to the other roles, this CTA's shared memory must outlive every copy issued
        // into it: wait (bounded, but not by the caller's limit) for the resident weight tile and for the
        // last pass over the ring.  In a normal run all of this has long landed and each probe succeeds.
        if (leader && prm.b_resident && has_tiles) {
          for (unsigned int w = 0; w < kDrainPolls; ++w)
            if (ptx::mbar_try_wait(ptx::smem_u32(&sh->b_full), 0u)) break;
        }
        const long long first = issued > prm.stages ? issued - prm.stages : 0;
        int st_i = static_cast<int>(first % prm.stages);
        uint32_t par = static_cast<uint32_t>(first / prm.stages) & 1u;
        for (long long i = first; i < issued; ++i) {
          const uint32_t bar = ptx::smem_u32(&sh->full[st_i]);
          for (unsigned int w = 0; w < kDrainPolls; ++w)
            if (ptx::mbar_try_wait(bar, par)) break;
          if (++st_i == prm.stages) { st_i = 0; par ^= 1u; }
        }
        // a CTA always waits for the previous kernel before it retires, so that "this kernel is complete"
        // implies "every kernel before it is complete" for the kernel after it
        if (leader) ptx::grid_dependency_wait();
      }
    }
    if (kSplit) { __syncwarp(); ptx::cluster_sync_all(); }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // One elected lane feeds the tensor core, and the tensor core queues next to nothing: whatever
    // happens between two MMAs is time the unit idles (a 128 x 128 x 32 MMA lasts 64 cycles).  So
    //  - the whole warp runs the loop with warp-uniform values, which lets descriptors and
    //    addresses live in uniform registers (the MMA takes its operands from those) instead of
    //    being moved there before every instruction; only the MMA / commit are predicated;
    //  - descriptors and ring position advance by additions;
    //  - a stage is awaited with one probe of its barrier (the bounded, abort-aware loop only on a miss)
    //    and no warp votes: a stage costs the issuing thread a few hundred cycles of dependent
    //    instructions, which is what bounds layers whose stages carry little tensor work.
    {
      const bool leader = ptx::elect_one();
      const uint32_t idesc = make_idesc_i8(kDw ? 32 : prm.BN);
      const int mma_per_stage = prm.BKC / 32;
      const uint32_t tiles_addr = ptx::smem_u32(tiles);
      const bool bres = prm.b_resident != 0;
      if (leader && bres && first_tile < total_tiles) {
        // the whole weight tile of this CTA's channel tile, once; weights never depend on the previous kernel
        int kt0;
        prm.fd_tiles_k.divmod(first_tile, &kt0);
        const int k0 = kt0 * prm.BN;
        const uint32_t bar = ptx::smem_u32(&sh->b_full);
        ptx::mbar_expect_tx(bar, prm.b_res_tx_bytes);
        // (halo form, one chunk per tap: a stage's three weight chunks are the columns 3 kb, 3 kb + 1, 3 kb + 2)
        const int per_stage = prm.halo_s ? prm.halo_s : 1;
        for (int kb = 0; kb < num_kb; ++kb)
          for (int hs = 0; hs < per_stage; ++hs)
            ptx::tma_load_2d(tiles_addr + b_res_off + static_cast<uint32_t>(kb) * prm.b_stage_bytes +
                                 static_cast<uint32_t>(hs) * prm.b_chunk_bytes,
                             &tmap_b, bar, (kb * per_stage + hs) * b_row, k0);
      }
      __syncwarp();
      const uint64_t a_desc0 = make_kmajor_desc(tiles_addr, prm.BKC);
      const uint64_t b_desc0 = make_kmajor_desc(tiles_addr + (bres ? b_res_off : prm.a_stage_bytes), b_row);
      const uint64_t desc_step = stage_bytes >> 4;          // start-address field counts 16-byte units
      // resident weights: chunk kb of the tile sits at its own place, whatever the ring position
      const uint64_t b_step = bres ? (prm.b_stage_bytes >> 4) : desc_step;
      uint64_t a_desc = a_desc0, b_desc = b_desc0;
      // taps of one stage: one pixel row further on in the same box (halo form) or the next box (grouped taps)
      const uint64_t halo_row = static_cast<uint64_t>(prm.tap_boxes ? prm.a_tap_bytes : static_cast<uint32_t>(prm.BKC)) >> 4;
      const uint64_t halo_bchunk = prm.b_chunk_bytes >> 4;
      // patch form: from a filter row's last tap to the next row's first one
      const uint64_t halo_next_row = static_cast<uint64_t>((prm.tq - prm.halo_w + 1) * prm.BKC) >> 4;
      const uint32_t full0 = ptx::smem_u32(&sh->full[0]), empty0 = ptx::smem_u32(&sh->empty[0]);
      // One tap's chunk: 32 bytes along K inside the swizzle span = +2 in the descriptor's 16-byte address units.
      // (depthwise: 32 channels each, against their own 1 KB of weights, into their own columns)
      auto tap_mmas = [&](uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
        constexpr uint32_t dn = kDw ? 32u : 0u;
        constexpr uint64_t bk = kDw ? 64u : 2u;
        const uint32_t later = kDw ? acc : 1u;
        ptx::mma_i8(d, a, b, idesc, acc);
        if (mma_per_stage > 1) ptx::mma_i8(d + dn, a + 2u, b + bk, idesc, later);
        if (mma_per_stage > 2) {
          ptx::mma_i8(d + 2u * dn, a + 4u, b + 2u * bk, idesc, later);
          ptx::mma_i8(d + 3u * dn, a + 6u, b + 3u * bk, idesc, later);
        }
      };
      int stage = 0, it = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = first_tile; tile < total_tiles && ok; tile += gridDim.x, ++it) {
        const int buf = (EpiTraits<EPI>::np && prm.acc_bufs == 1) ? 0 : it & 1;
        const uint32_t use = static_cast<uint32_t>((EpiTraits<EPI>::np && prm.acc_bufs == 1) ? it : it >> 1);
        // the epilogue must have drained this accumulator buffer (two tiles ago)
        ok = wait_bounded<0, kHint>(ptx::smem_u32(&sh->acc_empty[buf]), (use & 1u) ^ 1u, wait_limit, sh, status);
        if (!ok) break;
        ptx::tc_fence_after();
        uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * prm.tmem_cols);
        const uint32_t d_tmem0 = d_tmem;
        int np_chunk = 0, np_product = 0;                    // EPI_NP: position inside the tap's chunks
        uint32_t accumulate = 0;
        if (bres) {
          if (it == 0) {
            ok = wait_bounded<0, kHint>(ptx::smem_u32(&sh->b_full), 0u, wait_limit, sh, status);
            if (!ok) break;
          }
          b_desc = b_desc0;
        }
        for (int kb = kb_begin; kb < kb_end; ++kb) {
          // all lanes probe the same barrier with the same instruction, so they agree without a vote
          if (!(kHint ? ptx::mbar_try_wait_hint : ptx::mbar_try_wait)(full0 + 8u * stage, phase)) {
            ok = wait_bounded<0, kHint>(full0 + 8u * stage, phase, wait_limit, sh, status);
            if (!ok) break;
          }
          ptx::tc_fence_after();
          if (leader) {
            tap_mmas(d_tmem, a_desc, b_desc, accumulate);
            // halo form: the other horizontal taps are the same activation rows one pixel (one row of BKC
            // bytes) further on -- start address advanced by a row, the descriptor's base offset telling the
            // swizzle phase of the new first row -- against the next weight chunk of the stage
            uint64_t ah = a_desc, bh = b_desc;
            for (int hs = 1, hw = 1; hs < prm.halo_s; ++hs, ++hw) {
              if (hw == prm.halo_w) { ah += halo_next_row; hw = 0; }
              else ah += halo_row;
              bh += halo_bchunk;
              tap_mmas(d_tmem, ah, bh, 1u);
            }
            ptx::mma_commit(empty0 + 8u * stage);             // stage free once these MMAs retire
          }
          accumulate = 1;
          if (EpiTraits<EPI>::np) {
            // the next product starts its own columns, cleared by its first chunk of the first tap
            if (++np_chunk == prm.np_cpp) {
              np_chunk = 0;
              if (++np_product == prm.np_products) np_product = 0;
              d_tmem = d_tmem0 + static_cast<uint32_t>(np_product * prm.BN);
              accumulate = kb + 1 < prm.nchunks ? 0u : 1u;
            }
          }
          if (++stage == prm.stages) { stage = 0; phase ^= 1u; a_desc = a_desc0; if (!bres) b_desc = b_desc0; }
          else { a_desc += desc_step; if (!bres) b_desc += b_step; }
          if (bres) b_desc += b_step;
        }
        if (ok && leader) ptx::mma_commit(ptx::smem_u32(&sh->acc_full[buf]));
        if (kSplit) break;                                   // one tile per cluster
      }
      __syncwarp();
    }
    if (kSplit) ptx::cluster_sync_all();
  } else {
    // ------------------------------------------------------------------ epilogue
    // Eight warps: warp w reads the TMEM lane quadrant w % 4 (rows 32 * (w % 4) ...) and one half of
    // the tile's 16-column groups, so every scheduler has several epilogue warps to switch between.
    const int ew = warp - 2;
    const int quad = warp & 3;
    const int row = quad * 32 + lane;                        // tile row = accumulator lane
    int q_i, p_i;
    const int n_i = prm.fd_tp.divmod(prm.fd_tq.divmod(row, &q_i), &p_i);
    const int etid = threadIdx.x - 64;                       // 0 .. 255 among the epilogue threads
    const int groups16 = prm.BN / 16;
    const int g_split = (groups16 + 1) / 2;
    const int g_begin = (ew < 4) ? 0 : g_split;
    const int g_end = (ew < 4) ? g_split : groups16;
    int it = 0;
    bool ok = true;
    const int kpad = prm.tiles_k * prm.BN;
    const bool cst_all = static_cast<uint32_t>(kpad) * EpiTraits<EPI>::cst_bytes <= kCstBytes;
    if (cst_all) {
      for (int i = etid; i < kpad; i += kEpilogueWarps * 32) {
        stage_constant<EPI>(sh->cst, i, chan_table + i);
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kEpilogueWarps * 32) : "memory");
    }
    uint8_t* gen_stage = out_stage + ew * kGenWarpBytes;     // (general epilogues)
    float gen_max = 0.0f;
    TileWalker walk;
    walk.init(prm, first_tile);
    // the residual may come from the previous kernel (the constants above never do)
    ptx::grid_dependency_wait();
    const uint32_t cst_addr = ptx::smem_u32(&sh->cst);
    // Residual tiles come by TMA into the staged buffers, one tile ahead of the arithmetic (three buffers:
    // the tile being stored, the tile being computed, the residual of the next).  The thread that issues
    // the stores also issues these loads: it alone knows when a buffer's store has finished reading.
    constexpr bool res_staged = EpiTraits<EPI>::res && EpiTraits<EPI>::fast && RSTG == 1;   // the planner then provides three staged tiles
    // (no staged tiles of their own: the CTA's one tile is staged in the ring)
    const uint32_t stage0 = ptx::smem_u32(prm.out_stage_bufs == 0 ? tiles : out_stage);
    TileWalker walk_next = walk;
    int sbuf = 0;                              // staged buffer of the current tile
    uint32_t res_pending = 0;                  // bit i: a residual load into buffer i has not been consumed yet
    uint32_t res_phase = 0;                    // bit i: parity to wait for on res_full[i]
    if (res_staged && etid == 0 && first_tile < total_tiles) {
      const TileCoord t0 = walk.coord(prm);
      ptx::mbar_expect_tx(ptx::smem_u32(&sh->res_full[0]), prm.res_tx_bytes);
      ptx::tma_load_4d(stage0, &tmap_r, ptx::smem_u32(&sh->res_full[0]), t0.k0, t0.q0, t0.p0, t0.n0);
      res_pending = 1u;
    }
    // Lean form of a tile's epilogue, for staged tiles: no pixel coordinates (the TMA store clips), no predicates beyond
    // the warp's number of column groups, the swizzled position of this thread's 16-byte chunks from per-thread constants.
    // (Chunk c of the staged row r sits at c ^ (r & 7) in a 128-byte row, at c ^ ((r >> 1) & 3) in a 64-byte row: the
    // 16-byte chunk index XOR bits 7.. of the byte offset, masked to the row's chunks; tiles of other widths are not
    // swizzled.)  A residual is staged too, or comes in registers.
    constexpr bool kLeanOk = EpiTraits<EPI>::fast && !kPool && !kSplit && GPW == kGroupsPerWarp;
    const bool lean = kLeanOk && prm.out_stage_bytes != 0;
    // The integer epilogue with a residual and per-channel constants has no registers to spare: with both forms of the tile in
    // the kernel it spilled 128 bytes (276 read back; one form: 60 and 88), so this form also serves its direct stores.  us, 3 x
    // 3 with residual: 62 x 31 x 17 x 224 -> 576 58.3 -> 54.7, 35 x 42 x 29 x 160 -> 880 stride 2 33.7 -> 29.3, 2 x 38 x 33 x 240 -> 16 5.6 -> 4.75.
    constexpr bool kOneForm = kLeanOk && EPI == EPI_FAST_I8_RES;
    const int lean_groups = g_end - g_begin;
    const uint32_t lean_col0 = static_cast<uint32_t>(g_begin) * 16u;
    uint32_t lean_off[4];
    {
      const uint32_t row_off = static_cast<uint32_t>(row) * static_cast<uint32_t>(prm.BN);
      const uint32_t swz = ((row_off >> 7) & prm.out_swz_mask) << 4;
#pragma unroll
      for (int i = 0; i < 4; ++i) lean_off[i] = row_off + ((lean_col0 + 16u * i) ^ swz);
    }
    // A warp whose wait expired must not be missing from a later barrier of the eight epilogue warps:
    // it carries `ok == false` to the next barrier, which doubles as a vote, and all leave together.
    for (int tile = first_tile; tile < total_tiles; tile += gridDim.x, ++it, walk.next(prm)) {
      const TileCoord tc = walk.coord(prm);
      const int buf = (EpiTraits<EPI>::np && prm.acc_bufs == 1) ? 0 : it & 1;
      const uint32_t use = static_cast<uint32_t>((EpiTraits<EPI>::np && prm.acc_bufs == 1) ? it : it >> 1);
      // Slot of the per-tile channel constants: by the tile's parity even where there is one accumulator buffer.  A warp that
      // is done with a tile stages the next one's constants while slower warps still read theirs; past the vote behind the
      // staging every warp is done with the tile before, whose slot the tile after may then overwrite.
      const int cst_slot = it & 1;
      if (res_staged) {
        walk_next.next(prm);
        if (etid == 0 && tile + static_cast<int>(gridDim.x) < total_tiles) {
          // the next tile's buffer was last read by the store issued two tiles ago
          ptx::bulk_wait_read_but_one();
          const int nb = sbuf == 2 ? 0 : sbuf + 1;
          const TileCoord tn = walk_next.coord(prm);
          ptx::mbar_expect_tx(ptx::smem_u32(&sh->res_full[nb]), prm.res_tx_bytes);
          ptx::tma_load_4d(stage0 + static_cast<uint32_t>(nb) * prm.out_stage_bytes, &tmap_r,
                           ptx::smem_u32(&sh->res_full[nb]), tn.k0, tn.q0, tn.p0, tn.n0);
          res_pending |= 1u << nb;
        }
      }
      if (!cst_all) {
        // stage this tile's channel constants, then meet the other epilogue warps
        for (int i = etid; i < prm.BN; i += kEpilogueWarps * 32) {
          stage_constant<EPI>(sh->cst, cst_slot * 256 + i, chan_table + tc.k0 + i);
        }
        if (epilogue_vote(!ok)) { ok = false; break; }
      }
      bool row_ok = true;
      size_t pix = 0, pooled_pix = 0;
      if (!lean || (EpiTraits<EPI>::res && !res_staged)) {
        const int q = tc.q0 + q_i, p = tc.p0 + p_i, n = tc.n0 + n_i;
        row_ok = (n_i < prm.tn) && q_i < prm.q_step && q < prm.Q && p < prm.P && n < prm.Nimg;
        pix = (static_cast<size_t>(n) * prm.P + p) * prm.Q + q;
        // pooled output pixel of this row's 2 x 2 window (extents P / 2 x Q / 2)
        if (kPool) pooled_pix = (static_cast<size_t>(n) * (prm.P >> 1) + (p >> 1)) * (prm.Q >> 1) + (q >> 1);
      }
      // the residual does not depend on the accumulator: fetch it while the MMAs still run
      uint4 rres[kGroupsPerWarp];                            // (tiles wider than 128 carry no register-fetched residual)
#pragma unroll
      for (int i = 0; i < kGroupsPerWarp; ++i) {
        rres[i] = make_uint4(0u, 0u, 0u, 0u);
        if (EpiTraits<EPI>::res && !res_staged) {
          const int g = kSplit ? ((ew >> 2) + 2 * i) * prm.ksplit + ks_rank : g_begin + i;   // (split: this warp's own groups)
          const int k = tc.k0 + g * 16;
          if (row_ok && g < (kSplit ? groups16 : g_end) && k < prm.K)
            rres[i] = __ldg(reinterpret_cast<const uint4*>(res + pix * prm.K + k));
        }
      }
      // general epilogues: this warp's columns of the tile, and its residual rows by way of the staging rows
      const int gen_k0 = tc.k0 + g_begin * 16;
      const int gen_cols = max(0, min((g_end - g_begin) * 16, prm.K - gen_k0));
      // (int8 results overwrite it in place, group by group; words have rows of their own behind it)
      const bool gen_res = !EpiTraits<EPI>::fast && !EpiTraits<EPI>::np && res != nullptr;
      uint8_t* gen_out = (EPI == EPI_I32 || EPI == EPI_F32) && gen_res ? gen_stage + kEpilogueWarps * kGenWarpBytes : gen_stage;
      int gen_m = 0;
      if (gen_res) {
        int8_t* base = const_cast<int8_t*>(res) + gen_k0;
        const long long off = static_cast<long long>(pix) * prm.K;
        gen_m = static_cast<int>(reinterpret_cast<uintptr_t>(base + off) & 3u);
        __syncwarp();
        gen_copy<false>(prm.gen_vec_res, gen_stage, base, off, row_ok, gen_cols, lane);
        __syncwarp();
      }
      ok = wait_bounded<64, kHint>(ptx::smem_u32(&sh->acc_full[buf]), use & 1u, wait_limit, sh, status);
      if (res_staged && ok) {
        ok = wait_bounded<32, kHint>(ptx::smem_u32(&sh->res_full[sbuf]), (res_phase >> sbuf) & 1u, wait_limit, sh, status);
        if (ok) res_pending &= ~(1u << sbuf);
        res_phase ^= 1u << sbuf;
      }
      ok = __all_sync(0xffffffffu, ok);
      if constexpr (kSplit) {
        const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
        const uint32_t part = ptx::smem_u32(out_stage);
        const int ks = prm.ksplit;
        const uint32_t slot_bytes = 4u * 128u * 16u, row16 = static_cast<uint32_t>(row) * 16u;
        if (ok) {
          ptx::tc_fence_after();
          for (int g = g_begin; g < g_end; ++g) {
            const int owner = g % ks;
            if (owner == ks_rank || tc.k0 + g * 16 >= prm.K) continue;
            uint32_t acc[16];
            ptx::tmem_ld_32x16(t_addr + g * 16, acc);
            ptx::tmem_ld_wait();
            const int sender = ks_rank < owner ? ks_rank : ks_rank - 1;
            const uint32_t dst = ptx::map_to_cta(part, static_cast<uint32_t>(owner)) +
                                 static_cast<uint32_t>((g / ks) * (ks - 1) + sender) * slot_bytes + row16;
#pragma unroll
            for (int c = 0; c < 4; ++c)
              ptx::st_cluster_uint4(dst + static_cast<uint32_t>(c) * 2048u, acc[4 * c], acc[4 * c + 1], acc[4 * c + 2], acc[4 * c + 3]);
          }
        }
        __syncwarp();
        ptx::cluster_sync_all();                             // every sender's groups are here
        if (ok) {
          const uint32_t chan = cst_addr + static_cast<uint32_t>(cst_all ? tc.k0 : 0) * EpiTraits<EPI>::cst_bytes;
#pragma unroll
          for (int i = 0; i < kGroupsPerWarp; ++i) {
            const int own = (ew >> 2) + 2 * i, g = own * ks + ks_rank;
            if (g < groups16 && tc.k0 + g * 16 < prm.K) {
              uint32_t acc[16];
              ptx::tmem_ld_32x16(t_addr + g * 16, acc);
              ptx::tmem_ld_wait();
              for (int sender = 0; sender < ks - 1; ++sender) {
                const uint32_t src = part + static_cast<uint32_t>(own * (ks - 1) + sender) * slot_bytes + row16;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  const int4 v = lds_int4(src + static_cast<uint32_t>(c) * 2048u);
                  acc[4 * c] += v.x; acc[4 * c + 1] += v.y; acc[4 * c + 2] += v.z; acc[4 * c + 3] += v.w;
                }
              }
              if (row_ok) epilogue_16<EPI, RELU>(acc, chan, g * 16, tc.k0 + g * 16, pix, prm, ep, rres[i], y);
            }
          }
        }
        break;
      }
      const bool staged = EpiTraits<EPI>::fast && prm.out_stage_bytes != 0;
      if (!ok && !staged) {
        if (cst_all) break;          // no barrier ahead: this warp may leave by itself
        continue;                    // per-tile constants: meet the others at the next tile's barrier and vote
      }
      // staged tile of this iteration: this thread's row starts at row * BN bytes
      const uint32_t stage_base = stage0 + static_cast<uint32_t>(res_staged ? sbuf : buf) * prm.out_stage_bytes;
      if (ok) {
        ptx::tc_fence_after();
        const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) +
                                static_cast<uint32_t>(buf * prm.tmem_cols);
        // shared-memory address of this tile's first channel constant (16 bytes per channel, or 4 when
        // only the biases differ)
        const uint32_t chan = cst_addr + static_cast<uint32_t>(cst_all ? tc.k0 : cst_slot * 256) * EpiTraits<EPI>::cst_bytes;
        // This warp's 16-column groups, up to kGroupsPerWarp of them.  Tensor-memory loads run one
        // group ahead of the arithmetic; after the warp's last load the accumulator buffer goes back
        // to the MMA warp.
        auto release = [&]() {
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh->acc_empty[buf]));
        };
        uint32_t acc_a[16], acc_b[16];
        // general epilogues: group i of this warp; words leave group by group (64 bytes a row), bytes after the last
        [[maybe_unused]] auto gen_group = [&](const uint32_t (&acc)[16], int i) {
          if (i * 16 >= gen_cols) return;
          const uint32_t st_row = ptx::smem_u32(gen_out) + static_cast<uint32_t>(lane * kGenPitch);
          const uint4 r16 = gen_res ? gen_row_words(gen_stage + lane * kGenPitch, i, gen_m) : make_uint4(0u, 0u, 0u, 0u);
          const int ncols = gen_cols - i * 16;
          const uint32_t cst_g = chan + static_cast<uint32_t>(g_begin + i) * 16u * EpiTraits<EPI>::cst_bytes;
          const uint32_t at = st_row + (EpiTraits<EPI>::bytes ? static_cast<uint32_t>(i * 16) : 0u);
          if constexpr (EPI == EPI_I8) {
            if (!prm.gen_simple) general_int8_16<false, false>(acc, cst_g, r16, ep, at);
            else if (ep.rounding == 0) general_int8_16<true, true>(acc, cst_g, r16, ep, at);
            else general_int8_16<true, false>(acc, cst_g, r16, ep, at);
          } else if constexpr (EpiTraits<EPI>::gen) gen_flt_16<EPI>(acc, cst_g, r16, prm, ep, at);
          else general_16<EPI>(acc, cst_g, r16, ncols, row_ok, prm, ep, at, &gen_max);
          if (EPI == EPI_I32 || EPI == EPI_F32) {
            __syncwarp();
            gen_copy<true>(prm.gen_vec_y, gen_out, static_cast<int8_t*>(y) + 4ll * (prm.out_c_offset + gen_k0 + i * 16),
                           4ll * static_cast<long long>(pix) * prm.out_c_pitch, row_ok, 4 * min(16, ncols), lane);
            __syncwarp();
          }
        };
        if constexpr (EPI == EPI_NP3) {
          const Np3Encode f = {static_cast<uint32_t>(127 + prm.np_p) << 23, static_cast<uint32_t>(23 - prm.np_p) << 23,
                               (static_cast<uint32_t>(23 - prm.np_p) << 23) + (static_cast<uint32_t>(127 + prm.np_p) << prm.np_p),
                               (1u << prm.np_low) - 1u, prm.np_low, prm.np_p, prm.np_n - 1, prm.np_top};
          const uint32_t t0 = t_addr + static_cast<uint32_t>(g_begin) * 16u, bn = static_cast<uint32_t>(prm.BN);
          uint32_t acc_c[16];
          for (int i = 0; i * 16 < gen_cols; ++i) {
            ptx::tmem_ld_32x16(t0 + 16u * i, acc_a);
            ptx::tmem_ld_32x16(t0 + bn + 16u * i, acc_b);
            ptx::tmem_ld_32x16(t0 + 2u * bn + 16u * i, acc_c);
            ptx::tmem_ld_wait();
            if ((i + 1) * 16 >= gen_cols) release();
            const uint32_t cst_g = chan + (static_cast<uint32_t>(g_begin + i) * 16u) * EpiTraits<EPI>::cst_bytes;
            uint32_t wds[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              const int4 k01 = lds_int4(cst_g + static_cast<uint32_t>(g * 32)), k23 = lds_int4(cst_g + static_cast<uint32_t>(g * 32 + 16));
              const int32_t bias[4] = {k01.x, k01.y, k23.x, k23.y}, sc[4] = {k01.z, k01.w, k23.z, k23.w};
              uint32_t o[4];
#pragma unroll
              for (int b = 0; b < 4; ++b)
                o[b] = np3_encode<RELU == 1>(static_cast<int32_t>(acc_a[4 * g + b]), static_cast<int32_t>(acc_b[4 * g + b]),
                                             static_cast<int32_t>(acc_c[4 * g + b]), bias[b], __int_as_float(sc[b]), f);
              wds[g] = __byte_perm(__byte_perm(o[0], o[1], 0x0040), __byte_perm(o[2], o[3], 0x0040), 0x5410);
            }
            ptx::sts_uint4(ptx::smem_u32(gen_stage) + static_cast<uint32_t>(lane * kGenPitch + i * 16), wds[0], wds[1], wds[2], wds[3]);
          }
          if (gen_cols <= 0) release();
          __syncwarp();
          gen_copy<true>(prm.gen_vec_y, gen_stage, static_cast<int8_t*>(y) + prm.out_c_offset + gen_k0,
                         static_cast<long long>(pix) * prm.out_c_pitch, row_ok, gen_cols, lane);
          __syncwarp();
        } else if constexpr (EPI == EPI_NP) {
          const NpEncode f = {static_cast<uint32_t>(127 + prm.np_p) << 23, static_cast<uint32_t>(23 - prm.np_p) << 23,
                              (static_cast<uint32_t>(23 - prm.np_p) << 23) + (static_cast<uint32_t>(127 + prm.np_p) << prm.np_p),
                              prm.np_p, prm.np_n - 1, prm.np_top};
          for (int i = 0; i * 16 < gen_cols; ++i) {
            const uint32_t col = static_cast<uint32_t>(g_begin + i) * 16u;
            long long v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = lds_int4(chan + (col + j) * 16u).x;      // bias
            ptx::tmem_ld_32x16(t_addr + col, acc_a);
            for (int m = 0; m < prm.np_products; m += 2) {
              ptx::tmem_ld_wait();
              if (m + 1 < prm.np_products) ptx::tmem_ld_32x16(t_addr + static_cast<uint32_t>((m + 1) * prm.BN) + col, acc_b);
#pragma unroll
              for (int j = 0; j < 16; ++j) v[j] += static_cast<long long>(static_cast<int32_t>(acc_a[j])) * prm.np_coef[m];
              if (m + 1 < prm.np_products) {
                ptx::tmem_ld_wait();
                if (m + 2 < prm.np_products) ptx::tmem_ld_32x16(t_addr + static_cast<uint32_t>((m + 2) * prm.BN) + col, acc_a);
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] += static_cast<long long>(static_cast<int32_t>(acc_b[j])) * prm.np_coef[m + 1];
              }
            }
            if ((i + 1) * 16 >= gen_cols) release();
            uint32_t wds[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              uint32_t o[4];
#pragma unroll
              for (int b = 0; b < 4; ++b) {
                const long long w = v[g * 4 + b];
                const int s = lds_int4(chan + (col + g * 4 + b) * 16u).y;
                o[b] = np_encode(ep.relu && w < 0 ? 0ll : w, s, f);
              }
              wds[g] = __byte_perm(__byte_perm(o[0], o[1], 0x0040), __byte_perm(o[2], o[3], 0x0040), 0x5410);
            }
            ptx::sts_uint4(ptx::smem_u32(gen_stage) + static_cast<uint32_t>(lane * kGenPitch + i * 16), wds[0], wds[1], wds[2], wds[3]);
          }
          if (gen_cols <= 0) release();
          __syncwarp();
          gen_copy<true>(prm.gen_vec_y, gen_stage, static_cast<int8_t*>(y) + prm.out_c_offset + gen_k0,
                         static_cast<long long>(pix) * prm.out_c_pitch, row_ok, gen_cols, lane);
          __syncwarp();
        } else if (kLeanOk && (lean || kOneForm)) {
          // loads one group ahead of the arithmetic, as below, without the bookkeeping
          const uint32_t t0 = t_addr + lean_col0;
          const uint32_t c0 = chan + lean_col0 * EpiTraits<EPI>::cst_bytes;
          constexpr uint32_t kGroupCst = 16u * EpiTraits<EPI>::cst_bytes;
          auto group = [&](const uint32_t (&acc)[16], int i, const CstAhead<EPI>& ahead) {
            const uint32_t addr = stage_base + lean_off[i];
            uint32_t rw[4] = {0u, 0u, 0u, 0u}, wds[4];
            if (res_staged) {                                // the residual tile was brought there by TMA
              const int4 r4 = lds_int4(addr);
              rw[0] = r4.x; rw[1] = r4.y; rw[2] = r4.z; rw[3] = r4.w;
            } else if (EpiTraits<EPI>::res) {
              rw[0] = rres[i].x; rw[1] = rres[i].y; rw[2] = rres[i].z; rw[3] = rres[i].w;
            }
            convert_16<EPI, RELU>(acc, c0 + static_cast<uint32_t>(i) * kGroupCst, ahead, rw, ep, wds);
            const int k = tc.k0 + static_cast<int>(lean_col0) + 16 * i;
            if (!kOneForm || lean)
              ptx::sts_uint4(addr, wds[0], wds[1], wds[2], wds[3]);
            else if (row_ok && k < prm.K)
              *reinterpret_cast<uint4*>(static_cast<int8_t*>(y) + pix * prm.out_c_pitch + prm.out_c_offset + k) = make_uint4(wds[0], wds[1], wds[2], wds[3]);
          };
          // (a warp has up to four groups; one of the second four warps has none where the tile is 16 wide)
          if (lean_groups > 0) {
            ptx::tmem_ld_32x16(t0, acc_a);
            CstAhead<EPI> k0 = load_ahead<EPI>(c0, 0), k1 = k0;
            ptx::tmem_ld_wait();
            if (lean_groups > 1) {
              ptx::tmem_ld_32x16(t0 + 16, acc_b);
              k1 = load_ahead<EPI>(c0 + kGroupCst, 0);
              group(acc_a, 0, k0);
              ptx::tmem_ld_wait();
              if (lean_groups > 2) {
                ptx::tmem_ld_32x16(t0 + 32, acc_a);
                k0 = load_ahead<EPI>(c0 + 2 * kGroupCst, 0);
                group(acc_b, 1, k1);
                ptx::tmem_ld_wait();
                if (lean_groups > 3) {
                  ptx::tmem_ld_32x16(t0 + 48, acc_b);
                  k1 = load_ahead<EPI>(c0 + 3 * kGroupCst, 0);
                  group(acc_a, 2, k0);
                  ptx::tmem_ld_wait();
                  release();
                  group(acc_b, 3, k1);
                } else {
                  release();
                  group(acc_a, 2, k0);
                }
              } else {
                release();
                group(acc_b, 1, k1);
              }
            } else {
              release();
              group(acc_a, 0, k0);
            }
          } else {
            release();
          }
        } else {
        if (g_begin < g_end) {
          ptx::tmem_ld_32x16(t_addr + g_begin * 16, acc_a);
          ptx::tmem_ld_wait();
        }
#pragma unroll
        for (int i = 0; i < GPW; i += 2) {
          const int g0 = g_begin + i, g1 = g0 + 1, g2 = g0 + 2;
          if (g0 < g_end) {
            if (g1 < g_end) ptx::tmem_ld_32x16(t_addr + g1 * 16, acc_b); else release();
            if constexpr (kPool) {
              if (tc.k0 + g0 * 16 < prm.K)
                epilogue_pool_16<EPI, RELU>(acc_a, chan, g0 * 16, tc.k0 + g0 * 16, pooled_pix, row_ok, lane, prm.pool_bit, prm, ep, y);
            } else if constexpr (!EpiTraits<EPI>::fast) {
              gen_group(acc_a, i);
            } else if (row_ok && tc.k0 + g0 * 16 < prm.K)
              epilogue_16<EPI, RELU>(acc_a, chan, g0 * 16, tc.k0 + g0 * 16, pix, prm, ep, rres[i & (kGroupsPerWarp - 1)], y);
            if (g1 < g_end) {
              ptx::tmem_ld_wait();
              if (g2 < g_end && i + 2 < GPW) ptx::tmem_ld_32x16(t_addr + g2 * 16, acc_a); else release();
              if constexpr (kPool) {
                if (tc.k0 + g1 * 16 < prm.K)
                  epilogue_pool_16<EPI, RELU>(acc_b, chan, g1 * 16, tc.k0 + g1 * 16, pooled_pix, row_ok, lane, prm.pool_bit, prm, ep, y);
              } else if constexpr (!EpiTraits<EPI>::fast) {
                gen_group(acc_b, i + 1);
              } else if (row_ok && tc.k0 + g1 * 16 < prm.K)
                epilogue_16<EPI, RELU>(acc_b, chan, g1 * 16, tc.k0 + g1 * 16, pix, prm, ep, rres[(i + 1) & (kGroupsPerWarp - 1)], y);
              if (g2 < g_end && i + 2 < GPW) ptx::tmem_ld_wait();
            }
          }
        }
        if (g_begin >= g_end) release();                     // a warp without columns still hands back
        if (EpiTraits<EPI>::bytes) {
          __syncwarp();
          gen_copy<true>(prm.gen_vec_y, gen_stage, static_cast<int8_t*>(y) + prm.out_c_offset + gen_k0,
                         static_cast<long long>(pix) * prm.out_c_pitch, row_ok, gen_cols, lane);
          __syncwarp();
        }
        }
      }
      if (staged) {
        // The tile is complete in shared memory: one thread hands it to the TMA unit, which writes whole
        // rows (and clips what lies outside the tensor).  Before the barrier that thread makes sure the
        // previous tile's store has finished reading ITS buffer, which is the one the next tile fills.
        // The barrier also carries a vote: if any warp's wait expired, all eight leave together (a
        // warp must never be missing from a later barrier).
        if (etid == 0 && !res_staged) ptx::bulk_wait_read_all();
        ptx::fence_async_smem();
        if (epilogue_vote(!ok)) { ok = false; break; }
        if (etid == 0) {
          if (prm.store_rows) {
            for (int p = 0; p < prm.store_rows && tc.p0 + p < prm.P; ++p)
              ptx::tma_store_4d(&tmap_y, stage_base + static_cast<uint32_t>(p * prm.tq * prm.BN), tc.k0, tc.q0, tc.p0 + p, tc.n0);
          } else {
            ptx::tma_store_4d(&tmap_y, stage_base, tc.k0, tc.q0, tc.p0, tc.n0);
          }
          ptx::bulk_commit();
        }
        sbuf = sbuf == 2 ? 0 : sbuf + 1;
      }
    }
    if (EPI == EPI_MAX) {
      __syncwarp();
      flush_maxabs(gen_max, y);
    }
    if (EpiTraits<EPI>::fast && prm.out_stage_bytes && etid == 0) {
      // (read, not complete: the grid's completion covers the writes, and whoever depends on them waits for that)
      ptx::bulk_wait_read_all();
      // after an early exit residual tiles may still be on their way into this CTA's shared memory:
      // let them land (bounded) before the CTA retires
      if (res_staged) {
        for (int b = 0; b < 3; ++b)
          for (unsigned int w = 0; w < kDrainPolls && ((res_pending >> b) & 1u); ++w)
            if (ptx::mbar_try_wait(ptx::smem_u32(&sh->res_full[b]), (res_phase >> b) & 1u)) break;
      }
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, static_cast<uint32_t>(prm.acc_bufs * prm.tmem_cols));
  }
}

}  // namespace qc
