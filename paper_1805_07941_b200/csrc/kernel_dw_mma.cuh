// Depthwise 3x3 (Eq. 6 with g = C) on warp-level matrix instructions, rows staged by TMA.
//
// A warp owns 32 channels x 16 output pixels (two groups of 8 neighbouring ones) and walks down a strip of output rows.  One
// `mma.sync.m16n8k32` (int8, int32 sums) takes the 16 pixels as rows, 8 channels as columns, and along K the three taps of a
// filter row: k = (tap, channel), the weights on the diagonal channel == column.  So a filter row of 8 channels is one
// instruction whose A operand is nothing but 32-bit words of the staged row at shifted pixels -- no byte transposes, no windows --
// and every input row is read once for the (up to three) output rows in flight, whose sums start from bias + magic as the
// instruction's addend.
//
// K layout: a lane reads 8 bytes at channel 8 (j & 1) of a 16-channel chunk (j = lane % 4), at tap j / 2 for the lower half of
// K, at tap 2 for the upper one (lanes j > 1 meet zero weights there).  Its first word belongs to the 8 channels {0-3, 8-11}
// of the chunk, its second to {4-7, 12-15}; with columns 2 j, 2 j + 1 of both the pair of lanes (j, j ^ 1) holds 8 channels of
// both chunks, and one exchange leaves each lane 8 consecutive channels of a pixel.
//
// What it was made against: 128 x 32-byte operands per tcgen05.mma of N = 32 (54 cycles for 1/32 of useful products), and 17
// instructions an output in the dp4a form.  Here an output takes 12.1 (ncu, 64 x 56 x 56 x 128: issue slots 51 %, ALU pipe 28 %,
// matrix pipe 25 %, fixed latencies and long scoreboard among the stalls, 122 registers and so 16 warps an SM), and alone the
// kernel is no faster at large sizes (256 x 56 x 56 x 128 69 us, 71 on tcgen05, 74 with dp4a) and slower where narrow or short images
// leave its groups or strips partly empty (dw_tcgen05_wins, qconv_api.cu, chooses).  It is where launches follow one another: a
// third of the set-up, and short CTAs in place of a persistent grid whose two CTAs an SM finish 10 us apart.  MobileNet-v1 stack,
// batch 256: 818 -> 771 us; one image's layers 3.3-4.2 -> 2.8-3.2 us each.  Registers decide its speed: per-channel scales held in
// them instead of shared memory 782 us, a few more spilled 807-848.
//
// Every wait is bounded, its first probe counted as a poll: on expiry the CTA raises the status word and everybody leaves; the
// issuing lane stays until its copies have landed.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>
#include "kernel_dw_tma.cuh"     // DwTapParams, ptx:: wrappers

namespace qc {

constexpr int kDwMmaWarps = 8;
constexpr int kDwMmaStages = 8;

struct DwMmaParams {
  int cb;            // channels (bytes) of a staged pixel: 32, 64 or 128, also the swizzle span
  int wc_log2;       // log2 of the warps side by side on the channels (cb / 32)
  int swz_mask;      // 16-byte-chunk XOR mask of the staged row: cb / 16 - 1
  int warps;         // consumer warps
  int groups;        // 8-pixel groups of an image row that a CTA owns
  int images;        // images a CTA owns (narrow ones share it)
  int pix;           // pixels per staged image row
  int row_bytes;     // images * pix * cb
  int stage_bytes;   // rounded up to 1024
  int rows_per_cta;  // output rows per strip
  int q_blocks;
  FastDiv fd_q_blocks, fd_groups;
  int lo;            // saturation bound below (0 with ReLU)
  float c1, c2;      // 2^-s and 1.5 * 2^23 * (1 - 2^-s) where all channels share the shift
};

struct DwMmaShared {
  unsigned long long full[kDwMmaStages];
  unsigned long long empty[kDwMmaStages];
  int abort_flag;
  alignas(16) float4 conv[4][16];                            // [32 channels][4 ca + j]: a lane's two channels, 2^-s and M (1 - 2^-s)
};

__device__ __forceinline__ bool dw_mma_wait(uint32_t bar, uint32_t parity, unsigned int limit, DwMmaShared* sh, int* status) {
  for (unsigned int it = 1; it < limit; ++it) {               // (the caller has probed once)
    if (ptx::mbar_try_wait(bar, parity)) return true;
    if (*reinterpret_cast<volatile int*>(&sh->abort_flag)) return false;
  }
  *reinterpret_cast<volatile int*>(&sh->abort_flag) = 1;
  atomicExch(status, kStatusTimeout);
  return false;
}

__device__ __forceinline__ void mma_s8(int32_t (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1,
                                       int32_t c0, int32_t c1, int32_t c2, int32_t c3) {
  asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %11, %12, %13};"
      : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(c0), "r"(c1), "r"(c2), "r"(c3));
}
__device__ __forceinline__ uint2 lds_uint2(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
  return v;
}

template <int STRIDE, bool UNI, bool RELU>
__global__ void __launch_bounds__(kDwMmaWarps * 32, 2)
depthwise3x3_mma_kernel(const __grid_constant__ CUtensorMap tmap_x, const int8_t* __restrict__ weights /* [9][C] */,
                        int8_t* __restrict__ y, ConvGeom g, DwTapParams tp, DwMmaParams prm, int* __restrict__ status,
                        unsigned int wait_limit) {
  extern __shared__ uint8_t dw_mma_smem[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dw_mma_smem) + 1023) & ~static_cast<uintptr_t>(1023));
  DwMmaShared* sh = reinterpret_cast<DwMmaShared*>(tiles + static_cast<size_t>(kDwMmaStages) * prm.stage_bytes);

  int qb;
  const int cblock = prm.fd_q_blocks.divmod(static_cast<int>(blockIdx.x), &qb);
  const int p_start = blockIdx.y * prm.rows_per_cta;
  const int rows_out = min(prm.rows_per_cta, g.P - p_start);
  const int rows_in = (rows_out - 1) * STRIDE + 3;
  const int n0 = blockIdx.z * prm.images;
  const int q_base = qb * prm.groups * 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kDwMmaStages; ++s) {
      ptx::mbar_init(ptx::smem_u32(&sh->full[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&sh->empty[s]), prm.warps);           // one arrival per consumer warp
    }
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  ptx::grid_launch_dependents();

  // The first lane of the first warp also issues the copies, one box per input row: all stages at first, then row
  // i + kDwMmaStages - 2 ahead of its own work on row i, into the stage that row i - 2 has left (rarely a wait).  (With a ninth
  // warp for it, 18 warps an SM leave 96 registers a thread, and the sums spill; 16 leave 128.)
  const uint32_t base = ptx::smem_u32(tiles), full0 = ptx::smem_u32(&sh->full[0]), empty0 = ptx::smem_u32(&sh->empty[0]);
  const bool issuer = threadIdx.x == 0;
  int issued = 0;
  auto issue = [&]() {
    const uint32_t at = static_cast<uint32_t>(issued % kDwMmaStages);
    ptx::mbar_expect_tx(full0 + 8u * at, static_cast<uint32_t>(prm.row_bytes));
    ptx::tma_load_4d(base + at * prm.stage_bytes, &tmap_x, full0 + 8u * at, cblock * prm.cb, q_base * STRIDE - g.pad_w,
                     p_start * STRIDE - g.pad_h + issued, n0);
    ++issued;
  };
  if (issuer) {
    ptx::prefetch_tmap(&tmap_x);
    ptx::grid_dependency_wait();
    while (issued < kDwMmaStages && issued < rows_in) issue();
  }
  __syncwarp();

  const int row8 = lane >> 2, j = lane & 3;                  // pixel of a group (A's rows, B's column), quarter of K
  const int wch = (warp & ((1 << prm.wc_log2) - 1)) * 32;    // this warp's first channel of the staged ones
  const int c_warp = cblock * prm.cb + wch;
  // B: weights of filter row r, chunk c (16 channels), words a = 0: {0, 2} / 1: {1, 3} of the chunk
  uint32_t b0[3][4], b1[3][4];
  int32_t bias[4][2];
#pragma unroll
  for (int ca = 0; ca < 4; ++ca) {
    const int first = c_warp + 16 * (ca >> 1) + 4 * (ca & 1);
    const int ch = first + 8 * (row8 >> 2) + (row8 & 3);     // this column's channel
    const bool mine = (row8 >> 2) == (j & 1) && ch < g.C;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const uint32_t lo = mine ? static_cast<uint8_t>(__ldg(weights + static_cast<size_t>(3 * r + (j >> 1)) * g.C + ch)) : 0u;
      const uint32_t hi = mine && j < 2 ? static_cast<uint8_t>(__ldg(weights + static_cast<size_t>(3 * r + 2) * g.C + ch)) : 0u;
      b0[r][ca] = lo << (8 * (row8 & 3));
      b1[r][ca] = hi << (8 * (row8 & 3));
    }
    const int co = first + 8 * (j >> 1) + 2 * (j & 1);       // channels of this lane's two sums
#pragma unroll
    for (int k = 0; k < 2; ++k) bias[ca][k] = co + k < g.C ? __ldg(tp.bias_magic + co + k) : 0;
    if (!UNI && row8 == 0 && co < g.C) {                      // (warps of the same channels write the same values)
      const float2 s = __ldg(reinterpret_cast<const float2*>(tp.scale_f32 + co)), o = __ldg(reinterpret_cast<const float2*>(tp.offset_f32 + co));
      sh->conv[wch / 32][4 * ca + j] = make_float4(s.x, s.y, o.x, o.y);
    }
  }
  // this lane's words in a staged row, and its pixels in the output, per 8-pixel group
  uint32_t off01[2][2], off2[2][2];                          // [group][chunk]
  int8_t* yp[2];
  bool ok[2];
  const int unit = warp >> prm.wc_log2;
  const int c_out = c_warp + 16 * (j & 1) + 8 * (j >> 1);
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    int col;
    const int image = prm.fd_groups.divmod(2 * unit + u, &col);
    const bool there = image < prm.images;
    const int pixel = (there ? image * prm.pix + col * 8 * STRIDE : 0) + row8 * STRIDE;
    auto at = [&](int tap) {
      const uint32_t lin = static_cast<uint32_t>((pixel + tap) * prm.cb + wch + 8 * (j & 1));
      return lin ^ (((lin >> 7) & static_cast<uint32_t>(prm.swz_mask)) << 4);
    };
    off01[u][0] = at(j >> 1);
    off2[u][0] = at(2);
    off01[u][1] = off01[u][0] ^ 16u;
    off2[u][1] = off2[u][0] ^ 16u;
    const int q = q_base + col * 8 + row8, n = n0 + image;
    ok[u] = there && n < g.N && q < g.Q && c_out < g.C;
    yp[u] = y + (ok[u] ? ((static_cast<size_t>(n) * g.P + p_start) * g.Q + q) * g.out_c_pitch + g.out_c_offset + c_out : 0);
  }
  const size_t y_row = static_cast<size_t>(g.Q) * g.out_c_pitch;
  const uint32_t lo2 = static_cast<uint32_t>(prm.lo & 0xFFFF) * 0x10001u;
  const uint32_t sel_a = j & 1 ? 0x1054u : 0x5410u, sel_b = j & 1 ? 0x3276u : 0x7632u;
  const uint32_t conv = ptx::smem_u32(&sh->conv[wch / 32][j]);
  if (!UNI) __syncwarp();                                    // (each warp reads what it wrote itself)

  int32_t acc[3][4][4];
  // the sums of one output row -> codes
  auto emit = [&](const int32_t (&v)[4][4]) {
    uint32_t x[2][2];                                        // [chunk][group of pixels]: two channels of each word pair
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      uint32_t h[2][2];
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const int ca = 2 * c + a;
        float2 s = make_float2(prm.c1, prm.c1), o = make_float2(prm.c2, prm.c2);
        if (!UNI) {
          const int4 k = lds_int4(conv + 64u * ca);
          s = make_float2(__int_as_float(k.x), __int_as_float(k.y));
          o = make_float2(__int_as_float(k.z), __int_as_float(k.w));
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          // M + v as a float; M + v 2^-s in one rounding: the code in the low mantissa bits (|code| < 2^15 before the clamp)
          const float2 r = fma_pair(make_float2(__int_as_float(v[ca][2 * u]), __int_as_float(v[ca][2 * u + 1])), s, o);
          const uint32_t both = __byte_perm(__float_as_uint(r.x), __float_as_uint(r.y), 0x5410);
          h[a][u] = RELU ? __vimin_s16x2_relu(both, 0x007F007Fu) : __vmaxs2(__vmins2(both, 0x007F007Fu), lo2);
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) x[c][u] = __byte_perm(h[0][u], h[1][u], 0x6420);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const uint32_t keep = j & 1 ? x[1][u] : x[0][u], send = j & 1 ? x[0][u] : x[1][u];
      const uint32_t got = __shfl_xor_sync(0xffffffffu, send, 1);
      if (ok[u] && QC_IN(yp[u] - y + 7, static_cast<size_t>(g.N) * g.P * g.Q * g.out_c_pitch))
        *reinterpret_cast<uint2*>(yp[u]) = make_uint2(__byte_perm(keep, got, sel_a), __byte_perm(keep, got, sel_b));
      yp[u] += y_row;
    }
  };
  // One input row against filter rows: FIRST starts slot s0 (filter row 0), MID adds row 1 to s1, LAST row 2 to s2.
  bool go = wait_limit != 0;                                  // (no polls granted: every warp gives up here)
  int stage = 0, taken = 0;
  uint32_t parity = 0;
  auto take = [&](auto first, auto mid, auto last, int32_t (&s0)[4][4], int32_t (&s1)[4][4], int32_t (&s2)[4][4]) {
    const uint32_t bar = 8u * static_cast<uint32_t>(stage);
    if (issuer && taken >= 2 && issued < rows_in) {
      const uint32_t free = empty0 + 8u * static_cast<uint32_t>(issued % kDwMmaStages), left = static_cast<uint32_t>(issued / kDwMmaStages - 1) & 1u;
      if (ptx::mbar_try_wait(free, left) || dw_mma_wait(free, left, wait_limit, sh, status)) issue();
      else go = false;
    }
    ++taken;
    go = go && (ptx::mbar_try_wait(full0 + bar, parity) || dw_mma_wait(full0 + bar, parity, wait_limit, sh, status));
    go = __all_sync(0xffffffffu, go);                        // (the warp gives up together)
    if (!go) return;
    const uint32_t row = base + static_cast<uint32_t>(stage * prm.stage_bytes);
    uint2 w01[2][2], w2[2][2];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        w01[c][u] = lds_uint2(row + off01[u][c]);
        w2[c][u] = lds_uint2(row + off2[u][c]);
      }
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(empty0 + bar);            // the words are in registers
    if (++stage == kDwMmaStages) { stage = 0; parity ^= 1u; }
    // the row that this completes first: its conversion then runs beside the other rows' multiplications
#pragma unroll
    for (int r = 2; r >= 0; --r) {
#pragma unroll
      for (int ca = 0; ca < 4; ++ca) {
        const int c = ca >> 1;
        const uint32_t a0 = ca & 1 ? w01[c][0].y : w01[c][0].x, a1 = ca & 1 ? w01[c][1].y : w01[c][1].x;
        const uint32_t a2 = ca & 1 ? w2[c][0].y : w2[c][0].x, a3 = ca & 1 ? w2[c][1].y : w2[c][1].x;
        if (r == 2 && decltype(last)::value) mma_s8(s2[ca], a0, a1, a2, a3, b0[2][ca], b1[2][ca], s2[ca][0], s2[ca][1], s2[ca][2], s2[ca][3]);
        if (r == 1 && decltype(mid)::value) mma_s8(s1[ca], a0, a1, a2, a3, b0[1][ca], b1[1][ca], s1[ca][0], s1[ca][1], s1[ca][2], s1[ca][3]);
        if (r == 0 && decltype(first)::value) mma_s8(s0[ca], a0, a1, a2, a3, b0[0][ca], b1[0][ca], bias[ca][0], bias[ca][1], bias[ca][0], bias[ca][1]);
      }
    }
  };
  constexpr std::true_type yes{};
  constexpr std::false_type no{};
  if (STRIDE == 1) {
    // output row o meets input rows o, o + 1, o + 2; sums of row o sit in slot o % 3.  (Sums that the strip's last rows start
    // for rows past its end are never used.)
    take(yes, no, no, acc[0], acc[0], acc[0]);
    if (go) take(yes, yes, no, acc[1], acc[0], acc[0]);
    for (int o = 0; go && o < rows_out; o += 3) {
      take(yes, yes, yes, acc[2], acc[1], acc[0]);
      if (!go) break;
      emit(acc[0]);
      if (o + 1 >= rows_out) break;
      take(yes, yes, yes, acc[0], acc[2], acc[1]);
      if (!go) break;
      emit(acc[1]);
      if (o + 2 >= rows_out) break;
      take(yes, yes, yes, acc[1], acc[0], acc[2]);
      if (!go) break;
      emit(acc[2]);
    }
  } else {
    // output row o meets input rows 2 o, 2 o + 1, 2 o + 2
    take(yes, no, no, acc[0], acc[0], acc[0]);
    for (int o = 0; go && o < rows_out; o += 2) {
      take(no, yes, no, acc[0], acc[0], acc[0]);
      if (go) take(yes, no, yes, acc[1], acc[0], acc[0]);
      if (!go) break;
      emit(acc[0]);
      if (o + 1 >= rows_out) break;
      take(no, yes, no, acc[1], acc[1], acc[1]);
      if (go) take(yes, no, yes, acc[0], acc[1], acc[1]);
      if (!go) break;
      emit(acc[1]);
    }
  }
  // After a wait that expired, copies already on their way must land before this CTA's shared memory goes away, whatever the
  // caller's wait limit.  (A strip that was walked to its end has used every row.)
  if (issuer && !go) {
    if (wait_limit == 0) atomicExch(status, kStatusTimeout);
    for (int i = issued > kDwMmaStages ? issued - kDwMmaStages : 0; i < issued; ++i) {
      const uint32_t par = static_cast<uint32_t>(i / kDwMmaStages) & 1u;
      for (unsigned int it = 0; it < kDrainPolls; ++it)
        if (ptx::mbar_try_wait(full0 + 8u * (i % kDwMmaStages), par)) break;
    }
  }
  // every CTA waits for the kernel before it before it retires (see the chain in kernel_igemm.cuh)
  ptx::grid_dependency_wait();
}

}  // namespace qc
