// Host side of the C ABI declared in include/qconv.h: argument validation, the planner that
// maps a layer shape to a kernel and tile shape, weight repacking, TMA descriptors, launches.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <exception>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#include "../../include/qconv.h"
#include "epilogue.cuh"
#include "graph_inputs.cuh"
#include "host_weights.cuh"
#include "kernel_igemm.cuh"
#include "kernel_dw_mma.cuh"
#include "kernel_dw_tma.cuh"
#include "kernel_igemm_pair.cuh"
#include "kernel_mma_peak.cuh"
#include "kernels_calib.cuh"
#include "kernels_dynfloat.cuh"
#include "kernels_npconv.cuh"
#include "kernels_simple.cuh"
#include "kernels_threshold.cuh"
#include "per_device.cuh"

static_assert(QCALIB_STATIC_MAX_BINS <= qc::kCalibMaxBins, "built-in scratch holds kCalibMaxBins counters");

namespace {

thread_local char g_err[512] = "";

int fail(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return code;
}

#define CUDA_TRY(expr)                                                                        \
  do {                                                                                        \
    cudaError_t e_ = (expr);                                                                  \
    if (e_ != cudaSuccess)                                                                    \
      return fail(QCONV_ERR_CUDA, "%s failed: %s", #expr, cudaGetErrorString(e_));            \
  } while (0)

// cuTensorMapEncodeTiled is resolved through the runtime so the library links only cudart.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

CUtensorMapSwizzle swizzle_for(int bkc) {
  if (bkc == 0) return CU_TENSOR_MAP_SWIZZLE_NONE;
  return bkc == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (bkc == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                              : CU_TENSOR_MAP_SWIZZLE_32B);
}

int encode_map(CUtensorMap* map, const void* base, int rank, const cuuint64_t* dims,
               const cuuint64_t* strides_bytes /* rank-1 */, const cuuint32_t* box, int bkc,
               const cuuint32_t* elem_strides = nullptr) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return fail(QCONV_ERR_CUDA, "cuTensorMapEncodeTiled is not available from this driver");
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  for (int i = 0; i < rank && elem_strides; ++i) estr[i] = elem_strides[i];
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, static_cast<cuuint32_t>(rank), const_cast<void*>(base),
                  dims, strides_bytes, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(bkc),
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(QCONV_ERR_CUDA, "cuTensorMapEncodeTiled failed with CUresult %d", (int)r);
  return QCONV_OK;
}

int ceil_div(int a, int b) { return (a + b - 1) / b; }
long ceil_div_l(long a, long b) { return (a + b - 1) / b; }
size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Plan overrides of the calling thread (qconv_set_plan_hints); -1 / 0 = the planner decides.
constexpr qconv_plan_hints kNoHints = {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, 0, 0};
thread_local qconv_plan_hints g_hints = kNoHints;

enum IgemmMode { MODE_FLAT = 0, MODE_VIEW = 1, MODE_BOX = 2, MODE_STEM = 3, MODE_S2D = 4, MODE_WROW = 5 };
// modes whose activation operand is an overlapping window view of a packed, row-padded image
inline bool is_window_mode(int m) { return m == MODE_S2D || m == MODE_WROW; }

}  // namespace

// Device memory of the handles' tables and scratch.  A network's calibration builds and destroys two handles per layer;
// cudaMalloc and cudaFree took two thirds of that time, and at times a hundred milliseconds for one call.  Blocks given back are kept for the next handle, at most kKeep bytes per
// device, and all of them are freed when the last block in use is given back, or when the device has no memory left.  Any thread, any stream: a block is only
// given back after the device is idle, so whoever takes it next may overwrite it at once.
class DevicePool {
 public:
  struct Block {
    void* ptr = nullptr;
    size_t bytes = 0;
    int device = 0;
    Block() = default;
    Block(const Block&) = delete;
    Block& operator=(const Block&) = delete;
    ~Block() { if (ptr) pool().give(*this); }
  };
  static DevicePool& pool() {
    static DevicePool* p = new DevicePool;                 // never destroyed: handles may outlive static destructors
    return *p;
  }
  cudaError_t take(Block* b, size_t bytes) {
    bytes = (std::max<size_t>(bytes, 1) + 4095) / 4096 * 4096;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    b->device = dev;
    std::lock_guard<std::mutex> lock(mu_);
    PerDevice& d = per_device_[dev & 63];
    size_t best = d.free.size();
    for (size_t i = 0; i < d.free.size(); ++i)
      if (d.free[i].second >= bytes && d.free[i].second <= 2 * bytes && (best == d.free.size() || d.free[i].second < d.free[best].second))
        best = i;
    if (best < d.free.size()) {
      b->ptr = d.free[best].first;
      b->bytes = d.free[best].second;
      d.kept -= b->bytes;
      d.free.erase(d.free.begin() + static_cast<long>(best));
    } else {
      e = allocate(&b->ptr, bytes, d);
      if (e != cudaSuccess) { b->ptr = nullptr; return e; }
      b->bytes = bytes;
    }
    ++d.live;
    return cudaSuccess;
  }
  // cudaMalloc for memory that is not the pool's.
  template <typename T>
  cudaError_t plain(T** ptr, size_t bytes) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu_);
    return allocate(reinterpret_cast<void**>(ptr), bytes, per_device_[dev & 63]);
  }

 private:
  static constexpr size_t kKeep = 256u << 20;
  struct PerDevice {
    std::vector<std::pair<void*, size_t>> free;            // oldest first
    size_t kept = 0, live = 0;
  };
  std::mutex mu_;
  PerDevice per_device_[64];

  // On a full device what is kept for later handles goes first.  (Kept blocks are idle.)
  cudaError_t allocate(void** ptr, size_t bytes, PerDevice& d) {
    cudaError_t e = cudaMalloc(ptr, bytes);
    if (e != cudaErrorMemoryAllocation || d.free.empty()) return e;
    cudaGetLastError();
    for (auto& f : d.free) cudaFree(f.first);
    d.free.clear();
    d.kept = 0;
    return cudaMalloc(ptr, bytes);
  }
  void give(Block& b) {
    int dev = 0;
    const bool other = cudaGetDevice(&dev) == cudaSuccess && dev != b.device && cudaSetDevice(b.device) == cudaSuccess;
    const bool idle = cudaDeviceSynchronize() == cudaSuccess;
    std::vector<void*> drop;
    {
      std::lock_guard<std::mutex> lock(mu_);
      PerDevice& d = per_device_[b.device & 63];
      --d.live;
      if (idle) { d.free.emplace_back(b.ptr, b.bytes); d.kept += b.bytes; } else { drop.push_back(b.ptr); }
      size_t n = 0;
      while (n < d.free.size() && (d.live == 0 || d.kept > kKeep)) { drop.push_back(d.free[n].first); d.kept -= d.free[n].second; ++n; }
      d.free.erase(d.free.begin(), d.free.begin() + static_cast<long>(n));
    }
    for (void* p : drop) cudaFree(p);
    if (other) cudaSetDevice(dev);
    b.ptr = nullptr;
  }
};

struct qgraph_inputs {
  qc::GraphInputRecord rec;
};

// Digit products of a layer on floating-point operands (qconv_np_create): what the planner needs beyond the descriptor.
struct NpSpec {
  int products = 0, planes = 0;
  int a_plane[qc::kNpMaxProducts], coef[qc::kNpMaxProducts];
  int n_out, p_out;
  float top;                                               // beta_max of the output type
  long long largest_sum, largest_bias;                     // Eq. 9 with b = beta_max and the largest bias; that bias
  const int8_t* w[qc::kNpMaxProducts];                     // per product: the weights' digit combination, [K][R][S][C]
};

struct qconv_handle {
  qconv_desc d;
  int P, Q, Cg, Kg;
  int algo;                      // resolved QCONV_ALGO_*
  int lo, hi;
  // device copies: the small tables in one block, large weights in a second one that handles of the same weights share
  DevicePool::Block block, pack;
  std::shared_ptr<DevicePool::Block> weights;
  int a_channels = 0;            // channels of the activation tensor (planes * padded C for floating-point operands)
  const NpSpec* np = nullptr;    // set while the handle is built
  int np_products = 0;
  bool np3 = false;              // two-digit operands whose sums are recombined and converted in 32 bits
  bool weights_as_is = false;    // those weights lie as the host handed them over ([K][R][S][C])
  int8_t* d_w = nullptr;         // direct: [R][S][Cg][K]; depthwise: [R*S][C]; igemm: [Kpad][Kg_total]
  int32_t* d_bias = nullptr;
  int32_t* d_shift = nullptr;
  int32_t* d_lshift = nullptr;
  int32_t* d_accexp = nullptr;
  int* d_status = nullptr;
  int4* d_chan = nullptr;        // igemm: per-channel epilogue constants {bias, s, 2^(s-1)-1, s>0}
  long long acc_bound = 0;       // worst-case |accumulator| (Eq. 9 / Eq. 13 bound)
  int max_shift = 0;
  long walk_grid = -1;             // grid size the tile-walk constants in prm were made for
  int split = 1;                   // CTAs that shared a tile's contraction in the last run
  int gen_flt = 0;               // 1: the same bound with the rounding mode's half: float rounding in the general epilogue
  int flt_epilogue = 0;          // 1: |wide value| < 2^22 for any input (weight-aware bound): float-rounding epilogue
  int uniform_shift = 0;         // 1: all channels share the right shift and the residual left shift
  int uni_s = 0, uni_t = 0;
  int num_sms = 148;
  int ctas_per_sm = 2;
  int use_pdl = 1;
  int dw_warp = 0;               // depthwise on warp-level matrix instructions (kernel_dw_mma.cuh)
  qc::DwMmaParams dw_mma_prm = {};
  int dw_rows_n = -1;            // the batch that dw_mma_prm.rows_per_cta was found for
  int dw_mma = 0;                // depthwise on the tensor cores (prm, mode and the maps are then its plan)
  int8_t* d_w_mma = nullptr;     // its weights: [C][9][32]
  uint32_t* d_dw_tap = nullptr;  // tap-packed form: weight rows [3][C], bias + magic [C], 2^-s [C], rounding offset [C] (float bits)
  int dw_tap = 0;
  uint32_t plan_stage_bytes = 0; // staged output tiles as planned; a run may do without or use the ring (plan_staging)
  int plan_stage_bufs = 0;
  bool ring_out_fits = false;    // no staged tiles in the plan, but a CTA with one tile may stage it in its ring
  int patch = 0;                 // 1: patch form (one activation box of 16 x (tp + 2) pixels serves all nine taps)
  int pair = 0;                  // 1: tiles of 256 pixels x 256 channels on pairs of SMs (kernel_igemm_pair.cuh)
  int fold = 1;                  // flat GEMMs with few output channels: this many pixels form one GEMM row
  int dw_tma = 0;                // rows staged by TMA (C % 32 == 0)
  qc::DwTmaParams dw_prm = {};
  CUtensorMap dw_map;
  const void* dw_key_ptr = nullptr;
  int dw_key_n = -1, dw_key_form = 0;
  int8_t* d_pack = nullptr;      // stem: packed patches [N*P*Q][kg_pad]
  int stem_segp = 0;             // stem: bytes per filter-row segment of a packed row (0: taps back to back)
  // stride-2 stem in space-to-depth form: d_pack is [N][s2d_h][s2d_wp] 16-byte block pixels, the image starting
  // at pixel s2d_off_w of a row; the filter covers s2d_r x s2d_s blocks starting s2d_off_h / s2d_off_w blocks
  // up / left of block (p, q)
  int s2d_h = 0, s2d_w = 0, s2d_wp = 0, s2d_off_h = 0, s2d_off_w = 0, s2d_r = 0, s2d_s = 0;
  // MODE_WROW uses the same fields for a stride-1 layer on few channels: d_pack is the image itself with
  // zero-padded rows, a packed pixel is the layer's C bytes (win_pb; 16 for the space-to-depth stems)
  int win_pb = 16;
  // igemm plan
  int mode = 0;
  qc::IgemmParams prm{};
  int kg_pad = 0, kg_total = 0, kpad = 0;
  size_t smem_bytes = 0;
  CUtensorMap tmap_b;
  CUtensorMap tmap_a;
  const void* a_key_ptr = nullptr;
  int a_key_n = -1;
  CUtensorMap tmap_y;            // output tiles leave through TMA stores (fast int8 epilogues)
  const void* y_key_ptr = nullptr;
  int y_key_n = -1;
  CUtensorMap tmap_r;            // residual tiles arrive through TMA loads (same boxes, dense [pixels][K])
  const void* r_key_ptr = nullptr;
  int r_key_n = -1;
  unsigned int wait_limit = 1u << 22;
  cudaStream_t last_stream = nullptr;
  int device = 0;
  qconv_plan_hints hints = kNoHints;   // the creating thread's overrides at create time
};

namespace {

void free_handle(qconv_handle* h) {
  if (!h) return;
  delete h;
}

// A handle's small host tables on their way to the device, in one block and one copy.
class DeviceParts {
 public:
  // `bytes` bytes of `src` (NULL: zeros), which stays valid until upload(); *dst receives the device address.
  template <typename T>
  void add(T** dst, const void* src, size_t bytes) {
    parts_.push_back({reinterpret_cast<void**>(dst), src, bytes, total_});
    total_ = align_up(total_ + bytes, 256);
  }
  // Device memory behind the tables, not copied to.
  template <typename T>
  void reserve(T** dst, size_t bytes) {
    reserved_ = reinterpret_cast<void**>(dst);
    reserved_bytes_ = bytes;
  }
  // first: runs once the tables have their addresses, before they are copied (the copy is waited for, and so is what
  // `first` puts on the default stream).
  template <typename First>
  int upload(DevicePool::Block* block, First first) {
    CUDA_TRY(DevicePool::pool().take(block, total_ + reserved_bytes_));
    if (reserved_) *reserved_ = static_cast<uint8_t*>(block->ptr) + total_;
    std::vector<uint8_t> host(total_, 0);
    for (const Part& p : parts_) {
      *p.dst = static_cast<uint8_t*>(block->ptr) + p.at;
      if (p.src) std::memcpy(host.data() + p.at, p.src, p.bytes);
    }
    CUDA_TRY(first());
    CUDA_TRY(cudaMemcpy(block->ptr, host.data(), total_, cudaMemcpyHostToDevice));
    return QCONV_OK;
  }
  int upload(DevicePool::Block* block) { return upload(block, [] { return cudaSuccess; }); }
  // The part of destination `dst` to the device at once (inside `first`).
  template <typename T>
  cudaError_t copy_now(T** dst) const {
    for (const Part& p : parts_)
      if (p.dst == reinterpret_cast<void**>(dst)) return cudaMemcpyAsync(*dst, p.src, p.bytes, cudaMemcpyHostToDevice, nullptr);
    return cudaSuccess;                                    // (has a block of its own and is there already)
  }

 private:
  struct Part { void** dst; const void* src; size_t bytes, at; };
  std::vector<Part> parts_;
  size_t total_ = 0, reserved_bytes_ = 0;
  void** reserved_ = nullptr;
};

// The layer's weights: a part of the handle's block, or (from 64 KB) a block of their own that a second handle of the
// same weights can use too.  `from`: the handle they may be shared with, or NULL.
int place_weights(qconv_handle* h, DeviceParts& parts, const int8_t* w, size_t bytes, bool as_is, const qconv_handle* from) {
  h->weights_as_is = as_is;
  if (bytes < 64 * 1024) {
    parts.add(&h->d_w, w, bytes);
    return QCONV_OK;
  }
  if (as_is && from && from->weights && from->weights_as_is && from->device == h->device && from->d.K == h->d.K &&
      from->d.R == h->d.R && from->d.S == h->d.S && from->d.C == h->d.C && from->algo == h->algo) {
    h->weights = from->weights;
  } else {
    h->weights = std::make_shared<DevicePool::Block>();
    CUDA_TRY(DevicePool::pool().take(h->weights.get(), bytes));
    CUDA_TRY(cudaMemcpy(h->weights->ptr, w, bytes, cudaMemcpyHostToDevice));
  }
  h->d_w = static_cast<int8_t*>(h->weights->ptr);
  return QCONV_OK;
}

// Multiplier and shift for the kernel's divisions by d (1 <= d < 2^31) of n < 2^31.  With 2^shr < d <= 2^(shr+1) and
// mul = ceil(2^(32+shr) / d), e = mul d - 2^(32+shr) lies in [0, d), so n e < 2^31 2^(shr+1) = 2^(32+shr): the quotient
// n mul / 2^(32+shr) exceeds n / d by less than 1 / d and has the same whole part.
qc::FastDiv make_fastdiv(int d_in) {
  qc::FastDiv f = {0u, 0u, static_cast<uint32_t>(std::max(1, d_in))};
  if (f.d > 1u) {
    uint32_t lg = 0;
    while ((1ull << lg) < f.d) ++lg;                       // ceil(log2 d) >= 1
    f.shr = lg - 1;
    f.mul = static_cast<uint32_t>(((1ull << (32 + f.shr)) + f.d - 1) / f.d);
  }
  return f;
}

// Output-pixel box (tq x tp x tn <= 128) that wastes the fewest accumulator rows.
// pool: the epilogue takes a 2 x 2 max-pool with warp shuffles, so a window's four pixels must be lanes of one
// warp: tq a power of two up to 16 (rows run q fastest), tp even; Q and P are even.
void search_box(int Q, int P, int N, int* tq_o, int* tp_o, int* tn_o, bool pool, long slots) {
  long best_tiles = -1;
  int btq = 1, btp = 1, btn = 1;
  if (pool) {
    for (int tq = 2; tq <= 16; tq *= 2) {
      for (int tp = 2; tp <= std::min(P, 128 / tq); tp += 2) {
        const int tn = std::max(1, std::min(N, 128 / (tq * tp)));
        const long tiles = static_cast<long>(ceil_div(Q, tq)) * ceil_div(P, tp) * ceil_div(N, tn);
        if (best_tiles < 0 || tiles < best_tiles || (tiles == best_tiles && tq > btq)) {
          best_tiles = tiles; btq = tq; btp = tp; btn = tn;
        }
      }
    }
    *tq_o = btq; *tp_o = btp; *tn_o = btn;
    return;
  }
  // A box may take a patch of several images (a 4-D TMA box of the NHWC tensor): with 28 x 28 outputs, 4 x 4
  // pixels of 8 images fill the 128 accumulator rows where whole image rows (28 x 4) fill 112 -- an eighth fewer
  // tiles, which is what the tensor-bound layers gain (VGG conv3_2 / conv4_x: 10 %).  Fewest tiles win; then the
  // fewest images per box (squarer patches re-read less halo), then the widest patch.
  // slots (0: unknown): tiles that run at the same time.  A layer whose whole-row boxes all run at once gains
  // nothing from fewer tiles and keeps them: their long contiguous runs load a little faster.
  if (slots > 0) {
    long rows_tiles = -1;
    int rq = 1, rp = 1, rn = 1;
    for (int tq = 1; tq <= std::min(Q, 128); ++tq) {
      const int nq = ceil_div(Q, tq);
      if (tq != ceil_div(Q, nq)) continue;
      for (int tp = 1; tp <= std::min(P, 128 / tq); ++tp) {
        const int np = ceil_div(P, tp);
        if (tp != ceil_div(P, np)) continue;
        const int tn = (tq == Q && tp == P) ? std::max(1, std::min(N, 128 / (tq * tp))) : 1;
        const long tiles = static_cast<long>(nq) * np * ceil_div(N, tn);
        if (rows_tiles < 0 || tiles < rows_tiles || (tiles == rows_tiles && tq > rq)) {
          rows_tiles = tiles; rq = tq; rp = tp; rn = tn;
        }
      }
    }
    if (rows_tiles <= slots) {
      *tq_o = rq; *tp_o = rp; *tn_o = rn;
      return;
    }
  }
  for (int tq = 1; tq <= std::min(Q, 128); ++tq) {
    int nq = ceil_div(Q, tq);
    if (tq != ceil_div(Q, nq)) continue;
    int tpmax = std::min(P, 128 / tq);
    for (int tp = 1; tp <= tpmax; ++tp) {
      int np = ceil_div(P, tp);
      if (tp != ceil_div(P, np)) continue;
      const int tn = std::max(1, std::min(N, 128 / (tq * tp)));
      long tiles = static_cast<long>(nq) * np * ceil_div(N, tn);
      if (best_tiles < 0 || tiles < best_tiles || (tiles == best_tiles && (tn < btn || (tn == btn && tq > btq)))) {
        best_tiles = tiles; btq = tq; btp = tp; btn = tn;
      }
    }
  }
  *tq_o = btq; *tp_o = btp; *tn_o = btn;
}

// (a layer's plan asks for the same box several times, a search of some thousand steps each)
void choose_box(int Q, int P, int N, int* tq_o, int* tp_o, int* tn_o, bool pool = false, long slots = 0) {
  static thread_local struct { int Q = -1, P, N; bool pool; long slots; int tq, tp, tn; } last[2];
  for (const auto& l : last)
    if (l.Q == Q && l.P == P && l.N == N && l.pool == pool && l.slots == slots) { *tq_o = l.tq; *tp_o = l.tp; *tn_o = l.tn; return; }
  search_box(Q, P, N, tq_o, tp_o, tn_o, pool, slots);
  last[1] = last[0];
  last[0] = {Q, P, N, pool, slots, *tq_o, *tp_o, *tn_o};
}

// Bytes of the contraction axis per ring stage.  A stage costs about the same whether its rows are
// 32, 64 or 128 bytes long (the TMA unit works row by row), so the fewest chunks win and zero
// padding is cheap; among equals the narrowest chunk.
int choose_bkc(int c) {
  int best = 128, best_chunks = 1 << 30, best_pad = 1 << 30;
  for (int bkc : {128, 64, 32}) {
    const int chunks = ceil_div(c, bkc), padded = chunks * bkc;
    if (chunks < best_chunks || (chunks == best_chunks && padded < best_pad)) {
      best_chunks = chunks; best_pad = padded; best = bkc;
    }
  }
  return best;
}

typedef void (*IgemmKernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const qc::IgemmParams,
                            const qc::EpilogueParams,
                            const int4*, const int8_t*, void*, int*, unsigned int);

IgemmKernel igemm_kernel_for(const qconv_handle* h, bool maxabs = false);
typedef void (*PairKernel)(const CUtensorMap, const CUtensorMap, const qc::PairParams, const qc::IgemmParams,
                           const qc::EpilogueParams, const int4*, void*, int*, unsigned int);
PairKernel pair_kernel_for(const qconv_handle* h);

// Tile of the patch form: 16 accumulator rows per image row, 14 of them outputs (the other two are the halo's columns),
// so that image rows start at multiples of 16 rows; up to eight image rows.
struct PatchTile { int q_step, segs, tp, rows; };
PatchTile patch_tile(int Q, int P, bool pool) {
  PatchTile t;
  t.segs = ceil_div(Q, 14);
  t.q_step = ceil_div(Q, t.segs);
  if (pool) t.q_step += t.q_step & 1;                      // (a 2 x 2 window stays inside a tile)
  t.rows = ceil_div(P, 8);
  t.tp = ceil_div(P, t.rows);
  if (pool) t.tp += t.tp & 1;
  return t;
}

// Tile of the halo form: whole image rows with their halo, W + S - 1 accumulator rows per image row (S - 1 of them discarded);
// an image wider than that leaves room for is cut into equal column segments, each with its own halo.
int halo_segments(const qconv_desc& d) { return ceil_div(d.W, qc::kTileM - (d.S - 1)); }
void halo_box(const qconv_handle* h, int* tq, int* tp, int* tn, int* step) {
  const qconv_desc& d = h->d;
  const int segs = halo_segments(d);
  *step = ceil_div(d.W, segs);
  *tq = *step + d.S - 1;
  *tp = std::max(1, std::min(h->P, qc::kTileM / *tq));
  *tn = (segs == 1 && *tp == h->P) ? std::max(1, std::min(d.N, qc::kTileM / (*tq * *tp))) : 1;
}

// Tiles of a depthwise layer on tcgen05: channels (bytes) of a row, and at stride 1 the form (patch, or a box per filter row)
// whose tiles waste fewer accumulator rows.
struct DwTiles { int bkc; bool halo; long tiles; };
DwTiles dw_tiles(const qconv_handle* h) {
  const qconv_desc& d = h->d;
  const qconv_plan_hints& hint = h->hints;
  DwTiles t = {};
  // 128 wide unless the last tile would be mostly padding; at stride 2 rows of 64 bytes, the three taps of a filter row sharing
  // a stage
  const bool wide_row = d.stride_h == 1 && !(hint.bn_max > 0 && hint.bn_max < 128) && align_up(d.C, 128) * 7 <= align_up(d.C, 64) * 8;
  t.bkc = wide_row ? 128 : d.C > 32 ? 64 : 32;
  if (d.stride_h == 1) {
    const PatchTile pt = patch_tile(h->Q, h->P, false);
    int tq, tp, tn, step;
    halo_box(h, &tq, &tp, &tn, &step);
    const long patches = static_cast<long>(pt.segs) * pt.rows * d.N;
    const long halos = static_cast<long>(ceil_div(h->Q, step)) * ceil_div(h->P, tp) * ceil_div(d.N, tn);
    t.halo = hint.halo != 0 && halos < patches;
    t.tiles = t.halo ? halos : patches;
  } else {
    int tq, tp, tn;
    choose_box(h->Q, h->P, d.N, &tq, &tp, &tn);
    t.tiles = static_cast<long>(ceil_div(h->Q, tq)) * ceil_div(h->P, tp) * ceil_div(d.N, tn);
  }
  t.tiles *= ceil_div(d.C, t.bkc);
  return t;
}

int plan_igemm(qconv_handle* h, DeviceParts& parts, const qconv_handle* weights_of, const int8_t* w_krsc /* host [K][R][S][Cg] */,
               const int32_t* bias_host, const int32_t* shift_host, const int32_t* res_lshift_host, const int32_t* acc_exp_host) {
  const qconv_desc& d = h->d;
  const qconv_plan_hints& hint = h->hints;
  qc::IgemmParams& p = h->prm;
  int c_eff = d.C;                 // channels of the GEMM's activation operand
  const bool dw = h->dw_mma != 0;
  int taps_r = d.R, taps_s = d.S;
  if (h->mode == MODE_STEM) {
    // packed patch row: either the R*S*C taps back to back, or (when a filter row is at most 28
    // bytes) one 16- or 32-byte segment per filter row, which packs with aligned word copies
    h->stem_segp = d.S * d.C <= 16 ? 16 : (d.S * d.C <= 28 ? 32 : 0);
    const size_t row = h->stem_segp ? static_cast<size_t>(d.R) * h->stem_segp : static_cast<size_t>(d.R) * d.S * d.C;
    h->kg_pad = static_cast<int>(align_up(row, 32));
    c_eff = h->kg_pad;
    taps_r = taps_s = 1;
  }
  if (h->mode == MODE_S2D) {
    // y = 2p - pad + r = 2 (p - off) + j with off = ceil(pad / 2), j = r + 2 off - pad: block rows p - off ...
    h->s2d_off_h = (d.pad_h + 1) / 2;
    h->s2d_off_w = (d.pad_w + 1) / 2;
    h->s2d_r = ceil_div(d.R + 2 * h->s2d_off_h - d.pad_h, 2);
    h->s2d_s = ceil_div(d.S + 2 * h->s2d_off_w - d.pad_w, 2);
    h->s2d_h = ceil_div(d.H, 2);
    h->s2d_w = ceil_div(d.W, 2);
    c_eff = h->s2d_s * 16;         // one GEMM row per filter block row: s2d_s adjacent 16-byte block pixels
    taps_r = h->s2d_r;
    taps_s = 1;
  }
  if (h->mode == MODE_WROW) {
    // Stride 1 on few channels: the S taps of a filter row are S adjacent pixels, contiguous in memory,
    // so one (or two) wide TMA rows replace S narrow ones.  Needs rows padded with zeros left and right
    // (a copy of the image, cheap at these channel counts); rows above / below come from TMA's zero fill.
    // With at most 4 channels the padded copy also widens every pixel to 8 bytes (16 when rows are not
    // folded: a TMA row must start on a 16-byte boundary), zeros after the channels.
    h->win_pb = d.C >= 16 ? d.C : 8;
    h->s2d_off_h = d.pad_h; h->s2d_off_w = d.pad_w;
    h->s2d_r = d.R; h->s2d_s = d.S;
    h->s2d_h = d.H; h->s2d_w = d.W;
    c_eff = d.S * h->win_pb;
    taps_r = d.R;
    taps_s = 1;
  }
  // Narrow layers (K <= 64) would run tiles only K columns wide, and the cost of a tile hardly depends
  // on its width.  Consecutive pixels of a flat GEMM are contiguous in memory, so f of them can be
  // read as ONE row of f * C bytes against block-diagonal weights [f * K][f * C]: the product row is
  // those f pixels' outputs, again contiguous.  Same bytes, 1/f of the rows, tiles f times wider;
  // the extra multiply-adds (zeros) cost the tensor core nothing noticeable at this size.
  h->fold = 1;
  // only with the 16-byte-store epilogues, which index nothing but the (replicated) channel table
  const long long fold_round_room = h->max_shift > 0 ? (1ll << (h->max_shift - 1)) : 0;
  const NpSpec* np = h->np;
  const bool fast_possible = !np && d.out_mode == QCONV_OUT_INT8 && d.rounding == QCONV_ROUND_NEAREST_EVEN && d.n_out == 8 &&
                             h->acc_bound + fold_round_room <= 2147483647ll && hint.fast_epilogue != 0;
  if ((h->mode == MODE_FLAT || h->mode == MODE_STEM) && fast_possible && d.out_c_offset == 0 &&
      d.out_c_pitch == d.K && hint.fold != 0) {
    for (int f = 8; f >= 2; f /= 2) {
      // (a folded row of more than two 128-byte chunks costs more in zero multiply-adds and ring stages than the wider
      // tile saves: ResNet's 256 -> 64 layers 9.1 -> 7.2 us unfolded, inception's 5x5-reduce layers 9-19 % faster)
      if (f * d.K <= 128 && (f * d.K) % 16 == 0 && (h->P * h->Q) % f == 0 && f * c_eff <= 256 &&
          (static_cast<long>(f) * c_eff) % 16 == 0) {
        h->fold = f;
        break;
      }
    }
  }
  if (is_window_mode(h->mode) && fast_possible && d.out_c_offset == 0 && d.out_c_pitch == d.K &&
      hint.fold != 0) {
    // The same folding for the space-to-depth view: a row that starts at block q and spans f + s2d_s - 1
    // blocks holds the windows of the f outputs q ... q + f - 1; the weights repeat along the row, shifted
    // by one block per output (block Toeplitz).  Rows get longer (TMA moves long rows much faster than
    // 32- or 64-byte ones) and f times fewer.
    for (int f = 8; f >= 2; f /= 2) {
      if (f * d.K <= 128 && (f * d.K) % 16 == 0 && h->Q % f == 0 &&
          (f + h->s2d_s - 1) * h->win_pb <= (h->mode == MODE_WROW ? 256 : 128)) {
        h->fold = f;
        break;
      }
    }
  }
  if (h->mode == MODE_WROW && h->win_pb == 8 && h->fold == 1) h->win_pb = 16;
  const int c_row = c_eff;         // bytes of one pixel's GEMM row before folding
  const int k_eff = d.K * h->fold;
  if (is_window_mode(h->mode)) c_eff = (h->fold + h->s2d_s - 1) * h->win_pb;
  else c_eff *= h->fold;
  // Halo form of a 3-tap-wide stride-1 layer on a multiple of 128 channels: one activation box per filter row,
  // W + 2 pixels wide (the halo comes from TMA's zero fill), serves the three horizontal taps -- the tensor core
  // reads the same shared-memory rows shifted by one pixel per tap.  A third of the activation fill traffic.
  const int taps_s_w = taps_s;                             // taps per filter row in the packed weights
  // It costs three weight chunks per stage, so it is used where tiles are 64 channels wide anyway (layers below
  // one wave, which sit at the fill rate), not for the wide tiles of the tensor-bound layers.
  const bool halo_fits = h->mode == MODE_BOX && d.stride_h == 1 && d.stride_w == 1 && (d.S == 3 || d.S == 5) && d.pad_w == d.S / 2 &&
                         (dw || d.C > 32) && hint.halo != 0 && d.pool == 0;
  bool halo = false;
  const int halo_segs = halo_segments(d);
  const PatchTile pt = patch_tile(h->Q, h->P, d.pool != 0);
  p.BKC = choose_bkc(c_eff);
  if (is_window_mode(h->mode)) p.BKC = c_eff <= 32 ? 32 : (c_eff <= 64 ? 64 : 128);   // a row is one chunk (two at most)
  const DwTiles dwt = dw ? dw_tiles(h) : DwTiles{};
  if (dw) p.BKC = dwt.bkc;
  p.nchunks = dw ? 1 : ceil_div(c_eff, p.BKC);
  const int b_row = dw ? 32 : p.BKC;                       // bytes of a weight row per chunk
  h->a_channels = d.C;
  p.acc_bufs = 2;
  p.ksplit = 1;
  p.np_products = p.np_cpp = 0;
  if (np) {
    p.np_products = h->np_products = np->products;
    p.np_cpp = p.nchunks;
    p.nchunks *= np->products;
    h->a_channels = np->planes * p.np_cpp * p.BKC;
    for (int m = 0; m < np->products; ++m) { p.np_a[m] = np->a_plane[m]; p.np_coef[m] = np->coef[m]; }
    p.np_n = np->n_out; p.np_p = np->p_out; p.np_top = np->top;
    // Two-digit operands: the conversion in 32 bits (np3_encode) where the largest sum and the smallest shift leave room for it:
    // |v| < 2^(22 + low) and low <= s - 1 for some low >= 7; v / 128 and P0 + bias within an int32.  (Beyond: a sum of 2^33 with
    // a shift below 13, for instance.)
    int low = 7, min_shift = 31;
    while ((np->largest_sum >> low) >= (1ll << 22) - 1) ++low;
    for (int k = 0; k < d.K; ++k) min_shift = std::min(min_shift, shift_host ? shift_host[k] : 0);
    h->np3 = np->products == 3 && np->coef[0] == -127 && np->coef[1] == 16384 - 128 && np->coef[2] == 128 && low <= min_shift - 1 &&
             np->largest_sum < (1ll << 37) && np->largest_bias < (1ll << 30) && hint.float_rounding != 0;
    p.np_low = low - 7;
  }
  p.R = taps_r; p.S = taps_s;
  int bn_max = std::min(2 * qc::kGroupsPerWarp * 16, std::max(16, (hint.bn_max > 0 ? hint.bn_max : 128) / 16 * 16));
  cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
  // Tiles 256 channels wide, one CTA per SM: for tensor-bound layers (long contraction, at least 256 output
  // channels, at least one wave of such tiles).  A stage then feeds MMAs of N = 256: three quarters of the
  // operand bytes per multiply-add of a 128-wide tile, and twice the tensor work per stage, which hides
  // the issuing thread's per-stage instructions.  Only the 16-byte-store epilogues without residual exist
  // in this width.
  bool wide = false;
  {
    const bool shape_ok = (h->mode == MODE_BOX || h->mode == MODE_FLAT || h->mode == MODE_VIEW) && h->fold == 1 && fast_possible &&
                          !d.has_residual && d.out_c_pitch % 16 == 0 && d.out_c_offset % 16 == 0 && k_eff % 16 == 0 && k_eff > 128;
    long m_tiles;
    if (h->mode == MODE_FLAT) {
      m_tiles = ceil_div_l(static_cast<long>(d.N) * h->P * h->Q, 128);
    } else {
      int tq, tp, tn;
      choose_box(h->Q, h->P, d.N, &tq, &tp, &tn, d.pool != 0);
      m_tiles = static_cast<long>(ceil_div(h->Q, tq)) * ceil_div(h->P, tp) * ceil_div(d.N, tn);
    }
    const long contraction = static_cast<long>(taps_r) * taps_s * p.nchunks * p.BKC;
    if (dw) wide = false;
    else if (hint.bn_max > 128) wide = shape_ok;
    else if (hint.bn_max <= 0)
      wide = shape_ok && k_eff >= 256 && contraction >= 2048 && m_tiles * ceil_div(k_eff, 256) >= h->num_sms;
    if (wide) bn_max = 2 * qc::kGroupsPerWarpWide * 16;
    // ... and, with enough of them, 256-pixel tiles on pairs of SMs (each CTA loads half of the weight rows):
    // half the operand bytes per multiply-add of a 128 x 128 tile
    // (measured: worth it from about four rounds of pair tiles over the SM pairs; below that the 128-pixel
    // tiles balance better)
    h->pair = wide && hint.pair_tiles != 0 &&
              (hint.pair_tiles == 1 || ceil_div_l(m_tiles, 2) * ceil_div(k_eff, 256) >= 4L * (h->num_sms / 2));
  }
  if (hint.bn_max <= 0 && k_eff > 64 && !wide && !dw) {
    // A layer with fewer 128-wide tiles than SMs leaves SMs idle while each busy one walks a long
    // chain of MMAs: halve the tile width to spread the work (measured: helps below one wave only).
    long m_tiles;
    if (h->mode == MODE_FLAT || h->mode == MODE_STEM) {
      m_tiles = ceil_div_l(static_cast<long>(d.N) * h->P * h->Q / h->fold, 128);
    } else {
      int tq, tp, tn;
      const int q_rows = is_window_mode(h->mode) ? h->Q / h->fold : h->Q;
      choose_box(q_rows, h->P, d.N, &tq, &tp, &tn, d.pool != 0);
      m_tiles = static_cast<long>(ceil_div(q_rows, tq)) * ceil_div(h->P, tp) * ceil_div(d.N, tn);
    }
    if (m_tiles * ceil_div(k_eff, 128) < h->num_sms) bn_max = 64;
  }
  if (np) {
    // Every product has accumulator columns of its own, side by side: two buffers of them fill the tensor memory as long
    // as products * BN <= 256; five and six products take one buffer (their tiles are long, the epilogue is not).
    const int cols = np->products <= 4 ? 256 : 512;
    bn_max = std::min({bn_max, 128, cols / np->products / 16 * 16});
    p.acc_bufs = np->products <= 4 ? 2 : 1;
    // Few tiles: an MMA of N <= 96 takes the same time whatever its width, so narrower tiles on idle SMs have less to load
    // and less to convert each, for free.
    int tq, tp, tn;
    choose_box(h->Q, h->P, d.N, &tq, &tp, &tn);
    const long m_tiles = h->mode == MODE_FLAT ? ceil_div_l(static_cast<long>(d.N) * h->P * h->Q, 128)
                                              : static_cast<long>(ceil_div(h->Q, tq)) * ceil_div(h->P, tp) * ceil_div(d.N, tn);
    for (int next; hint.bn_max <= 0 && bn_max > 16 && m_tiles * ceil_div(k_eff, next = std::max(16, bn_max / 32 * 16)) <= h->num_sms;) bn_max = next;
  }
  halo = halo_fits && (bn_max <= 64 || k_eff <= 64 || (np && np->products >= 3) || hint.halo == 1);
  if (halo && hint.halo != 1 && !dw) {
    // ... unless its rows' waste makes many more tiles of it, more than run at once; and five weight chunks per stage only
    // where they are small or the layer's CTAs have an SM each.
    int tq, tp, tn, step, bq, bp, bn;
    halo_box(h, &tq, &tp, &tn, &step);
    choose_box(h->Q, h->P, d.N, &bq, &bp, &bn);
    const int tk = ceil_div(k_eff, std::min(bn_max, 64));
    const long halo_tiles = static_cast<long>(ceil_div(h->Q, step)) * ceil_div(h->P, tp) * ceil_div(d.N, tn) * tk;
    const long box_tiles = static_cast<long>(ceil_div(h->Q, bq)) * ceil_div(h->P, bp) * ceil_div(d.N, bn) * tk;
    halo = (halo_tiles <= h->num_sms || halo_tiles * 10 <= box_tiles * 13) && (d.S == 3 || k_eff <= 32 || halo_tiles <= h->num_sms);
  }
  if (dw) {
    bn_max = p.BKC;
    halo = halo_fits && dwt.halo;
  }
  if (halo) {
    wide = false;
    h->pair = 0;
    if (!dw && !(hint.halo == 1 && hint.bn_max >= 128)) bn_max = std::min(bn_max, 64);   // three weight chunks per stage: keep the stage small
    taps_s = 1;                                            // what the kernel's stage loop sees
    p.S = 1;
  }
  // Patch form of a 3 x 3 / stride 1 layer on one chunk of channels: ONE box of (tp + 2) x 16 pixels serves all nine taps
  // (row and column shifts of the same shared-memory rows), against resident weights.  A box per filter row reads every
  // activation three times, a box per tap nine times; where that traffic and not the tensor pipe is the bound (up to 128
  // channels), this is what limits the layer.  us: 64 x 224 x 224 x 64 -> 64 with its pool 167 -> 129, 64 x 112 x 112 x 64
  // -> 128 72 -> 60, x 128 -> 128 with its pool 102 -> 84, 128 x 28 x 28 x 96 -> 128 20.0 -> 14.8, 128 x 14 x 14 x 112 -> 224
  // 14.8 -> 9.1; at one wave of tiles (32 x 28 x 28 x 128 -> 128: 7.2 -> 6.8) it is about even.
  const bool patch_fits = h->mode == MODE_BOX && d.R == 3 && d.S == 3 && d.stride_h == 1 && d.stride_w == 1 && d.pad_h == 1 && d.pad_w == 1 &&
                          p.nchunks == 1 && fast_possible && d.K % 16 == 0 && d.out_c_pitch % 16 == 0 && d.out_c_offset % 16 == 0;
  bool patch = false;
  if (patch_fits && hint.patch_halo != 0 && hint.bn_max <= 0 && hint.halo != 1 && hint.group_taps != 1 && hint.pair_tiles != 1) {
    const long tiles = static_cast<long>(pt.segs) * pt.rows * d.N * ceil_div(k_eff, 128);
    const double used = static_cast<double>(h->Q) * h->P / (static_cast<double>(pt.segs) * pt.rows * 128);
    // from a wave of tiles on, as long as most accumulator rows are outputs and the activations are read for two channel
    // tiles at most
    // ... and at up to 32 channels (rows of 32 bytes) also below a wave, where the one box is one wait instead of three: 32 x 32
    // x 16 -> 16 3.6 -> 3.0 us, 56 x 56 x 32 -> 32 3.3 -> 3.1; with rows of 64 or 128 bytes three boxes are 0.2 us faster there.
    // (Whatever part of a tile the images fill: small ones take a tile each where boxes put several into one, and still gain. us,
    // boxes / patch, 32 channels: 16 x 7 x 7 -> 256 3.6 / 2.8, 64 x 7 x 7 -> 128 3.7 / 3.3, 64 x 4 x 4 -> 256 3.7 / 3.7; at worst 64 x 9 x 5 -> 128
    // 3.7 / 3.9.)
    patch = hint.patch_halo == 1 || (k_eff <= 256 && hint.halo != 0 && hint.resident_weights != 0 &&
                                     ((tiles >= h->num_sms && used >= 0.75) || (p.BKC == 32 && tiles <= h->num_sms)));
  }
  if (dw) patch = !halo && halo_fits && d.S == 3 && hint.patch_halo != 0;
  if (np && halo && d.R == 3 && d.pad_h == 1 && p.np_cpp == 1 && bn_max <= 64 && hint.patch_halo != 0 && hint.halo != 1) {
    // Floating-point operands: a stage of a digit product is a patch and its nine weight chunks.  The layer runs at the rate
    // its operands arrive, so the form with fewer bytes on the busiest SM wins.
    int tq, tp, tn, step;
    halo_box(h, &tq, &tp, &tn, &step);
    auto busiest = [&](long boxes, long activations) {
      return ceil_div_l(boxes * ceil_div(k_eff, bn_max), h->num_sms) * (activations + 9l * bn_max * p.BKC);
    };
    patch = hint.patch_halo == 1 ||
            busiest(static_cast<long>(pt.segs) * pt.rows * d.N, 16l * (pt.tp + 2) * p.BKC) <
                busiest(static_cast<long>(ceil_div(h->Q, step)) * ceil_div(h->P, tp) * ceil_div(d.N, tn), 3l * tq * tp * tn * p.BKC);
  }
  if (patch) {
    wide = false;
    halo = false;
    h->pair = 0;
    // (64 wide only below a wave of its own tiles, which are more than the boxes': 20 x 28 x 28 x 64 -> 128 5.6 us 64 wide, 4.9 128;
    // x 128 -> 128 6.45 / 5.7)
    const bool below_a_wave = static_cast<long>(pt.segs) * pt.rows * d.N * ceil_div(k_eff, 128) < h->num_sms;
    bn_max = dw ? p.BKC : np ? bn_max : bn_max <= 64 && below_a_wave ? 64 : 128;
    taps_r = taps_s = 1;
    p.R = p.S = 1;
  }
  h->patch = patch ? 1 : 0;
  // Grouped taps: on few channels (rows of at most 64 bytes) a ring stage of ONE tap carries one or two
  // MMAs, far less tensor work than the few hundred cycles of instructions a stage costs the issuing
  // thread.  The S taps of a filter row then share a stage -- S activation boxes side by side, S weight
  // chunks -- and the stage loop runs over filter rows only.
  bool group = !halo && !wide && !patch && h->mode == MODE_BOX && d.S >= 2 && d.S <= 4 && p.nchunks == 1 && p.BKC <= 64 &&
               hint.group_taps != 0;
  if (group && hint.group_taps != 1) {
    // ... as long as the fatter stages still form a ring of three, or the weights can stay resident beside
    // two activation stages (the rule applied further down); a ring of two stages costs more than it saves
    const int tk = ceil_div(k_eff, bn_max);
    const int bn = static_cast<int>(align_up(ceil_div(k_eff, tk), 16));
    const int a_tap = static_cast<int>(align_up(static_cast<size_t>(qc::kTileM) * p.BKC, 1024));
    const int b_chunk = static_cast<int>(align_up(static_cast<size_t>(bn) * b_row, 1024));
    const int budget = 113 * 1024 - 1024 - static_cast<int>(sizeof(qc::IgemmShared));
    int tq, tp, tn;
    choose_box(h->Q, h->P, d.N, &tq, &tp, &tn, d.pool != 0);
    const long tiles = static_cast<long>(ceil_div(h->Q, tq)) * ceil_div(h->P, tp) * ceil_div(d.N, tn) * tk;
    const int w_bytes = taps_r * d.S * b_chunk;
    const bool resident = hint.resident_weights != 0 && w_bytes <= 72 * 1024 && (budget - w_bytes) / (d.S * a_tap) >= 2 &&
                          tiles > 2L * h->num_sms;
    group = resident || budget / (d.S * (a_tap + b_chunk)) >= 3;
  }
  if (group) {
    taps_s = 1;
    p.S = 1;
  }
  const int tps = patch ? 9 : halo ? d.S : (group ? d.S : 1);   // taps (weight chunks) per ring stage
  p.halo_s = (halo || group || patch) ? tps : 0;
  p.halo_w = patch ? 3 : std::max(1, tps);
  p.store_rows = 0;
  p.tap_boxes = group ? 1 : 0;
  p.tiles_k = ceil_div(k_eff, bn_max);
  p.BN = dw ? p.BKC : static_cast<int>(align_up(ceil_div(k_eff, p.tiles_k), 16));
  h->kpad = p.tiles_k * p.BN;
  const int all_taps = patch ? 9 : taps_r * taps_s_w;
  h->kg_total = all_taps * p.nchunks * b_row;
  p.K = k_eff;
  p.out_c_offset = d.out_c_offset;
  p.out_c_pitch = h->fold > 1 ? k_eff : d.out_c_pitch;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.BN * std::max(1, p.np_products)) p.tmem_cols *= 2;   // acc_bufs such buffers are allocated
  cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
  h->ctas_per_sm = hint.ctas_per_sm == 1 ? 1 : 2;
  h->use_pdl = hint.pdl != 0 ? 1 : 0;
  if (p.acc_bufs * p.tmem_cols * h->ctas_per_sm > 512 || np) h->ctas_per_sm = 1;
  if (halo) {
    // A halo-form layer with no more tiles than SMs runs one CTA per SM at most: give that CTA the whole
    // shared memory (its stages are large, and its one chain of stages is as fast as the ring is deep).
    int tq, tp, tn, step;
    halo_box(h, &tq, &tp, &tn, &step);
    const long m_tiles = static_cast<long>(halo_segs) * ceil_div(h->P, tp) * ceil_div(d.N, tn);
    if (m_tiles * p.tiles_k <= h->num_sms) h->ctas_per_sm = 1;
  }
  if (!halo && !patch && !dw && !is_window_mode(h->mode) && hint.ctas_per_sm == 0 && taps_r * taps_s * p.nchunks >= 9) {
    // Tiles that all run at once, one per SM, as chains of stages: a chain is as fast as its ring is deep (four stages cover
    // half of the latency of a load), so such a layer's CTAs get the whole shared memory.  Random layers
    // (1 x 1 to 5 x 5 filters, 16 to 1024 channels, 7 to 112 pixels a side) of 2 to 128 tiles and 9 to 175 stages: 0 to
    // 25 % faster, 9 % on average; from 150 tiles on they no longer run at once (1.2 to 1.5 times slower), and with fewer
    // stages the next kernel's set-up beside them is worth more.
    int tq, tp, tn;
    choose_box(h->Q, h->P, d.N, &tq, &tp, &tn, d.pool != 0);
    const long m_tiles = h->mode == MODE_FLAT || h->mode == MODE_STEM ? ceil_div_l(static_cast<long>(d.N) * h->P * h->Q / h->fold, 128)
                                                                      : static_cast<long>(ceil_div(h->Q, tq)) * ceil_div(h->P, tp) * ceil_div(d.N, tn);
    if (m_tiles * p.tiles_k <= h->num_sms) h->ctas_per_sm = 1;
  }
  p.vec_store = (p.out_c_pitch % 16 == 0 && d.out_c_offset % 16 == 0 && k_eff % 16 == 0) ? 1 : 0;
  const long long round_room = h->max_shift > 0 ? (1ll << (h->max_shift - 1)) : 0;
  p.fast_epilogue = (!np && d.out_mode == QCONV_OUT_INT8 && d.rounding == QCONV_ROUND_NEAREST_EVEN && p.vec_store &&
                     d.n_out == 8 &&
                     h->acc_bound + round_room <= 2147483647ll) ? 1 : 0;
  if (hint.fast_epilogue == 0) p.fast_epilogue = 0;
  // (no other epilogue knows the depthwise operands: create_layer takes the tensor cores only where this one serves)
  if (dw && !p.fast_epilogue) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "internal: depthwise on the tensor cores without its epilogue");
  if (p.fast_epilogue || d.out_mode != QCONV_OUT_INT8 || np || dw) h->gen_flt = 0;
  p.gen_down = d.rounding != QCONV_ROUND_NEAREST_EVEN ? 1 : 0;
  p.gen_away = d.rounding == QCONV_ROUND_HALF_AWAY && !d.relu ? 1 : 0;
  // rounding adds at most 2^(s-1) before the shift: in one pass when the accumulator bound leaves that room
  p.gen_simple = h->acc_bound + round_room <= 2147483647ll ? 1 : 0;
  p.gen_stage_bytes = p.fast_epilogue ? 0u : static_cast<uint32_t>((d.has_residual && d.out_mode != QCONV_OUT_INT8 ? 2 : 1) *
                                                                   qc::kEpilogueWarps * qc::kGenWarpBytes);
  // Shared memory: the operand ring, plus -- for the fast epilogues of short contractions, where the
  // epilogue and not the operand ring sets the pace -- staged output tiles that leave by TMA stores:
  // two of them, or three when the residual tile is also brought into them by TMA one tile ahead
  // (as long as the ring keeps enough stages beside them).
  const int full_budget = (h->ctas_per_sm == 2 ? 113 : 226) * 1024 - 1024 - static_cast<int>(sizeof(qc::IgemmShared)) -
                          static_cast<int>(p.gen_stage_bytes);
  const int out_tile = static_cast<int>(align_up(static_cast<size_t>(qc::kTileM) * p.BN, 1024));
  const int patch_a = static_cast<int>(align_up(static_cast<size_t>(qc::kTileM + 2 * 16 + 8) * p.BKC, 1024));
  auto ring_stages = [&](int bkc, int staged_tiles) {
    const int a = patch ? patch_a : static_cast<int>(align_up(static_cast<size_t>(qc::kTileM + (halo ? 8 : 0)) * bkc, 1024)) * (group ? tps : 1);
    const int b = static_cast<int>(align_up(static_cast<size_t>(h->pair ? p.BN / 2 : p.BN) * (dw ? 32 : bkc), 1024)) * tps;
    return (full_budget - staged_tiles * out_tile) / (a + b);
  };
  const bool force_stage = hint.tma_store == 1;
  const bool short_k = taps_r * taps_s * p.nchunks * p.BKC <= 512;
  p.out_stage_bytes = 0;
  p.out_stage_bufs = 2;
  if (p.BN > 128 && !p.fast_epilogue)
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "internal: a tile wider than 128 channels needs a 16-byte-store epilogue");
  // (not for halo tiles of image segments: a staged tile leaves as one box, and the halo's columns are clipped
  // by the tensor's edge only)
  if (p.fast_epilogue && hint.tma_store != 0 && (short_k || force_stage) && p.BN <= 128 && !(halo && halo_segs > 1) && d.pool == 0) {
    const int want[2] = {d.has_residual && h->flt_epilogue && hint.tma_residual != 0 ? 3 : 2, 2};
    for (int w = 0; w < 2 && !p.out_stage_bytes; ++w) {
      const int st = ring_stages(p.BKC, want[w]);
      // (a tile whose operands are one stage needs no second one: the epilogue outlasts the next load)
      if (st >= 1 && (st >= std::min(taps_r * taps_s * p.nchunks, 3) || force_stage)) {
        p.out_stage_bytes = static_cast<uint32_t>(out_tile);
        p.out_stage_bufs = want[w];
      }
    }
  }
  // (patch form: resident weights and at least two activation boxes; two CTAs per SM where they fit, staged tiles where
  // they still do)
  if (patch && !np) {
    const int b_res = 9 * static_cast<int>(align_up(static_cast<size_t>(p.BN) * b_row, 1024));
    const bool may_stage = p.fast_epilogue && hint.tma_store != 0 && (p.BN == 64 || p.BN == 128) && !d.pool && !d.has_residual;
    bool placed = false;
    p.out_stage_bytes = 0;
    for (int ctas : {2, 1}) {
      if (ctas == 2 && (hint.ctas_per_sm == 1 || 4 * p.tmem_cols > 512)) continue;
      const int budget = (ctas == 2 ? 113 : 226) * 1024 - 1024 - static_cast<int>(sizeof(qc::IgemmShared)) - b_res;
      for (int staged : {2, 0}) {
        if (placed || (staged && !may_stage) || (budget - staged * out_tile) / patch_a < 2) continue;
        placed = true;
        h->ctas_per_sm = ctas;
        p.out_stage_bytes = staged ? static_cast<uint32_t>(out_tile) : 0u;
        p.out_stage_bufs = 2;
      }
    }
    if (!placed || !p.fast_epilogue) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "internal: the patch form does not fit");
    p.store_rows = may_stage ? pt.tp : 0;
  }
  const int staged_tiles = p.out_stage_bytes ? p.out_stage_bufs : 0;
  h->kg_total = all_taps * p.nchunks * b_row;
  // (halo form: the shifted operand reads up to two rows past the 128th, and a stage holds three weight chunks)
  p.a_tap_bytes = patch ? static_cast<uint32_t>(patch_a)
                        : static_cast<uint32_t>(align_up(static_cast<size_t>(qc::kTileM + (halo ? 8 : 0)) * p.BKC, 1024));
  p.a_stage_bytes = p.a_tap_bytes * (group ? static_cast<uint32_t>(tps) : 1u);
  p.b_chunk_bytes = static_cast<uint32_t>(align_up(static_cast<size_t>(h->pair ? p.BN / 2 : p.BN) * b_row, 1024));
  p.b_stage_bytes = p.b_chunk_bytes * static_cast<uint32_t>(tps);
  p.out_swz_mask = p.BN == 128 ? 7u : (p.BN == 64 ? 3u : (p.BN == 32 ? 1u : 0u));
  int stages = ring_stages(p.BKC, staged_tiles);
  stages = std::max(staged_tiles ? 1 : 2, std::min(stages, qc::kMaxStages));   // the ring runs on across tiles
  // Resident weights: when a CTA walks several tiles and the weight tile of its channel tile (all
  // chunks) is small, load it once -- before the wait on the previous kernel -- and let the ring carry
  // activations only: half the bytes (and TMA rows) per tile for a 128-wide tile, and a deeper ring.
  const int num_kb_plan = taps_r * taps_s * p.nchunks;
  p.b_resident = 0;
  {
    long m_tiles;
    if (h->mode == MODE_FLAT || h->mode == MODE_STEM) {
      m_tiles = ceil_div_l(static_cast<long>(d.N) * h->P * h->Q / h->fold, 128);
    } else {
      int tq, tp, tn;
      const int q_rows = is_window_mode(h->mode) ? h->Q / h->fold : h->Q;
      choose_box(q_rows, h->P, d.N, &tq, &tp, &tn, d.pool != 0);
      m_tiles = static_cast<long>(ceil_div(q_rows, tq)) * ceil_div(h->P, tp) * ceil_div(d.N, tn);
    }
    const long grid_max = static_cast<long>(h->num_sms) * h->ctas_per_sm;
    const int b_res_bytes = num_kb_plan * static_cast<int>(p.b_stage_bytes);
    const int mode_env = hint.resident_weights;                      // 0: never, 1: whenever it fits
    if (patch && !np) {
      p.b_resident = 1;
      const int budget = (h->ctas_per_sm == 2 ? 113 : 226) * 1024 - 1024 - static_cast<int>(sizeof(qc::IgemmShared));
      stages = std::min((budget - staged_tiles * out_tile - b_res_bytes) / patch_a, qc::kMaxStages);
    } else if (mode_env != 0 && !patch && !h->pair && (!(halo || group) || p.nchunks == 1) && b_res_bytes <= 72 * 1024 &&
        (m_tiles * p.tiles_k > grid_max || mode_env == 1)) {
      const int st = (full_budget - staged_tiles * out_tile - b_res_bytes) / static_cast<int>(p.a_stage_bytes);
      if (st >= std::min(num_kb_plan + 1, 2)) {
        p.b_resident = 1;
        stages = std::min(st, qc::kMaxStages);
      }
    }
  }
  p.stages = stages;
  // (of the widths that the store's box swizzles, 64 only with two CTAs on an SM: with one, whose ring is several times as deep,
  // staging costs 0.2 us: 4 x 28 x 25 x 176 -> 272, 3 x 3 6.2 direct, 6.4 staged; with two 24 x 11 x 28 x 544 -> 128, 1 x 1 4.15 / 3.8)
  h->ring_out_fits = p.fast_epilogue && !p.out_stage_bytes && hint.tma_store != 0 && (p.BN == 128 || (p.BN == 64 && h->ctas_per_sm == 2)) && !h->pair && !d.pool &&
                     !(halo && halo_segs > 1) && !(patch && d.has_residual) &&
                     static_cast<size_t>(stages) * (p.a_stage_bytes + (p.b_resident ? 0 : p.b_stage_bytes)) >= static_cast<size_t>(out_tile);
  h->plan_stage_bytes = p.out_stage_bytes;
  h->plan_stage_bufs = p.out_stage_bufs;
  h->smem_bytes = 1024 + static_cast<size_t>(stages) * (p.a_stage_bytes + (p.b_resident ? 0 : p.b_stage_bytes)) +
                  (p.b_resident ? static_cast<size_t>(num_kb_plan) * p.b_stage_bytes : 0) +
                  static_cast<size_t>(staged_tiles) * p.out_stage_bytes + p.gen_stage_bytes + sizeof(qc::IgemmShared);
  p.stride_h = p.stride_w = 1;
  p.pad_h = p.pad_w = 0;
  if (h->mode == MODE_FLAT || h->mode == MODE_STEM) {
    p.tq = 128; p.tp = 1; p.tn = 1;
  } else if (h->mode == MODE_VIEW) {
    choose_box(h->Q, h->P, d.N, &p.tq, &p.tp, &p.tn, d.pool != 0, static_cast<long>(h->num_sms) * h->ctas_per_sm / p.tiles_k);
  } else if (is_window_mode(h->mode)) {
    choose_box(h->Q / h->fold, h->P, d.N, &p.tq, &p.tp, &p.tn, d.pool != 0);
    p.pad_h = h->s2d_off_h;        // the horizontal offset is built into the packed rows
    // a row's window may run past the image's last pixel: the packed row is long enough for that
    h->s2d_wp = std::max(h->s2d_off_w + h->s2d_w, h->Q - h->fold + ceil_div(p.nchunks * p.BKC, h->win_pb));
    if (h->win_pb % 16) h->s2d_wp += h->s2d_wp & 1;        // the row pitch in bytes is a multiple of 16 as well
  } else {
    choose_box(h->Q, h->P, d.N, &p.tq, &p.tp, &p.tn, d.pool != 0, static_cast<long>(h->num_sms) * h->ctas_per_sm / p.tiles_k);
    if (halo) halo_box(h, &p.tq, &p.tp, &p.tn, &p.q_step);
    if (patch) { p.tq = 16; p.tp = pt.tp; p.tn = 1; p.q_step = pt.q_step; }
    p.pad_h = d.pad_h; p.pad_w = d.pad_w;
    p.stride_h = d.stride_h; p.stride_w = d.stride_w;
  }
  if (!halo && !patch) p.q_step = p.tq;
  p.pool_bit = d.pool ? p.tq : 0;
  if (d.pool && (!p.fast_epilogue || h->mode != MODE_BOX)) {
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "pool: needs the tensor-core path with per-tap boxes and an int8 output at 8 bits "
                "with nearest-even rounding, K %% 16 == 0 and an accumulator bound below 2^31 - 2^(s-1)");
  }
  p.tx_bytes = static_cast<uint32_t>((group ? tps : 1) * p.tq * p.tp * p.tn * p.BKC + (p.b_resident ? 0 : tps * p.BN * b_row));
  if (patch) p.tx_bytes = static_cast<uint32_t>(16 * (p.tp + 2) * p.BKC + (p.b_resident ? 0 : tps * p.BN * b_row));
  p.b_res_tx_bytes = static_cast<uint32_t>(num_kb_plan * tps * p.BN * b_row);
  p.res_tx_bytes = static_cast<uint32_t>(p.tq * p.tp * p.tn * p.BN);

  // weights -> [kpad][kg_total], K-major rows, zero padded (already in that form when nothing is padded or folded)
  const size_t w_bytes = static_cast<size_t>(h->kpad) * h->kg_total;
  const bool as_is = h->fold == 1 && !is_window_mode(h->mode) && h->mode != MODE_STEM && h->kpad == d.K && p.nchunks * p.BKC == d.C &&
                     !np && !dw;
  std::vector<int8_t> wp(as_is || dw ? 0 : w_bytes, 0);
  std::vector<int8_t> row(static_cast<size_t>(std::max(c_row, 1)), 0);
  for (int m = 0; np && m < np->products; ++m)             // [product][chunk] inside a tap
    for (int k = 0; k < d.K; ++k)
      for (int t = 0; t < d.R * d.S; ++t)
        std::memcpy(wp.data() + static_cast<size_t>(k) * h->kg_total + (static_cast<size_t>(t) * p.nchunks + m * p.np_cpp) * p.BKC,
                    np->w[m] + (static_cast<size_t>(k) * d.R * d.S + t) * d.C, d.C);
  for (int k = 0; k < d.K && !as_is && !np && !dw; ++k) {
    const int8_t* src = w_krsc + static_cast<size_t>(k) * d.R * d.S * h->Cg;
    if (h->fold > 1 && !is_window_mode(h->mode)) {
      // one pixel's row as the unfolded GEMM would see it, then once per folded pixel on the diagonal
      std::fill(row.begin(), row.end(), 0);
      if (h->mode == MODE_STEM && h->stem_segp) {
        for (int r = 0; r < d.R; ++r)
          std::memcpy(row.data() + static_cast<size_t>(r) * h->stem_segp, src + static_cast<size_t>(r) * d.S * d.C, d.S * d.C);
      } else if (h->mode == MODE_STEM) {
        std::memcpy(row.data(), src, static_cast<size_t>(d.R) * d.S * d.C);
      } else {
        std::memcpy(row.data(), src, d.C);
      }
      for (int j = 0; j < h->fold; ++j)
        std::memcpy(wp.data() + static_cast<size_t>(j * d.K + k) * h->kg_total + static_cast<size_t>(j) * c_row, row.data(), c_row);
      continue;
    }
    int8_t* dst = wp.data() + static_cast<size_t>(k) * h->kg_total;
    if (h->mode == MODE_WROW) {
      // filter row r of folded output j: tap s at pixel j + s of the window, channels as they are
      for (int j = 0; j < h->fold; ++j) {
        int8_t* dj = wp.data() + static_cast<size_t>(j * d.K + k) * h->kg_total;
        for (int r = 0; r < d.R; ++r)
          for (int sx = 0; sx < d.S; ++sx)
            std::memcpy(dj + static_cast<size_t>(r) * p.nchunks * p.BKC + static_cast<size_t>(j + sx) * h->win_pb,
                        src + (static_cast<size_t>(r) * d.S + sx) * d.C, d.C);
      }
      continue;
    }
    if (h->mode == MODE_S2D) {
      // tap (r, s) sits in block row (r + jh) / 2, block column (s + jw) / 2, at sub-pixel ((r + jh) % 2, (s + jw) % 2)
      const int jh = 2 * h->s2d_off_h - d.pad_h, jw = 2 * h->s2d_off_w - d.pad_w;
      for (int j = 0; j < h->fold; ++j) {                  // folded output j of a row: window shifted by j blocks
        int8_t* dj = wp.data() + static_cast<size_t>(j * d.K + k) * h->kg_total;
        for (int r = 0; r < d.R; ++r)
          for (int sx = 0; sx < d.S; ++sx)
            for (int c = 0; c < d.C; ++c) {
              const int jr = r + jh, js = sx + jw;
              dj[static_cast<size_t>(jr / 2) * p.BKC + (j + js / 2) * 16 + ((jr % 2) * 2 + (js % 2)) * d.C + c] =
                  src[(static_cast<size_t>(r) * d.S + sx) * d.C + c];
            }
      }
      continue;
    }
    if (h->mode == MODE_STEM && h->stem_segp) {
      for (int r = 0; r < d.R; ++r)
        std::memcpy(dst + static_cast<size_t>(r) * h->stem_segp, src + static_cast<size_t>(r) * d.S * d.C, d.S * d.C);
    } else if (h->mode == MODE_STEM) {
      std::memcpy(dst, src, static_cast<size_t>(d.R) * d.S * d.C);
    } else {
      for (int t = 0; t < d.R * d.S; ++t)
        std::memcpy(dst + static_cast<size_t>(t) * p.nchunks * p.BKC, src + static_cast<size_t>(t) * d.C, d.C);
    }
  }
  int rc = QCONV_OK;
  if (dw) parts.reserve(&h->d_w_mma, w_bytes);             // (filled below, from the table of the other kernels)
  else rc = place_weights(h, parts, as_is ? w_krsc : wp.data(), w_bytes, as_is, weights_of);
  if (rc) return rc;
  std::vector<int4> chan(h->kpad, make_int4(0, 0, 0, 0));
  for (int k = 0; k < d.K; ++k) {
    const int sft = shift_host ? shift_host[k] : 0;
    const int t = (d.has_residual && res_lshift_host) ? res_lshift_host[k] : 0;
    chan[k] = make_int4(bias_host ? bias_host[k] : 0, sft, sft > 0 ? (1 << ((sft - 1) & 31)) - 1 : 0,
                        (sft > 0 ? 1 : 0) | ((1 << t) << 1));
    if (np) {                                                // (shifts up to 40)
      if (h->np3) {
        const float scale = std::ldexp(1.0f, p.np_low + 6 - sft);
        std::memcpy(&chan[k].y, &scale, sizeof(int));
      }
      chan[k].z = chan[k].w = 0;
      continue;
    }
    if (d.out_mode == QCONV_OUT_INT8 && !p.fast_epilogue && !h->gen_flt) chan[k].y = sft | t << 8;
    if (h->gen_flt) {
      // {magic + bias + half, bits of 2^-s, half - 1 (half away by sign: not in the bias then), 2^t << 1}
      const float scale = std::ldexp(1.0f, -sft);
      const int half = sft > 0 && (d.rounding == QCONV_ROUND_HALF_AWAY || d.rounding == QCONV_ROUND_HALF_UP) ? 1 << (sft - 1) : 0;
      int bits;
      std::memcpy(&bits, &scale, sizeof(int));
      chan[k] = make_int4(qc::kMagicBits + (bias_host ? bias_host[k] : 0) + (p.gen_away ? 0 : half), bits, half - 1, (1 << t) << 1);
    }
    if (h->flt_epilogue && p.fast_epilogue) {
      // r = (M + v) * 2^-s + M * (1 - 2^-s) with M = 1.5 * 2^23: both constants are exact in binary32
      // for s <= 22; beyond that |v| < 2^22 always rounds to 0, which scale 0 and addend M give
      const float c1 = sft <= 22 ? std::ldexp(1.0f, -sft) : 0.0f;
      const float c2 = static_cast<float>(12582912.0 * (1.0 - static_cast<double>(c1)));
      int c1bits, c2bits;
      std::memcpy(&c1bits, &c1, sizeof(int));
      std::memcpy(&c2bits, &c2, sizeof(int));
      chan[k].x += qc::kMagicBits;
      chan[k].y = c1bits;
      chan[k].z = c2bits;
    }
    // (wide output: the float 2^(e_x + e_w[k]) with the residual's shift in the lowest bits)
    if (d.out_mode != QCONV_OUT_INT8) chan[k].y = (d.out_mode == QCONV_OUT_FLOAT ? ((acc_exp_host ? acc_exp_host[k] : 0) + 127) << 23 : 0) | t;
  }
  for (int j = 1; j < h->fold; ++j)
    for (int k = 0; k < d.K; ++k) chan[static_cast<size_t>(j) * d.K + k] = chan[k];
  parts.add(&h->d_chan, chan.data(), sizeof(int4) * chan.size());
  rc = parts.upload(&h->block, [&] {
    if (!dw) return cudaSuccess;
    const cudaError_t e = parts.copy_now(&h->d_w);
    if (e != cudaSuccess) return e;
    qc::depthwise_blocks_kernel<<<ceil_div(h->kpad * 18, 256), 256>>>(h->d_w, reinterpret_cast<uint4*>(h->d_w_mma), d.C, h->kpad);
    return cudaGetLastError();
  });
  if (rc) return rc;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(h->kg_total), static_cast<cuuint64_t>(h->kpad)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(h->kg_total)};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(b_row), static_cast<cuuint32_t>(h->pair ? p.BN / 2 : p.BN)};
  rc = encode_map(&h->tmap_b, dw ? h->d_w_mma : h->d_w, 2, dims, strides, box, b_row);
  if (rc) return rc;
  size_t pack_bytes = 0;
  if (is_window_mode(h->mode)) pack_bytes = static_cast<size_t>(d.N) * h->s2d_h * h->s2d_wp * h->win_pb;
  if (h->mode == MODE_STEM) pack_bytes = static_cast<size_t>(d.N) * h->P * h->Q * h->kg_pad;
  if (pack_bytes) {
    // cleared once: padding pixels, ragged edges and the padding bytes of each row stay zero
    CUDA_TRY(DevicePool::pool().take(&h->pack, pack_bytes));
    h->d_pack = static_cast<int8_t*>(h->pack.ptr);
    CUDA_TRY(cudaMemsetAsync(h->d_pack, 0, pack_bytes, nullptr));
    CUDA_TRY(cudaStreamSynchronize(nullptr));              // (the stream of the first run need not wait for this one)
  }
  // the attribute belongs to the current device: once per device, not once per process
  static qc::PerDevice<cudaError_t> attrs;
  const cudaError_t attr_err = attrs.once(h->device, [] {
    for (IgemmKernel k : {static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FAST_I8>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FAST_I8_RES>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8, 0>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES, 0>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 0>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES_U, 0>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8, 1>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES, 1>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 1>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES_U, 1>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES, 0, 1>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES_U, 0, 1>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES, 1, 1>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES_U, 1, 1>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FAST_I8_U>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FAST_I8_RES_U>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 1, 0, qc::kGroupsPerWarpWide>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8, 1, 0, qc::kGroupsPerWarpWide>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 0, 0, qc::kGroupsPerWarpWide>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8, 0, 0, qc::kGroupsPerWarpWide>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FAST_I8_U, 2, 0, qc::kGroupsPerWarpWide>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FAST_I8, 2, 0, qc::kGroupsPerWarpWide>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_I8>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 0, 5>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8, 0, 5>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 1, 5>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8, 1, 5>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_GEN>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_GEN_RES>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_I32>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_F32>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_MAX>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_NP>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_NP3, 0>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_NP3, 1>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 2, 4>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8, 2, 4>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES_U, 2, 4>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES, 2, 4>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FAST_I8_U, 2, 4>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FAST_I8, 2, 4>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FAST_I8_RES_U, 2, 4>),
                          static_cast<IgemmKernel>(qc::igemm_i8_kernel<qc::EPI_FAST_I8_RES, 2, 4>)}) {
      const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  });
  if (attr_err != cudaSuccess)
    return fail(QCONV_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(attr_err));
  if (h->pair) {
    PairKernel pk = pair_kernel_for(h);
    CUDA_TRY(cudaFuncSetAttribute(pk, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  } else if (d.pool) {
    CUDA_TRY(cudaFuncSetAttribute(igemm_kernel_for(h), cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  }
  return QCONV_OK;
}

PairKernel pair_kernel_for(const qconv_handle* h) {
  const bool uni = h->uniform_shift && h->hints.uniform_shift != 0;
  if (h->d.pool) {
    if (h->flt_epilogue) return uni ? qc::igemm_i8_pair_kernel<qc::EPI_FLT_I8_U, 2, 1> : qc::igemm_i8_pair_kernel<qc::EPI_FLT_I8, 2, 1>;
    return uni ? qc::igemm_i8_pair_kernel<qc::EPI_FAST_I8_U, 2, 1> : qc::igemm_i8_pair_kernel<qc::EPI_FAST_I8, 2, 1>;
  }
  if (h->flt_epilogue) {
    if (h->d.relu) return uni ? qc::igemm_i8_pair_kernel<qc::EPI_FLT_I8_U, 1> : qc::igemm_i8_pair_kernel<qc::EPI_FLT_I8, 1>;
    return uni ? qc::igemm_i8_pair_kernel<qc::EPI_FLT_I8_U, 0> : qc::igemm_i8_pair_kernel<qc::EPI_FLT_I8, 0>;
  }
  return uni ? qc::igemm_i8_pair_kernel<qc::EPI_FAST_I8_U, 2> : qc::igemm_i8_pair_kernel<qc::EPI_FAST_I8, 2>;
}

IgemmKernel igemm_kernel_for(const qconv_handle* h, bool maxabs) {
  if (maxabs) return qc::igemm_i8_kernel<qc::EPI_MAX>;
  if (h->np3) return h->d.relu ? qc::igemm_i8_kernel<qc::EPI_NP3, 1> : qc::igemm_i8_kernel<qc::EPI_NP3, 0>;
  if (h->np_products) return qc::igemm_i8_kernel<qc::EPI_NP>;
  if (h->d.out_mode == QCONV_OUT_INT32) return qc::igemm_i8_kernel<qc::EPI_I32>;
  if (h->d.out_mode == QCONV_OUT_FLOAT) return qc::igemm_i8_kernel<qc::EPI_F32>;
  if (!h->prm.fast_epilogue) {
    if (h->gen_flt) return h->d.has_residual || h->prm.gen_away ? qc::igemm_i8_kernel<qc::EPI_GEN_RES> : qc::igemm_i8_kernel<qc::EPI_GEN>;
    return qc::igemm_i8_kernel<qc::EPI_I8>;
  }
  const bool uni = h->uniform_shift && h->hints.uniform_shift != 0;
  if (h->dw_mma) {
    constexpr int G = qc::kGroupsPerWarp;
    if (h->d.relu) return uni ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 1, 5, G> : qc::igemm_i8_kernel<qc::EPI_FLT_I8, 1, 5, G>;
    return uni ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 0, 5, G> : qc::igemm_i8_kernel<qc::EPI_FLT_I8, 0, 5, G>;
  }
  if (h->d.pool) {                                         // 2 x 2 max-pool in the epilogue (ReLU read at run time)
    constexpr int W = qc::kGroupsPerWarpWide;
    if (h->prm.BN > 128) {
      if (h->flt_epilogue) return uni ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 2, 2, W> : qc::igemm_i8_kernel<qc::EPI_FLT_I8, 2, 2, W>;
      return uni ? qc::igemm_i8_kernel<qc::EPI_FAST_I8_U, 2, 2, W> : qc::igemm_i8_kernel<qc::EPI_FAST_I8, 2, 2, W>;
    }
    if (h->flt_epilogue) return uni ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 2, 2> : qc::igemm_i8_kernel<qc::EPI_FLT_I8, 2, 2>;
    return uni ? qc::igemm_i8_kernel<qc::EPI_FAST_I8_U, 2, 2> : qc::igemm_i8_kernel<qc::EPI_FAST_I8, 2, 2>;
  }
  if (h->prm.BN > 128) {                                   // 256-wide tiles: no residual (the planner saw to that)
    constexpr int W = qc::kGroupsPerWarpWide;
    if (h->flt_epilogue) {
      if (h->d.relu) return uni ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 1, 0, W> : qc::igemm_i8_kernel<qc::EPI_FLT_I8, 1, 0, W>;
      return uni ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 0, 0, W> : qc::igemm_i8_kernel<qc::EPI_FLT_I8, 0, 0, W>;
    }
    return uni ? qc::igemm_i8_kernel<qc::EPI_FAST_I8_U, 2, 0, W> : qc::igemm_i8_kernel<qc::EPI_FAST_I8, 2, 0, W>;
  }
  if (h->flt_epilogue) {
    const bool res = h->d.has_residual != 0;
    if (res && h->prm.out_stage_bytes && h->prm.out_stage_bufs == 3) {      // residual tiles arrive by TMA
      if (h->d.relu) return uni ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES_U, 1, 1> : qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES, 1, 1>;
      return uni ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES_U, 0, 1> : qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES, 0, 1>;
    }
    if (h->d.relu) {
      if (uni) return res ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES_U, 1> : qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 1>;
      return res ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES, 1> : qc::igemm_i8_kernel<qc::EPI_FLT_I8, 1>;
    }
    if (uni) return res ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES_U, 0> : qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 0>;
    return res ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES, 0> : qc::igemm_i8_kernel<qc::EPI_FLT_I8, 0>;
  }
  if (uni)
    return h->d.has_residual ? qc::igemm_i8_kernel<qc::EPI_FAST_I8_RES_U> : qc::igemm_i8_kernel<qc::EPI_FAST_I8_U>;
  return h->d.has_residual ? qc::igemm_i8_kernel<qc::EPI_FAST_I8_RES> : qc::igemm_i8_kernel<qc::EPI_FAST_I8>;
}

// CTAs that share a tile's contraction in this run (1: none).
int choose_ksplit(const qconv_handle* h, long tiles) {
  const qc::IgemmParams& p = h->prm;
  const int num_kb = p.R * p.S * p.nchunks, groups = p.BN / 16, want = h->hints.split_k;
  if (!p.fast_epilogue || h->d.pool || p.b_resident || h->pair || h->dw_mma || p.BN > 128 || want == 0) return 1;
  auto fits = [&](int ks) { return groups % ks == 0 && tiles * ks <= h->num_sms && num_kb >= ks; };
  if (want > 0) return (want == 2 || want == 4) && fits(want) ? want : 1;
  // A stage of a chain costs a quarter of a microsecond, one of three taps 0.4, the exchange about one.  In these units (2
  // and 3 a stage) halves pay from 18 on (6 three-tap stages: 4.6 -> 4.3 us; 8 single ones: 4.0 either way), quarters from
  // 16 on while the clusters fill half of the SMs at most: with more, the next kernel's CTAs find no room to set up beside
  // them (14 x 14 x 256 3 x 3 on 16 tiles 4.6 -> 4.0, on 28 tiles 4.7 -> 5.1).
  const int work = num_kb * (p.halo_s ? std::max(3, p.halo_s) : 2);
  if (work >= 16 && fits(4) && tiles * 8 <= h->num_sms) return 4;
  if (work >= 18 && fits(2)) return 2;
  return 1;
}

IgemmKernel split_kernel_for(const qconv_handle* h) {
  const bool uni = h->uniform_shift && h->hints.uniform_shift != 0, res = h->d.has_residual != 0;
  if (h->flt_epilogue) {
    if (uni) return res ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES_U, 2, 4> : qc::igemm_i8_kernel<qc::EPI_FLT_I8_U, 2, 4>;
    return res ? qc::igemm_i8_kernel<qc::EPI_FLT_I8_RES, 2, 4> : qc::igemm_i8_kernel<qc::EPI_FLT_I8, 2, 4>;
  }
  if (uni) return res ? qc::igemm_i8_kernel<qc::EPI_FAST_I8_RES_U, 2, 4> : qc::igemm_i8_kernel<qc::EPI_FAST_I8_U, 2, 4>;
  return res ? qc::igemm_i8_kernel<qc::EPI_FAST_I8_RES, 2, 4> : qc::igemm_i8_kernel<qc::EPI_FAST_I8, 2, 4>;
}

// Activation tensor map and tile counts for this run (depends on the pointer and n_run).
int prepare_a_map(qconv_handle* h, const int8_t* a_ptr, int n_run) {
  if (h->a_key_ptr == a_ptr && h->a_key_n == n_run) return QCONV_OK;
  const qconv_desc& d = h->d;
  qc::IgemmParams& p = h->prm;
  const cuuint64_t ac = static_cast<cuuint64_t>(h->a_channels);
  cuuint64_t dims[4], strides[3];
  cuuint32_t estr[4] = {1, 1, 1, 1};
  cuuint32_t box[4] = {static_cast<cuuint32_t>(p.BKC), static_cast<cuuint32_t>(p.tq),
                       static_cast<cuuint32_t>(p.tp), static_cast<cuuint32_t>(p.tn)};
  if (h->mode == MODE_FLAT || h->mode == MODE_STEM) {
    const cuuint64_t c = static_cast<cuuint64_t>(h->mode == MODE_STEM ? h->kg_pad : ac) * h->fold;
    const cuuint64_t m = static_cast<cuuint64_t>(n_run) * h->P * h->Q / h->fold;
    dims[0] = c; dims[1] = m; dims[2] = 1; dims[3] = 1;
    strides[0] = c; strides[1] = m * c; strides[2] = m * c;
    p.Q = static_cast<int>(m); p.P = 1; p.Nimg = 1;
  } else if (is_window_mode(h->mode)) {
    // overlapping view of the packed block pixels: GEMM row q of a filter block row is the BKC bytes that
    // start at packed pixel q (pitch 16 bytes), i.e. blocks q - off_w ... of the image
    const cuuint64_t pb = static_cast<cuuint64_t>(h->win_pb);
    dims[0] = static_cast<cuuint64_t>(p.nchunks) * p.BKC; dims[1] = h->Q / h->fold; dims[2] = h->s2d_h; dims[3] = n_run;
    strides[0] = pb * h->fold;
    strides[1] = pb * h->s2d_wp;
    strides[2] = pb * h->s2d_wp * h->s2d_h;
    p.Q = h->Q / h->fold; p.P = h->P; p.Nimg = n_run;
  } else if (h->mode == MODE_VIEW) {
    dims[0] = ac; dims[1] = h->Q; dims[2] = h->P; dims[3] = n_run;
    strides[0] = static_cast<cuuint64_t>(d.stride_w) * ac;
    strides[1] = static_cast<cuuint64_t>(d.stride_h) * d.W * ac;
    strides[2] = static_cast<cuuint64_t>(d.H) * d.W * ac;
    p.Q = h->Q; p.P = h->P; p.Nimg = n_run;
  } else {
    dims[0] = ac; dims[1] = d.W; dims[2] = d.H; dims[3] = n_run;
    strides[0] = ac;
    strides[1] = static_cast<cuuint64_t>(d.W) * ac;
    strides[2] = static_cast<cuuint64_t>(d.H) * d.W * ac;
    p.Q = h->Q; p.P = h->P; p.Nimg = n_run;
    // strided filters: the box spans (t - 1) * stride + 1 input pixels per axis and the copy engine keeps
    // every stride-th one (traversal strides of the tensor map), so the tile still has tq x tp rows
    estr[1] = static_cast<cuuint32_t>(d.stride_w); estr[2] = static_cast<cuuint32_t>(d.stride_h);
    box[1] = static_cast<cuuint32_t>((p.tq - 1) * d.stride_w + 1);
    box[2] = static_cast<cuuint32_t>((p.tp - 1) * d.stride_h + 1);
    if (p.halo_s && !p.tap_boxes) box[1] = static_cast<cuuint32_t>(p.tq);
    if (h->patch) box[2] = static_cast<cuuint32_t>(p.tp + 2);
  }
  p.tiles_q = ceil_div(p.Q, p.q_step);
  p.tiles_p = ceil_div(p.P, p.tp);
  p.tiles_n = ceil_div(p.Nimg, p.tn);
  h->walk_grid = -1;                                       // the walk's digits depend on the tile counts too
  p.fd_tiles_k = make_fastdiv(p.tiles_k); p.fd_tiles_q = make_fastdiv(p.tiles_q); p.fd_tiles_p = make_fastdiv(p.tiles_p);
  p.fd_tq = make_fastdiv(p.tq); p.fd_tp = make_fastdiv(p.tp);
  p.fd_nchunks = make_fastdiv(p.nchunks); p.fd_S = make_fastdiv(p.S);
  p.fd_np_cpp = make_fastdiv(std::max(1, p.np_cpp));
  int rc = encode_map(&h->tmap_a, a_ptr, 4, dims, strides, box, p.BKC, estr);
  if (rc) return rc;
  h->a_key_ptr = a_ptr;
  h->a_key_n = n_run;
  return QCONV_OK;
}

// How this run's output tiles leave (fast epilogues).  As planned, beside the ring; or, where the plan has no room for that (long
// contractions) and every CTA has one tile, staged in the ring, which is idle once the accumulators are complete: staged tiles
// take the lean epilogue and leave by TMA in whole rows, where 32 lanes storing 16 bytes of 32 rows each touch 32 half sectors per
// instruction (32 x 28 x 28 x 512 -> 128, 1 x 1: 6.05 -> 5.8 us; 128 x 14 x 14 x 512 -> 128 6.1 -> 5.8).  Up to a third of the SMs'
// worth of tiles is stored by the threads themselves whatever the plan: there it is the chain of one tile that counts, and
// barrier, TMA store and its wait lengthen it (us per launch, staged / direct: 14 tiles of 28 x 28 x 512 -> 128, 1 x 1 3.1 / 2.9; 32
// of 7 x 7 x 512 -> 2048 with residual 3.4 / 3.15; 56 of 28 x 28 x 128 -> 512 2.7 / 2.8; 100 of 56 x 56 x 64 -> 256 2.85 / 3.06;
// ResNet-50 on one image 195.2 -> 191.7).  The patch form, whose tiles leave by one store per image row, as long as every CTA has one
// tile: 3 x 3, 32 channels, 64 x 9 x 5 -> 256 4.3 -> 3.9, 110 x 5 x 5 -> 128 4.0 -> 3.5; 20 x 28 x 28 x 64 -> 64 4.3 -> 3.8.
void plan_staging(qconv_handle* h, long tiles) {
  qc::IgemmParams& p = h->prm;
  if (!p.fast_epilogue) return;
  uint32_t bytes = h->plan_stage_bytes;
  int bufs = h->plan_stage_bufs;
  const long one_each = static_cast<long>(h->num_sms) * h->ctas_per_sm;
  if (!bytes && h->ring_out_fits && tiles <= one_each) {
    bytes = static_cast<uint32_t>(align_up(static_cast<size_t>(qc::kTileM) * p.BN, 1024));
    bufs = 0;
  }
  const long most = h->patch ? one_each : h->num_sms / 3;
  if (tiles <= most && h->hints.tma_store != 1) bytes = 0;
  if (bytes != p.out_stage_bytes) h->y_key_ptr = h->r_key_ptr = nullptr;
  p.out_stage_bytes = bytes;
  p.out_stage_bufs = bufs;
}

// Output tensor map for the TMA stores of the fast epilogues: the same pixel boxes as the accumulator
// rows (q fastest, then p, then image), BN channels wide, over the caller's buffer with its channel
// offset and pitch.  Must follow prepare_a_map (which sets the run's pixel extents).
int prepare_y_map(qconv_handle* h, const void* y_ptr, int n_run) {
  if (h->y_key_ptr == y_ptr && h->y_key_n == n_run) return QCONV_OK;
  const qc::IgemmParams& p = h->prm;
  const cuuint64_t pitch = static_cast<cuuint64_t>(p.out_c_pitch);
  cuuint64_t dims[4] = {static_cast<cuuint64_t>(p.K), static_cast<cuuint64_t>(p.Q), static_cast<cuuint64_t>(p.P),
                        static_cast<cuuint64_t>(p.Nimg)};
  cuuint64_t strides[3] = {pitch, pitch * p.Q, pitch * p.Q * p.P};
  cuuint32_t box[4] = {static_cast<cuuint32_t>(p.BN), static_cast<cuuint32_t>(p.tq), static_cast<cuuint32_t>(p.tp),
                       static_cast<cuuint32_t>(p.tn)};
  if (p.store_rows) { box[1] = static_cast<cuuint32_t>(p.q_step); box[2] = 1; }
  const int swz = (p.BN == 128 || p.BN == 64 || p.BN == 32) ? p.BN : 0;
  int rc = encode_map(&h->tmap_y, static_cast<const int8_t*>(y_ptr) + p.out_c_offset, 4, dims, strides, box, swz);
  if (rc) return rc;
  h->y_key_ptr = y_ptr;
  h->y_key_n = n_run;
  return QCONV_OK;
}

int prepare_r_map(qconv_handle* h, const void* r_ptr, int n_run) {
  if (h->r_key_ptr == r_ptr && h->r_key_n == n_run) return QCONV_OK;
  const qc::IgemmParams& p = h->prm;
  const cuuint64_t pitch = static_cast<cuuint64_t>(p.K);
  cuuint64_t dims[4] = {static_cast<cuuint64_t>(p.K), static_cast<cuuint64_t>(p.Q), static_cast<cuuint64_t>(p.P),
                        static_cast<cuuint64_t>(p.Nimg)};
  cuuint64_t strides[3] = {pitch, pitch * p.Q, pitch * p.Q * p.P};
  cuuint32_t box[4] = {static_cast<cuuint32_t>(p.BN), static_cast<cuuint32_t>(p.tq), static_cast<cuuint32_t>(p.tp),
                       static_cast<cuuint32_t>(p.tn)};
  const int swz = (p.BN == 128 || p.BN == 64 || p.BN == 32) ? p.BN : 0;
  int rc = encode_map(&h->tmap_r, r_ptr, 4, dims, strides, box, swz);
  if (rc) return rc;
  h->r_key_ptr = r_ptr;
  h->r_key_n = n_run;
  return QCONV_OK;
}

// Tile shape of the TMA-staged depthwise kernel: the channel width of a CTA trades idle columns
// (few wide column groups on a narrow image) against halo re-reads (many narrow ones).
void plan_dw_tma(qconv_handle* h) {
  const qconv_desc& d = h->d;
  const int st = d.stride_h;
  double best = 0.0;
  qc::DwTmaParams bp = {};
  for (int cwb = 8; cwb <= 128 && cwb * 4 <= d.C; cwb *= 2) {
    if ((d.C / 4) % cwb) continue;
    qc::DwTmaParams p = {};
    p.cwb = cwb;
    p.cwb_box = std::min(cwb, 64);
    p.nbox = cwb / p.cwb_box;
    const int qt_max = qc::kDwConsumers / cwb;
    p.q_blocks = ceil_div(ceil_div(h->Q, 4), qt_max);
    p.qt_per_cta = ceil_div(ceil_div(h->Q, 4), p.q_blocks);          // even split, no more columns than needed
    p.consumers = ceil_div(p.qt_per_cta * cwb, 32) * 32;
    p.pix = 4 * p.qt_per_cta * st + 3 - st;
    if (p.pix > 256) continue;
    p.box_words = p.pix * p.cwb_box;
    p.row_bytes = p.nbox * p.box_words * 4;
    p.stage_bytes = static_cast<int>(align_up(p.row_bytes, 128));
    const double threads = static_cast<double>(p.q_blocks) * p.qt_per_cta * 4 / h->Q;     // >= 1: idle columns
    const double bytes = static_cast<double>(p.q_blocks) * p.pix / (static_cast<double>(h->Q) * st);   // >= 1: halo + overhang
    const double cost = threads * bytes;
    if (bp.cwb == 0 || cost <= best) { best = cost; bp = p; }
  }
  if (bp.cwb == 0) return;
  while ((1 << bp.cwb_log2) < bp.cwb) ++bp.cwb_log2;
  while ((1 << bp.cwb_box_log2) < bp.cwb_box) ++bp.cwb_box_log2;
  bp.fd_q_blocks = make_fastdiv(bp.q_blocks);
  h->dw_prm = bp;
  h->dw_tma = 1;
}

size_t dw_mma_smem(const qc::DwMmaParams& p) {
  return 1024 + static_cast<size_t>(qc::kDwMmaStages) * p.stage_bytes + sizeof(qc::DwMmaShared);
}

// CTAs of that kernel on an SM: 16 warps at 128 registers a thread, 227 KB of shared memory.  (Five warps: three.  Strips chosen for
// two: 128 x 72 x 72 x 32 24.0 -> 17.1 us, 64 x 75 x 75 x 96 34.2 -> 25.9, 64 x 33 x 65 x 128 22.3 -> 17.6.)
int dw_mma_ctas_per_sm(const qc::DwMmaParams& p) {
  return static_cast<int>(std::max<size_t>(1, std::min<size_t>(16 / p.warps, 227 * 1024 / (dw_mma_smem(p) + 1024))));
}

using DwMmaKernel = decltype(&qc::depthwise3x3_mma_kernel<1, true, true>);
constexpr DwMmaKernel kDwMmaKernels[2][2][2] = {             // [stride - 1][one scale for all channels][ReLU]
    {{qc::depthwise3x3_mma_kernel<1, false, false>, qc::depthwise3x3_mma_kernel<1, false, true>},
     {qc::depthwise3x3_mma_kernel<1, true, false>, qc::depthwise3x3_mma_kernel<1, true, true>}},
    {{qc::depthwise3x3_mma_kernel<2, false, false>, qc::depthwise3x3_mma_kernel<2, false, true>},
     {qc::depthwise3x3_mma_kernel<2, true, false>, qc::depthwise3x3_mma_kernel<2, true, true>}}};

// Their shared memory, at creation: the attribute belongs to the current device, which then is the handle's.
int allow_dw_mma_smem(int device) {
  static qc::PerDevice<cudaError_t> attrs;
  CUDA_TRY(attrs.once(device, [] {
    for (const auto& by_stride : kDwMmaKernels)
      for (const auto& by_scale : by_stride)
        for (DwMmaKernel k : by_scale) {
          const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024);
          if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
  }));
  return QCONV_OK;
}

// Output rows per strip of that kernel: a CTA's fixed cost is about six rows' worth (set-up, filling its ring), its halo two
// rows.  The strip length whose rounds of CTAs take the fewest rows in all; it depends on the batch alone and is kept with it (the
// search takes the host 0.4 us at 112 rows, 22 at 8192).
void plan_dw_mma_strips(qconv_handle* h, int n_run) {
  if (h->dw_rows_n == n_run) return;
  qc::DwMmaParams& p = h->dw_mma_prm;
  const long columns = static_cast<long>(ceil_div(h->d.C, p.cb)) * p.q_blocks * ceil_div(n_run, p.images);
  const long slots = static_cast<long>(dw_mma_ctas_per_sm(p)) * h->num_sms;
  long best = -1;
  for (int strips = 1; strips <= std::max(1, h->P / 2); ++strips) {
    const int rows = ceil_div(h->P, strips);
    if (ceil_div(h->P, rows) != strips) continue;
    const long cost = ceil_div_l(columns * strips, slots) * ((rows - 1) * h->d.stride_h + 3 + 6);
    if (best < 0 || cost < best) { best = cost; p.rows_per_cta = rows; }
  }
  h->dw_rows_n = n_run;
}

// Tile of the depthwise kernel on warp-level matrix instructions: eight warps, each 32 channels x two groups of 8 pixels, over
// 32, 64 or 128 channels; narrow images share a CTA.  The width whose padding (channels, groups, halo columns) costs least.
// Unless `whatever_it_costs`, none where a third of the work would be padding and rows are narrow: 64 x 33 x 33 x 512 stride 2 14.4 us
// against tcgen05's 11.8, 128 x 36 x 36 x 128 stride 2 8.4 against 7.7 (128 channels wide it is faster all the same: 128 x 9 x 9 x 512 at
// a cost of 1.84 7.8 against 8.3).
void plan_dw_mma(qconv_handle* h, bool whatever_it_costs) {
  const qconv_desc& d = h->d;
  const int st = d.stride_h;
  double best = 0.0;
  qc::DwMmaParams bp = {};
  for (int cb : {128, 64, 32}) {
    qc::DwMmaParams p = {};
    p.cb = cb;
    p.swz_mask = cb / 16 - 1;
    const int wc = cb / 32, all = ceil_div(h->Q, 8);
    int most = 2 * (qc::kDwMmaWarps / wc);
    while (most * 8 * st + 3 - st > 256) --most;           // (a copy's box spans at most 256 pixels)
    p.q_blocks = ceil_div(all, most);
    p.groups = ceil_div(all, p.q_blocks);
    p.images = p.q_blocks > 1 ? 1 : std::max(1, std::min(d.N, most / p.groups));
    p.pix = p.groups * 8 * st + 3 - st;
    p.warps = ceil_div(p.groups * p.images, 2) * wc;
    p.row_bytes = p.images * p.pix * cb;
    p.stage_bytes = static_cast<int>(align_up(p.row_bytes, 1024));
    const double channels = static_cast<double>(align_up(d.C, cb)) / d.C;
    const double pixels = static_cast<double>(p.q_blocks) * (p.warps / wc) * 16 / (static_cast<double>(h->Q) * p.images);
    const double halo = static_cast<double>(p.pix) / (p.groups * 8 * st);
    const double cost = channels * pixels * (0.7 + 0.3 * halo);
    if (bp.cb == 0 || cost < best * 0.999) { best = cost; bp = p; }
  }
  if (!whatever_it_costs && bp.cb < 128 && best > 1.3) return;
  while ((32 << bp.wc_log2) < bp.cb) ++bp.wc_log2;
  bp.fd_q_blocks = make_fastdiv(bp.q_blocks);
  bp.fd_groups = make_fastdiv(bp.groups);
  bp.lo = d.relu ? 0 : h->lo;
  const float c1 = h->uni_s <= 22 ? std::ldexp(1.0f, -h->uni_s) : 0.0f;
  bp.c1 = c1;
  bp.c2 = static_cast<float>(12582912.0 * (1.0 - static_cast<double>(c1)));
  h->dw_mma_prm = bp;
  h->dw_warp = 1;
}

// Whether tcgen05 takes a large layer in clearly less time than the kernel on warp-level instructions, by a model of both in us,
// fitted to 130 layers of 1 to 115 million outputs (it meets their times within 5 and 7 %).  Warp level: the busiest SM's rows of
// CTAs at the rate of 16 warps, or the rounds of CTAs at a CTA's own pace where there are fewer warps, and the bytes; tcgen05: its
// tiles.  Narrow images leave the groups of 8 columns partly empty, few CTAs more than the SMs hold leave most of them idle.
// us, warp level / tcgen05: 212 x 41 x 9 x 512 stride 2 19.8 / 12.8, 96 x 28 x 28 x 256 18.8 / 15.2, 200 x 10 x 10 x 512 13.7 / 11.0, 128 x 36 x 36 x 128
// 18.5 / 16.5, 128 x 28 x 28 x 512 38.0 / 32.0; the other way round 64 x 28 x 28 x 576 19.9 / 23.5, 128 x 14 x 14 x 512 11.0 / 12.9.  Stride 1 keeps a
// margin: between other layers, short CTAs without a tail are worth a few us (MobileNet-v1, batch 256, with its 56 x 56 x 128 or
// its 14 x 14 x 512 layers on tcgen05: + 6 and + 20 us of 774, where alone these take 71 and 19 there, 69 and 21 here).
bool dw_tcgen05_wins(qconv_handle* h) {
  const qconv_desc& d = h->d;
  plan_dw_mma_strips(h, d.N);
  const qc::DwMmaParams& p = h->dw_mma_prm;
  const bool s1 = d.stride_h == 1;
  const double mb = 1e-6 * d.N * d.C * (static_cast<double>(d.H) * d.W + static_cast<double>(h->P) * h->Q);
  const long ctas = static_cast<long>(ceil_div(d.C, p.cb)) * p.q_blocks * ceil_div(d.N, p.images) * ceil_div(h->P, p.rows_per_cta);
  const double rows = (p.rows_per_cta - 1) * d.stride_h + 3;
  const double busiest = ceil_div_l(ctas, h->num_sms) * p.warps / 16.0, rounds = ceil_div_l(ctas, static_cast<long>(h->num_sms) * dw_mma_ctas_per_sm(p));
  const double warp_level = s1 ? 0.8 + std::max(0.50 * busiest, 0.45 * rounds) * (rows + 1.3) + 0.065 * mb
                               : 1.2 + std::max(0.337 * busiest, 0.308 * rounds) * (rows + 2.3) + 0.05 * mb;
  const double budget = (s1 ? 0.90 : 0.97) * warp_level - 4.0;
  if (budget <= 0.0) return false;
  const DwTiles t = dw_tiles(h);
  return static_cast<double>(t.tiles) / h->num_sms * (!s1 ? 1.08 : t.bkc == 128 ? 1.23 : 0.77) < budget;
}

// Box of the depthwise kernels' row copies: `channels` x `pixels` x one row x `images`.
int prepare_dw_map(qconv_handle* h, const int8_t* x, int n_run, int channels, int pixels, int images, int swizzle) {
  const int form = channels + 1024 * swizzle;
  if (h->dw_key_ptr == x && h->dw_key_n == n_run && h->dw_key_form == form) return QCONV_OK;
  const qconv_desc& d = h->d;
  cuuint64_t dims[4] = {static_cast<cuuint64_t>(d.C), static_cast<cuuint64_t>(d.W), static_cast<cuuint64_t>(d.H),
                        static_cast<cuuint64_t>(n_run)};
  cuuint64_t strides[3] = {static_cast<cuuint64_t>(d.C), static_cast<cuuint64_t>(d.W) * d.C,
                           static_cast<cuuint64_t>(d.H) * d.W * d.C};
  cuuint32_t box[4] = {static_cast<cuuint32_t>(channels), static_cast<cuuint32_t>(pixels), 1, static_cast<cuuint32_t>(images)};
  int rc = encode_map(&h->dw_map, x, 4, dims, strides, box, swizzle);
  if (rc) return rc;
  h->dw_key_ptr = x;
  h->dw_key_n = n_run;
  h->dw_key_form = form;
  return QCONV_OK;
}

// Launch with the programmatic-dependent-launch attribute (the kernel must call qc::chain_sync first).
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = g_hints.pdl != 0 ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// What the calling thread records between qgraph_record_begin and qgraph_record_end (NULL: nothing).
thread_local std::unique_ptr<qc::GraphInputRecord> g_graph_inputs;

// launch_chained for the kernels that read the network's float input (their first argument): under capture the
// node is noted, so that a replay can be pointed at another input.
template <typename... KArgs, typename... Args>
cudaError_t launch_input(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t st, Args... args) {
  const cudaError_t e = launch_chained(kernel, grid, block, 0, st, args...);
  if (e == cudaSuccess && g_graph_inputs)
    qc::note_graph_input(g_graph_inputs.get(), st, kernel, grid, block, size_t{0}, static_cast<KArgs>(args)...);
  return e;
}

int grid_for(size_t work_items, int threads, int max_blocks) {
  size_t b = (work_items + threads - 1) / threads;
  return static_cast<int>(std::max<size_t>(1, std::min<size_t>(b, max_blocks)));
}

}  // namespace

namespace {
int create_layer(qconv_handle** out, const qconv_desc* desc, const int8_t* w_host, const int32_t* bias_host,
                 const int32_t* shift_host, const int32_t* res_lshift_host, const int32_t* acc_exp_host,
                 const qconv_handle* weights_of, const NpSpec* np);
}

extern "C" {

const char* qconv_last_error_string(void) { return g_err; }

int qconv_checked_faults(int* first_line_out) {
  int v[2] = {0, 0};
#ifdef QCONV_CHECKED
  if (cudaDeviceSynchronize() != cudaSuccess ||
      cudaMemcpyFromSymbol(v, qc::g_checked_fault, sizeof(v)) != cudaSuccess)
    return fail(QCONV_ERR_CUDA, "qconv_checked_faults: cannot read the fault word");
  const int zero[2] = {0, 0};
  cudaMemcpyToSymbol(qc::g_checked_fault, zero, sizeof(zero));
#else
  v[0] = -1;                                               // not a checked build
#endif
  if (first_line_out) *first_line_out = v[1];
  return v[0];
}

int qconv_set_plan_hints(const qconv_plan_hints* hints) {
  g_hints = hints ? *hints : kNoHints;
  return QCONV_OK;
}

int qconv_create(qconv_handle** out, const qconv_desc* desc, const int8_t* w_host,
                 const int32_t* bias_host, const int32_t* shift_host,
                 const int32_t* res_lshift_host, const int32_t* acc_exp_host) {
  return qconv_create_sharing(out, desc, w_host, bias_host, shift_host, res_lshift_host, acc_exp_host, nullptr);
}

int qconv_create_sharing(qconv_handle** out, const qconv_desc* desc, const int8_t* w_host, const int32_t* bias_host,
                         const int32_t* shift_host, const int32_t* res_lshift_host, const int32_t* acc_exp_host,
                         const qconv_handle* weights_of) {
  return create_layer(out, desc, w_host, bias_host, shift_host, res_lshift_host, acc_exp_host, weights_of, nullptr);
}

}  // extern "C"

namespace {
// np: the layer runs on the digit planes of floating-point operands (w_host is then only a placeholder for the checks).
int create_layer(qconv_handle** out, const qconv_desc* desc, const int8_t* w_host, const int32_t* bias_host,
                 const int32_t* shift_host, const int32_t* res_lshift_host, const int32_t* acc_exp_host,
                 const qconv_handle* weights_of, const NpSpec* np) {
  if (!out) return fail(QCONV_ERR_BAD_ARG, "out is NULL");
  *out = nullptr;
  if (!desc || !w_host) return fail(QCONV_ERR_BAD_ARG, "desc or w_host is NULL");
  qconv_desc d = *desc;
  if (d.N <= 0 || d.H <= 0 || d.W <= 0 || d.C <= 0 || d.K <= 0 || d.R <= 0 || d.S <= 0 ||
      d.stride_h <= 0 || d.stride_w <= 0 || d.pad_h < 0 || d.pad_w < 0 || d.groups <= 0)
    return fail(QCONV_ERR_BAD_ARG, "non-positive dimension in descriptor");
  if (d.n_in < 2 || d.n_in > 8 || d.n_w < 2 || d.n_w > 8 || d.n_out < 2 || d.n_out > 8)
    return fail(QCONV_ERR_BAD_ARG, "bit widths must be in [2, 8]");
  if (d.rounding < 0 || d.rounding > 3 || d.out_mode < 0 || d.out_mode > 2 || d.weight_layout < 0 ||
      d.weight_layout > 1 || d.algo < 0 || d.algo > 3)
    return fail(QCONV_ERR_BAD_ARG, "unknown enum value in descriptor");
  if (d.C % d.groups || d.K % d.groups)
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "groups must divide C and K");
  const int P = (d.H + 2 * d.pad_h - d.R) / d.stride_h + 1;
  const int Q = (d.W + 2 * d.pad_w - d.S) / d.stride_w + 1;
  if (d.H + 2 * d.pad_h < d.R || d.W + 2 * d.pad_w < d.S || P <= 0 || Q <= 0)
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "filter larger than padded input");
  if (d.out_c_pitch == 0) d.out_c_pitch = d.K;
  if (d.out_c_offset < 0 || d.out_c_offset + d.K > d.out_c_pitch)
    return fail(QCONV_ERR_BAD_ARG, "output channel window [%d, %d) exceeds pitch %d", d.out_c_offset,
                d.out_c_offset + d.K, d.out_c_pitch);
  if (static_cast<size_t>(d.N) * P * Q * d.out_c_pitch >= (1ull << 40) ||
      static_cast<size_t>(d.N) * d.H * d.W * d.C >= (1ull << 40))
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "tensor too large");
  if (d.has_residual && !res_lshift_host)
    return fail(QCONV_ERR_BAD_ARG, "has_residual needs res_lshift_host");
  if (d.pool != 0 && d.pool != 2) return fail(QCONV_ERR_BAD_ARG, "pool must be 0 or 2");
  if (d.pool && (d.has_residual || d.out_mode != QCONV_OUT_INT8 || (P & 1) || (Q & 1) || d.groups != 1))
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "pool: needs groups == 1, int8 output, no residual, even P and Q");
  const int Cg = d.C / d.groups;
  int max_t = 0;
  int64_t max_bias = 0;
  for (int k = 0; k < d.K; ++k) {
    if (shift_host && !np && (shift_host[k] < 0 || shift_host[k] > 31))
      return fail(QCONV_ERR_BAD_SHIFT, "shift[%d] = %d outside [0, 31]", k, shift_host[k]);
    if (d.has_residual) {
      if (res_lshift_host[k] < 0 || res_lshift_host[k] > 23)
        return fail(QCONV_ERR_RESIDUAL_SCALE, "res_lshift[%d] = %d outside [0, 23]", k, res_lshift_host[k]);
      max_t = std::max(max_t, res_lshift_host[k]);
    }
    if (bias_host) max_bias = std::max<int64_t>(max_bias, std::llabs(static_cast<int64_t>(bias_host[k])));
    if (acc_exp_host && (acc_exp_host[k] < -126 || acc_exp_host[k] > 96))
      return fail(QCONV_ERR_BAD_ARG, "acc_exp[%d] = %d outside [-126, 96]", k, acc_exp_host[k]);
  }
  // Eq. 9 / Eq. 13: the longest sum must fit a 32-bit two's-complement accumulator.
  const int64_t bound = static_cast<int64_t>(d.R) * d.S * Cg * (1ll << (d.n_in - 1)) * (1ll << (d.n_w - 1)) +
                        max_bias + (d.has_residual ? (128ll << max_t) : 0);
  if (bound > 2147483647ll + (np ? max_bias : 0))          // (with digit products the bias meets the 64-bit sum)
    return fail(QCONV_ERR_OVERFLOW_RISK, "worst-case |accumulator| %lld exceeds 2^31 - 1", (long long)bound);

  qconv_handle* h = new qconv_handle();
  h->hints = g_hints;
  h->d = d;
  h->P = P; h->Q = Q; h->Cg = Cg; h->Kg = d.K / d.groups;
  h->acc_bound = bound;
  h->uniform_shift = 1;
  h->uni_s = shift_host ? shift_host[0] : 0;
  h->uni_t = d.has_residual ? res_lshift_host[0] : 0;
  for (int k = 0; k < d.K; ++k) {
    if ((shift_host ? shift_host[k] : 0) != h->uni_s) h->uniform_shift = 0;
    if (d.has_residual && res_lshift_host[k] != h->uni_t) h->uniform_shift = 0;
  }
  for (int k = 0; k < d.K && shift_host; ++k) h->max_shift = std::max(h->max_shift, shift_host[k]);
  h->hi = (1 << (d.n_out - 1)) - 1;
  h->lo = d.symmetric ? -h->hi : -(1 << (d.n_out - 1));
  cudaGetDevice(&h->device);
  cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);

  // weights to [K][R][S][Cg] on the host
  const size_t wcount = static_cast<size_t>(d.K) * d.R * d.S * Cg;
  std::vector<int8_t> w_turned;
  const int8_t* w_krsc = w_host;
  if (d.weight_layout != 0) {
    w_turned.resize(wcount);
    const size_t per_k = static_cast<size_t>(d.R) * d.S * Cg;
    for (int k = 0; k < d.K; ++k)
      for (size_t j = 0; j < per_k; ++j) w_turned[k * per_k + j] = w_host[j * d.K + k];
    w_krsc = w_turned.data();
  }

  // Weight-aware bound of the wide value: 2^(n_in-1) * sum|w[k,.]| + |bias[k]| + 128 * 2^t[k].  Below 2^22 the
  // tensor-core epilogue may round in fp32 (exactly).
  h->np = np;
  if (d.out_mode == QCONV_OUT_INT8 && (d.groups == 1 || (Cg == 1 && d.C == d.K)) && h->hints.float_rounding != 0 && !np) {
    // ... and below 2^15 after the shift, where the clamp works on 16-bit halves.
    long long worst = 0, worst_out = 0, worst_gen = 0, worst_gen_out = 0;
    bool unscaled = false;
    const size_t per_k = static_cast<size_t>(d.R) * d.S * Cg;
    for (int k = 0; k < d.K && worst < (1ll << 22) && worst_out < 32767; ++k) {
      const long long bnd = qc::host_abs_sum(w_krsc + k * per_k, per_k) * (1ll << (d.n_in - 1)) +
                            (bias_host ? std::llabs(static_cast<long long>(bias_host[k])) : 0) +
                            (d.has_residual ? (128ll << res_lshift_host[k]) : 0);
      worst = std::max(worst, bnd);
      const int sft = shift_host ? shift_host[k] : 0;
      const long long with_half = bnd + (sft > 0 && (d.rounding == QCONV_ROUND_HALF_AWAY || d.rounding == QCONV_ROUND_HALF_UP) ? 1ll << (sft - 1) : 0);
      worst_out = std::max(worst_out, (bnd >> sft) + 1);
      worst_gen = std::max(worst_gen, with_half);
      worst_gen_out = std::max(worst_gen_out, (with_half >> sft) + 1);
      unscaled |= sft == 0;
    }
    h->gen_flt = worst < (1ll << 22) && worst_out < 32767 && worst_gen < (1ll << 22) && worst_gen_out < 32767 && !(d.rounding == QCONV_ROUND_HALF_AWAY && !d.relu && unscaled);
    h->flt_epilogue = worst < (1ll << 22) && worst_out < 32767;
  }

  // choose the algorithm
  const bool dw_ok = d.groups == d.C && d.C == d.K && d.R == 3 && d.S == 3 && d.stride_h == d.stride_w &&
                     (d.stride_h == 1 || d.stride_h == 2) && d.C % 4 == 0 && d.out_c_pitch % 4 == 0 &&
                     d.out_c_offset % 4 == 0;
  const bool is_1x1 = d.R == 1 && d.S == 1 && d.pad_h == 0 && d.pad_w == 0;
  const bool s1 = d.stride_h == 1 && d.stride_w == 1;
  int mode = -1;
  if (d.groups == 1) {
    if (d.C % 16 == 0 && is_1x1 && s1) mode = MODE_FLAT;
    else if (d.C % 16 == 0 && is_1x1) mode = MODE_VIEW;
    else if (d.C % 16 == 0 && s1 && d.C <= 64 && d.S >= 4 && d.S * d.C <= 1024 &&
             static_cast<long long>(d.N) * d.H * d.W * d.C <= (64ll << 20) && h->hints.window_rows != 0 && d.pool == 0 && !np) mode = MODE_WROW;
    else if (d.C % 16 == 0 && d.stride_h <= 2 && d.stride_w <= 2) mode = MODE_BOX;   // (strides: see prepare_a_map)
    else if (d.C <= 4 && d.stride_h == 2 && d.stride_w == 2 && d.S + 1 <= 16 && d.R * d.S * d.C <= 1024 &&
             h->hints.space_to_depth != 0) mode = MODE_S2D;
    else if (d.C <= 4 && s1 && d.S >= 2 && d.S <= 16 && h->hints.window_rows != 0 &&
             static_cast<long long>(d.N) * d.H * (d.W + d.S + 16) < (1ll << 31)) mode = MODE_WROW;
    else if (d.C <= 4 && d.R * d.S * d.C <= 1024) mode = MODE_STEM;
  }
  if (d.pool && (mode != MODE_BOX || (d.algo != QCONV_ALGO_AUTO && d.algo != QCONV_ALGO_IGEMM))) {
    free_handle(h);
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "pool: only the tensor-core path with per-tap boxes takes the pool inside the layer");
  }
  int algo = d.algo;
  if (algo == QCONV_ALGO_AUTO) algo = mode >= 0 ? QCONV_ALGO_IGEMM : (dw_ok ? QCONV_ALGO_DEPTHWISE : QCONV_ALGO_DIRECT);
  if (algo == QCONV_ALGO_IGEMM && mode < 0) {
    free_handle(h);
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "implicit GEMM needs groups == 1 and C %% 16 == 0 with strides up to 2 "
                "(any stride for a 1x1 filter), or C <= 4");
  }
  if (algo == QCONV_ALGO_DEPTHWISE && !dw_ok) {
    free_handle(h);
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "depthwise kernel needs 3x3, groups == C == K, C %% 4 == 0");
  }
  h->algo = algo;
  h->mode = mode;

  DeviceParts parts;
  parts.add(&h->d_status, nullptr, 2 * sizeof(int));       // status word, maximum of qconv_run_maxabs
  int rc = QCONV_OK;
  if (algo == QCONV_ALGO_IGEMM) {
    rc = plan_igemm(h, parts, weights_of, w_krsc, bias_host, shift_host, res_lshift_host, acc_exp_host);
  } else {
    if (bias_host) parts.add(&h->d_bias, bias_host, sizeof(int32_t) * d.K);
    parts.add(&h->d_shift, shift_host, sizeof(int32_t) * d.K);
    if (d.has_residual) parts.add(&h->d_lshift, res_lshift_host, sizeof(int32_t) * d.K);
    parts.add(&h->d_accexp, acc_exp_host, sizeof(int32_t) * d.K);
    std::vector<int8_t> wp(wcount);
    const size_t per_k = static_cast<size_t>(d.R) * d.S * Cg;
    // [R][S][Cg][K]; for depthwise Cg == 1 this is [R*S][C]
    for (int k = 0; k < d.K; ++k)
      for (size_t j = 0; j < per_k; ++j) wp[j * d.K + k] = w_krsc[k * per_k + j];
    rc = place_weights(h, parts, wp.data(), wcount, false, nullptr);
    // Depthwise fast path (tap-packed dp4a with float-magic requantization, exact while
    // |bias| + 9 * 128 * 128 < 2^22): int8 output, nearest-even, 8-bit saturation, no residual.
    std::vector<uint32_t> t;
    if (algo == QCONV_ALGO_DEPTHWISE && d.out_mode == QCONV_OUT_INT8 && d.n_out == 8 &&
        d.rounding == QCONV_ROUND_NEAREST_EVEN && !d.has_residual && max_bias <= 4000000 &&
        h->hints.depthwise_form != 0) {
      t.resize(static_cast<size_t>(6) * d.C);
      for (int c = 0; c < d.C; ++c) {
        for (int r = 0; r < 3; ++r) {
          uint32_t word = 0;
          for (int sx = 0; sx < 3; ++sx)
            word |= static_cast<uint32_t>(static_cast<uint8_t>(wp[static_cast<size_t>(r * 3 + sx) * d.C + c])) << (8 * sx);
          t[static_cast<size_t>(r) * d.C + c] = word;
        }
        t[static_cast<size_t>(3) * d.C + c] = static_cast<uint32_t>((bias_host ? bias_host[c] : 0) + 0x4B400000);
        const int sh_c = shift_host ? shift_host[c] : 0;
        const float sc = sh_c <= 22 ? std::ldexp(1.0f, -sh_c) : 0.0f;
        const float off = static_cast<float>(12582912.0 * (1.0 - static_cast<double>(sc)));   // exact for s <= 22
        std::memcpy(&t[static_cast<size_t>(4) * d.C + c], &sc, 4);
        std::memcpy(&t[static_cast<size_t>(5) * d.C + c], &off, 4);
      }
      parts.add(&h->d_dw_tap, t.data(), t.size() * 4);
      h->dw_tap = 1;
      if (d.C % 32 == 0 && h->hints.depthwise_form != 1) plan_dw_tma(h);
      // On the tensor cores by warp-level instructions (kernel_dw_mma.cuh) where the channels fill its groups of 32, and for
      // small layers whatever they do; by tcgen05, in rows of 64 or 128 channels with an eighth of padding at most, where they do
      // not or where that is faster (dw_tcgen05_wins); else dp4a.  us per launch, warp level / tcgen05 / dp4a: 256 x 112 x 112 x 32
      // 67 / 91 / 73, 256 x 56 x 56 x 128 stride 2 27.4 / 27.8 / 30.2, 32 x 56 x 56 x 96 8.1 / 12.8 / 14.6, 64 x 56 x 56 x 144 26.3 / 34 / 25.4, 13 x 13 x
      // 13 x 1008 4.6 / 5.4 / 5.6; one image of those 2.8 to 3.2 / 3.3 to 4.0 / 3.9 to 4.2.  (With both planned, an output that is
      // 8-byte aligned only still takes the warp level.)
      const long long outputs = static_cast<long long>(d.N) * P * Q * d.C;
      const int form = h->hints.depthwise_form;
      const bool tensor_cores = h->flt_epilogue && h->hints.fast_epilogue != 0 && d.C % 16 == 0;
      if (tensor_cores && d.out_c_pitch % 8 == 0 && d.out_c_offset % 8 == 0 &&
          (form == 4 || (form < 0 && (d.C % 32 == 0 || outputs <= (4ll << 20)))))
        plan_dw_mma(h, form == 4 || outputs <= (4ll << 20) || align_up(d.C, 64) != static_cast<size_t>(d.C));
      h->dw_mma = tensor_cores && d.pad_h == 1 && d.pad_w == 1 && (form == 3 || align_up(d.C, 64) * 7 <= static_cast<size_t>(d.C) * 8) &&
                  d.out_c_pitch % 16 == 0 && d.out_c_offset % 16 == 0 && (form < 0 || form == 3) && (!h->dw_warp || dw_tcgen05_wins(h));
    }
    if (!rc && h->dw_warp) rc = allow_dw_mma_smem(h->device);
    if (!rc && h->dw_mma) {
      h->mode = MODE_BOX;
      rc = plan_igemm(h, parts, nullptr, w_krsc, bias_host, shift_host, nullptr, nullptr);
    } else if (!rc) {
      rc = parts.upload(&h->block);
    }
  }
  if (rc) {
    free_handle(h);
    return rc;
  }
  h->np = nullptr;
  *out = h;
  return QCONV_OK;
}

// Padded, widened copy of a stride-1 layer's input on at most 4 channels (from int8 or from float).
template <int C, int PB>
cudaError_t launch_row_pack_c(const qconv_handle* h, const void* src, bool f32, int e_x, int n_run, cudaStream_t st) {
  const qconv_desc& d = h->d;
  const unsigned int pixels = static_cast<unsigned int>(n_run) * d.H * d.W;
  const dim3 grid((pixels / 4 + 256) / 256);
  if (f32)
    return launch_input(qc::stem_row_pack_kernel<C, PB, true>, grid, dim3(256), st, src, h->d_pack, pixels, d.W, h->s2d_wp,
                          h->s2d_off_w, e_x, d.n_in);
  return launch_chained(qc::stem_row_pack_kernel<C, PB, false>, grid, dim3(256), 0, st, src, h->d_pack, pixels, d.W, h->s2d_wp,
                        h->s2d_off_w, 0, d.n_in);
}

cudaError_t launch_row_pack(const qconv_handle* h, const void* src, bool f32, int e_x, int n_run, cudaStream_t st) {
  const bool p8 = h->win_pb == 8;
  switch (h->d.C) {
    case 1: return p8 ? launch_row_pack_c<1, 8>(h, src, f32, e_x, n_run, st) : launch_row_pack_c<1, 16>(h, src, f32, e_x, n_run, st);
    case 2: return p8 ? launch_row_pack_c<2, 8>(h, src, f32, e_x, n_run, st) : launch_row_pack_c<2, 16>(h, src, f32, e_x, n_run, st);
    case 3: return p8 ? launch_row_pack_c<3, 8>(h, src, f32, e_x, n_run, st) : launch_row_pack_c<3, 16>(h, src, f32, e_x, n_run, st);
    default: return p8 ? launch_row_pack_c<4, 8>(h, src, f32, e_x, n_run, st) : launch_row_pack_c<4, 16>(h, src, f32, e_x, n_run, st);
  }
}

int run_dw_mma(qconv_handle* h, const int8_t* x, int8_t* y, int n_run, const qc::ConvGeom& g, const qc::DwTapParams& tp, cudaStream_t st) {
  qc::DwMmaParams& p = h->dw_mma_prm;
  int rc = prepare_dw_map(h, x, n_run, p.cb, p.pix, p.images, p.cb);
  if (rc) return rc;
  plan_dw_mma_strips(h, n_run);
  const dim3 grid(ceil_div(g.C, p.cb) * p.q_blocks, ceil_div(h->P, p.rows_per_cta), ceil_div(n_run, p.images));
  const size_t smem = dw_mma_smem(p);
  const bool uni = h->uniform_shift && h->hints.uniform_shift != 0;
  const DwMmaKernel kernel = kDwMmaKernels[g.stride_h - 1][uni][h->d.relu != 0];
  const int8_t* weights = h->d_w;
  CUDA_TRY(launch_chained(kernel, grid, dim3(p.warps * 32), smem, st, h->dw_map, weights, y, g, tp, p, h->d_status, h->wait_limit));
  return QCONV_OK;
}

// One layer launch.  input_is_packed: d_x is the handle's own space-to-depth scratch, already filled
// (qconv_run_f32 converts and packs in one kernel).  maxabs: d_y is the word of a running maximum (float bits of the
// largest |float output|) and nothing else is written.
int run_layer(qconv_handle* h, const int8_t* d_x, const int8_t* d_residual, void* d_y, int n_run,
              void* cuda_stream, bool input_is_packed, bool maxabs = false) {
  if (!h || !d_x || !d_y) return fail(QCONV_ERR_BAD_ARG, "NULL handle or tensor pointer");
  const qconv_desc& d = h->d;
  if (n_run <= 0 || n_run > d.N) return fail(QCONV_ERR_BAD_ARG, "n_run %d outside [1, %d]", n_run, d.N);
  if ((d.has_residual != 0) != (d_residual != nullptr))
    return fail(QCONV_ERR_BAD_ARG, "residual pointer does not match has_residual");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  h->last_stream = st;
  const float uni_c1 = h->uni_s <= 22 ? std::ldexp(1.0f, -h->uni_s) : 0.0f;
  qc::EpilogueParams ep{h->d_bias, h->d_shift, h->d_lshift, h->d_accexp, d.relu, d.rounding,
                        h->lo, h->hi, maxabs ? qc::kOutMaxAbs : d.out_mode, h->uni_s, h->uni_s > 0 ? (1 << (h->uni_s - 1)) - 1 : 0,
                        (h->uni_s > 0 ? 1 : 0) | ((1 << h->uni_t) << 1), uni_c1,
                        static_cast<float>(12582912.0 * (1.0 - static_cast<double>(uni_c1)))};
  qc::ConvGeom g{n_run, d.H, d.W, d.C, d.K, d.R, d.S, d.stride_h, d.stride_w, d.pad_h, d.pad_w,
                 d.groups, h->P, h->Q, d.out_c_offset, d.out_c_pitch};
  const size_t outs = static_cast<size_t>(n_run) * h->P * h->Q;
  if (h->algo == QCONV_ALGO_DIRECT) {
    qc::direct_conv_kernel<<<grid_for(outs * d.K, 256, h->num_sms * 64), 256, 0, st>>>(d_x, h->d_w, d_residual, d_y,
                                                                                g, ep);
  } else if (h->algo == QCONV_ALGO_DEPTHWISE &&
             !(h->dw_mma && ((reinterpret_cast<uintptr_t>(d_x) | reinterpret_cast<uintptr_t>(d_y)) & 15) == 0)) {
    if ((reinterpret_cast<uintptr_t>(d_x) | reinterpret_cast<uintptr_t>(d_y) |
         reinterpret_cast<uintptr_t>(d_residual)) & 3)
      return fail(QCONV_ERR_ALIGNMENT, "depthwise kernel needs 4-byte aligned tensors");
    constexpr int TW = 4;
    const bool mma_aligned = (reinterpret_cast<uintptr_t>(d_x) & 15) == 0 && (reinterpret_cast<uintptr_t>(d_y) & 7) == 0;
    if (h->dw_tap && n_run <= 65535) {
      const qc::DwTapParams tp{h->d_dw_tap, reinterpret_cast<const int32_t*>(h->d_dw_tap + static_cast<size_t>(3) * d.C),
                               reinterpret_cast<const float*>(h->d_dw_tap + static_cast<size_t>(4) * d.C),
                               reinterpret_cast<const float*>(h->d_dw_tap + static_cast<size_t>(5) * d.C),
                               12582912.0f + static_cast<float>(d.relu ? 0 : h->lo), 12582912.0f + static_cast<float>(h->hi)};
      if (h->dw_warp && mma_aligned) return run_dw_mma(h, d_x, static_cast<int8_t*>(d_y), n_run, g, tp, st);
      const int per_row = ceil_div(h->Q, TW) * (d.C / 4);
      // rows per thread: long strips amortise the per-thread tables, but the grid must still fill the GPU
      int rows = 16;
      while (rows > 4 && static_cast<long>(ceil_div(per_row, 256)) * ceil_div(h->P, rows) * n_run < 4L * h->num_sms) rows /= 2;
      rows = std::min(rows, h->P);
      dim3 grid(ceil_div(per_row, 256), ceil_div(h->P, rows), n_run);
      if (h->dw_tma && (reinterpret_cast<uintptr_t>(d_x) & 15) == 0) {
        int rc = prepare_dw_map(h, d_x, n_run, h->dw_prm.cwb_box * 4, h->dw_prm.pix, 1, 0);
        if (rc) return rc;
        qc::DwTmaParams prm = h->dw_prm;
        const int ctas_row = (d.C / 4 / prm.cwb) * prm.q_blocks;
        int rpc = 16;
        while (rpc > 4 && static_cast<long>(ctas_row) * ceil_div(h->P, rpc) * n_run < 4L * h->num_sms) rpc /= 2;
        prm.rows_per_cta = std::min(rpc, h->P);
        dim3 tgrid(ctas_row, ceil_div(h->P, prm.rows_per_cta), n_run);
        const size_t smem = static_cast<size_t>(qc::kDwStages) * prm.stage_bytes + sizeof(qc::DwTmaShared);
        if (d.stride_h == 1)
          qc::depthwise3x3_tma_kernel<1><<<tgrid, qc::kDwThreads, smem, st>>>(h->dw_map, static_cast<int8_t*>(d_y), g, tp, prm,
                                                                             h->d_status, h->wait_limit);
        else
          qc::depthwise3x3_tma_kernel<2><<<tgrid, qc::kDwThreads, smem, st>>>(h->dw_map, static_cast<int8_t*>(d_y), g, tp, prm,
                                                                             h->d_status, h->wait_limit);
      } else if (d.stride_h == 1) {
        qc::depthwise3x3_tap_kernel<1><<<grid, 256, 0, st>>>(d_x, static_cast<int8_t*>(d_y), g, tp, rows);
      } else {
        qc::depthwise3x3_tap_kernel<2><<<grid, 256, 0, st>>>(d_x, static_cast<int8_t*>(d_y), g, tp, rows);
      }
      cudaError_t e2 = cudaGetLastError();
      if (e2 != cudaSuccess) return fail(QCONV_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(e2));
      return QCONV_OK;
    }
    const size_t items = static_cast<size_t>(n_run) * h->P * ceil_div(h->Q, TW) * (d.C / 4);
    const int grid = grid_for(items, 256, h->num_sms * 64);
    if (d.stride_h == 1)
      qc::depthwise3x3_kernel<1, TW><<<grid, 256, 0, st>>>(d_x, h->d_w, d_residual, d_y, g, ep);
    else
      qc::depthwise3x3_kernel<2, TW><<<grid, 256, 0, st>>>(d_x, h->d_w, d_residual, d_y, g, ep);
  } else {
    if (reinterpret_cast<uintptr_t>(d_x) & 15)
      return fail(QCONV_ERR_ALIGNMENT, "d_x must be 16-byte aligned");
    if (h->prm.vec_store && !maxabs && !h->np_products && ((reinterpret_cast<uintptr_t>(d_y) | reinterpret_cast<uintptr_t>(d_residual)) & 15))
      return fail(QCONV_ERR_ALIGNMENT, "d_y and d_residual must be 16-byte aligned");
    const int8_t* a_ptr = d_x;
    if (h->mode == MODE_STEM) {
      if (h->stem_segp) {
        if (reinterpret_cast<uintptr_t>(d_x) & 3) return fail(QCONV_ERR_ALIGNMENT, "d_x must be 4-byte aligned");
        if (n_run > 65535 || static_cast<long long>(h->P) * h->Q * d.R >= (1ll << 31))
          return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "stem packing: image or batch too large");
        const long long x_bytes = static_cast<long long>(n_run) * d.H * d.W * d.C;
        const long long x_words = x_bytes / 4;             // whole words; the tail goes byte by byte
        const int x_tail = static_cast<int>(x_bytes % 4);
        const dim3 grid(ceil_div(h->Q, 64), ceil_div(h->P, 4), n_run);
        const int nw = (d.S * d.C + 3) / 4;                  // words holding segment bytes: 1..4 or 5..7
#define QC_PACK(SEGW, NW)                                                                                      \
  qc::stem_pack_rows_kernel<SEGW, NW><<<grid, 256, 0, st>>>(d_x, h->d_pack, n_run, d.H, d.W, d.C, d.R, d.S,    \
                                                            d.stride_h, d.stride_w, d.pad_h, d.pad_w, h->P,    \
                                                            h->Q, h->kg_pad, x_words, x_tail)
        if (h->stem_segp == 16) {
          switch (nw) {
            case 1: QC_PACK(4, 1); break;
            case 2: QC_PACK(4, 2); break;
            case 3: QC_PACK(4, 3); break;
            default: QC_PACK(4, 4); break;
          }
        } else {
          switch (nw) {
            case 5: QC_PACK(8, 5); break;
            case 6: QC_PACK(8, 6); break;
            default: QC_PACK(8, 7); break;
          }
        }
#undef QC_PACK
      } else {
        const size_t vecs = outs * (h->kg_pad / 16);
        qc::stem_pack_kernel<<<grid_for(vecs, 256, 148 * 32), 256, 0, st>>>(
            d_x, h->d_pack, n_run, d.H, d.W, d.C, d.R, d.S, d.stride_h, d.stride_w, d.pad_h, d.pad_w, h->P, h->Q,
            d.R * d.S * d.C, h->kg_pad);
      }
      a_ptr = h->d_pack;
    }
    if (h->mode == MODE_WROW && d.C < 16) {
      if (!input_is_packed) {
        cudaError_t pe = launch_row_pack(h, d_x, false, 0, n_run, st);
        if (pe != cudaSuccess) return fail(QCONV_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(pe));
      }
      a_ptr = h->d_pack;
    } else if (h->mode == MODE_WROW) {
      const size_t vecs = static_cast<size_t>(n_run) * d.H * d.W * (d.C / 16);
      if (vecs > 2147483647ull) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "row padding: image or batch too large");
      cudaError_t pe = launch_chained(qc::pad_rows_kernel, dim3(static_cast<unsigned int>((vecs + 255) / 256)), dim3(256), 0, st,
                                      reinterpret_cast<const uint4*>(d_x), reinterpret_cast<uint4*>(h->d_pack),
                                      static_cast<unsigned int>(vecs), n_run * d.H, d.W, d.C / 16, h->s2d_wp, h->s2d_off_w);
      if (pe != cudaSuccess) return fail(QCONV_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(pe));
      a_ptr = h->d_pack;
    }
    if (h->mode == MODE_S2D && input_is_packed) {
      a_ptr = h->d_pack;
    } else if (h->mode == MODE_S2D) {
      if (n_run > 65535 || h->s2d_h > 65535) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "stem packing: image or batch too large");
      const dim3 grid(ceil_div(h->s2d_w, 128), h->s2d_h, n_run);
      uint4* pk = reinterpret_cast<uint4*>(h->d_pack);
      cudaError_t pe;
      switch (d.C) {
        case 1: pe = launch_chained(qc::stem_s2d_pack_kernel<1>, grid, dim3(128), 0, st, d_x, pk, n_run, d.H, d.W, h->s2d_h, h->s2d_w, h->s2d_wp, h->s2d_off_w); break;
        case 2: pe = launch_chained(qc::stem_s2d_pack_kernel<2>, grid, dim3(128), 0, st, d_x, pk, n_run, d.H, d.W, h->s2d_h, h->s2d_w, h->s2d_wp, h->s2d_off_w); break;
        case 3: pe = launch_chained(qc::stem_s2d_pack_kernel<3>, grid, dim3(128), 0, st, d_x, pk, n_run, d.H, d.W, h->s2d_h, h->s2d_w, h->s2d_wp, h->s2d_off_w); break;
        default: pe = launch_chained(qc::stem_s2d_pack_kernel<4>, grid, dim3(128), 0, st, d_x, pk, n_run, d.H, d.W, h->s2d_h, h->s2d_w, h->s2d_wp, h->s2d_off_w); break;
      }
      if (pe != cudaSuccess) return fail(QCONV_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(pe));
      a_ptr = h->d_pack;
    }
    int rc = prepare_a_map(h, a_ptr, n_run);
    if (rc) return rc;
    if (!h->prm.fast_epilogue) {
      // bytes at which every row piece of the output and the residual is aligned
      auto widest = [](uintptr_t bits) { return bits & 7 ? 0 : bits & 8 ? 8 : 16; };
      const uintptr_t es = d.out_mode == QCONV_OUT_INT8 ? 1 : 4;
      h->prm.gen_vec_y = widest(reinterpret_cast<uintptr_t>(d_y) | es * d.out_c_pitch | es * d.out_c_offset | es * d.K);
      h->prm.gen_vec_res = widest(reinterpret_cast<uintptr_t>(d_residual) | static_cast<uintptr_t>(d.K));
    }
    const long tiles = static_cast<long>(h->prm.tiles_q) * h->prm.tiles_p * h->prm.tiles_n * h->prm.tiles_k;
    const int ksplit = maxabs || h->pair || tiles <= 0 ? 1 : choose_ksplit(h, tiles);
    h->split = ksplit;
    if (ksplit == 1) plan_staging(h, tiles);
    if (h->prm.out_stage_bytes && ksplit == 1) {
      rc = prepare_y_map(h, d_y, n_run);
      if (rc) return rc;
      if (d.has_residual && h->prm.out_stage_bufs == 3) {
        rc = prepare_r_map(h, d_residual, n_run);
        if (rc) return rc;
      }
    }
    const qc::IgemmParams& p = h->prm;
    if (h->pair) {
      qc::PairParams pp = {};
      pp.tq = p.tq; pp.tp = p.tp; pp.tn = p.tn;
      pp.tiles_q = p.tiles_q; pp.tiles_p = p.tiles_p; pp.tiles_n = p.tiles_n;
      const long boxes = static_cast<long>(p.tiles_q) * p.tiles_p * p.tiles_n;
      pp.pairs_m = static_cast<int>((boxes + 1) / 2);
      pp.tiles_k = p.tiles_k; pp.BN = p.BN; pp.BKC = p.BKC; pp.nchunks = p.nchunks; pp.R = p.R; pp.S = p.S;
      pp.pad_h = p.pad_h; pp.pad_w = p.pad_w; pp.stride_h = p.stride_h; pp.stride_w = p.stride_w;
      pp.stages = p.stages; pp.Q = p.Q; pp.P = p.P; pp.Nimg = p.Nimg; pp.K = p.K;
      pp.out_c_offset = p.out_c_offset; pp.out_c_pitch = p.out_c_pitch; pp.tmem_cols = p.tmem_cols;
      pp.a_stage_bytes = p.a_stage_bytes; pp.b_stage_bytes = p.b_stage_bytes;
      pp.tx_bytes = 2u * static_cast<uint32_t>(p.tq * p.tp * p.tn * p.BKC + (p.BN / 2) * p.BKC);
      const long pair_tiles = static_cast<long>(pp.pairs_m) * pp.tiles_k;
      if (pair_tiles <= 0 || pair_tiles > 1073741823l) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "tile count out of range");
      const long pairs = std::min<long>(pair_tiles, h->num_sms / 2);
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(static_cast<unsigned int>(2 * pairs));
      cfg.blockDim = dim3(qc::kIgemmThreads);
      cfg.dynamicSmemBytes = h->smem_bytes;
      cfg.stream = st;
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
      attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[1].val.programmaticStreamSerializationAllowed = h->use_pdl;
      cfg.attrs = attr;
      cfg.numAttrs = 2;
      const int4* chan_ptr = h->d_chan;
      cudaError_t le = cudaLaunchKernelEx(&cfg, pair_kernel_for(h), h->tmap_a, h->tmap_b, pp, p, ep, chan_ptr, d_y,
                                          h->d_status, h->wait_limit);
      if (le != cudaSuccess) return fail(QCONV_ERR_CUDA, "kernel launch (SM pairs): %s", cudaGetErrorString(le));
      return QCONV_OK;
    }
    if (tiles <= 0 || tiles > 2147483647l) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "tile count out of range");
    if (ksplit > 1) {
      qc::IgemmParams q = h->prm;
      const int num_kb = p.R * p.S * p.nchunks, own = p.BN / 16 / ksplit;
      q.ksplit = ksplit;
      q.out_stage_bytes = 0;
      q.gen_stage_bytes = static_cast<uint32_t>(own * (ksplit - 1) * 4 * 128 * 16);       // exchange area
      const size_t fixed = 1024 + q.gen_stage_bytes + sizeof(qc::IgemmShared), stage = p.a_stage_bytes + p.b_stage_bytes;
      q.stages = std::min<int>({ceil_div(num_kb, ksplit), qc::kMaxStages, static_cast<int>((226 * 1024 - fixed) / stage)});
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(static_cast<unsigned int>(tiles * ksplit));
      cfg.blockDim = dim3(qc::kIgemmThreads);
      cfg.dynamicSmemBytes = fixed + q.stages * stage;
      cfg.stream = st;
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = static_cast<unsigned int>(ksplit); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
      attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[1].val.programmaticStreamSerializationAllowed = h->use_pdl;
      cfg.attrs = attr;
      cfg.numAttrs = 2;
      const int4* chan_ptr = h->d_chan;
      cudaError_t le = cudaLaunchKernelEx(&cfg, split_kernel_for(h), h->tmap_a, h->tmap_b, h->tmap_a, h->tmap_a, q, ep, chan_ptr, d_residual,
                                          d_y, h->d_status, h->wait_limit);
      if (le != cudaSuccess) return fail(QCONV_ERR_CUDA, "kernel launch (split contraction): %s", cudaGetErrorString(le));
      return QCONV_OK;
    }
    long grid = std::min<long>(tiles, static_cast<long>(h->num_sms) * h->ctas_per_sm);
    // with resident weights a CTA must stay on one channel tile: the stride over tiles is a multiple of tiles_k
    if (p.b_resident && p.tiles_k > 1) grid = std::max<long>(p.tiles_k, grid / p.tiles_k * p.tiles_k);
    {
      // what depends on the grid size: its mixed-radix digits (the walk from one tile of a CTA to its next)
      qc::IgemmParams& pw = h->prm;
      if (h->walk_grid != grid) {
      long m = grid;
      pw.walk_dk = static_cast<int>(m % p.tiles_k); m /= p.tiles_k;
      pw.walk_dq = static_cast<int>(m % p.tiles_q); m /= p.tiles_q;
      pw.walk_dp = static_cast<int>(m % p.tiles_p); pw.walk_dn = static_cast<int>(m / p.tiles_p);
      pw.fd_grid = make_fastdiv(static_cast<int>(grid));
      h->walk_grid = grid;
      }
    }
    // Programmatic dependent launch: the kernel's set-up may overlap the tail of the previous
    // kernel in the stream; the kernel itself waits (griddepcontrol.wait) before touching tensors.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned int>(grid));
    cfg.blockDim = dim3(qc::kIgemmThreads);
    cfg.dynamicSmemBytes = h->smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = h->use_pdl;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int4* chan_ptr = h->d_chan;
    cudaError_t le = cudaLaunchKernelEx(&cfg, igemm_kernel_for(h, maxabs), h->tmap_a, h->tmap_b,
                                        p.out_stage_bytes ? h->tmap_y : h->tmap_a,
                                        (p.out_stage_bytes && p.out_stage_bufs == 3) ? h->tmap_r : h->tmap_a, p, ep, chan_ptr, d_residual,
                                        d_y, h->d_status, h->wait_limit);
    if (le != cudaSuccess) return fail(QCONV_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(le));
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(QCONV_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(e));
  return QCONV_OK;
}
}  // namespace

extern "C" {

int qconv_run(qconv_handle* h, const int8_t* d_x, const int8_t* d_residual, void* d_y, int n_run,
              void* cuda_stream) {
  return run_layer(h, d_x, d_residual, d_y, n_run, cuda_stream, false);
}

int qconv_run_maxabs(qconv_handle* h, const int8_t* d_x, const int8_t* d_residual, int n_run, float* maxabs_out,
                     void* cuda_stream) {
  if (!h || !maxabs_out) return fail(QCONV_ERR_BAD_ARG, "NULL handle or result pointer");
  if (h->d.out_mode != QCONV_OUT_FLOAT) return fail(QCONV_ERR_BAD_ARG, "qconv_run_maxabs serves layers with float output");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  int* word = h->d_status + 1;
  CUDA_TRY(cudaMemsetAsync(word, 0, sizeof(int), st));
  int rc = run_layer(h, d_x, d_residual, word, n_run, cuda_stream, false, true);
  if (rc) return rc;
  int host[2] = {0, 0};                                    // status and maximum in one read
  CUDA_TRY(cudaMemcpyAsync(host, h->d_status, sizeof(host), cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  if (host[0]) {
    CUDA_TRY(cudaMemset(h->d_status, 0, sizeof(int)));
    return fail(host[0], "a bounded device-side wait expired (status %d)", host[0]);
  }
  std::memcpy(maxabs_out, &host[1], sizeof(float));
  return QCONV_OK;
}

int qconv_run_f32(qconv_handle* h, const float* d_x_f32, int e_x, const int8_t* d_residual, void* d_y, int n_run,
                  void* cuda_stream) {
  if (!h || !d_x_f32 || !d_y) return fail(QCONV_ERR_BAD_ARG, "NULL handle or tensor pointer");
  const qconv_desc& d = h->d;
  const bool rows_form = h->algo == QCONV_ALGO_IGEMM && h->mode == MODE_WROW && d.C < 16;
  if (h->algo != QCONV_ALGO_IGEMM || (h->mode != MODE_S2D && !rows_form))
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "qconv_run_f32 serves layers that repack their input (at most 4 channels, "
                "stride 2 in space-to-depth form or stride 1 in padded rows); convert with qquantize_f32 and call "
                "qconv_run otherwise");
  if (n_run <= 0 || n_run > d.N) return fail(QCONV_ERR_BAD_ARG, "n_run %d outside [1, %d]", n_run, d.N);
  if (e_x < -126 || e_x > 126) return fail(QCONV_ERR_BAD_ARG, "e_x outside [-126, 126]");
  if (reinterpret_cast<uintptr_t>(d_x_f32) & 3) return fail(QCONV_ERR_ALIGNMENT, "d_x_f32 must be 4-byte aligned");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (rows_form) {
    cudaError_t re = launch_row_pack(h, d_x_f32, true, e_x, n_run, st);
    if (re != cudaSuccess) return fail(QCONV_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(re));
    return run_layer(h, h->d_pack, d_residual, d_y, n_run, cuda_stream, true);
  }
  if (n_run > 65535 || h->s2d_h > 65535) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "stem packing: image or batch too large");
  const dim3 grid(ceil_div(h->s2d_w, 128), h->s2d_h, n_run);
  uint4* pk = reinterpret_cast<uint4*>(h->d_pack);
  cudaError_t pe;
  switch (d.C) {
    case 1: pe = launch_input(qc::stem_s2d_pack_f32_kernel<1>, grid, dim3(128), st, d_x_f32, pk, n_run, d.H, d.W, h->s2d_h, h->s2d_w, h->s2d_wp, h->s2d_off_w, e_x, d.n_in); break;
    case 2: pe = launch_input(qc::stem_s2d_pack_f32_kernel<2>, grid, dim3(128), st, d_x_f32, pk, n_run, d.H, d.W, h->s2d_h, h->s2d_w, h->s2d_wp, h->s2d_off_w, e_x, d.n_in); break;
    case 3: pe = launch_input(qc::stem_s2d_pack_f32_kernel<3>, grid, dim3(128), st, d_x_f32, pk, n_run, d.H, d.W, h->s2d_h, h->s2d_w, h->s2d_wp, h->s2d_off_w, e_x, d.n_in); break;
    default: pe = launch_input(qc::stem_s2d_pack_f32_kernel<4>, grid, dim3(128), st, d_x_f32, pk, n_run, d.H, d.W, h->s2d_h, h->s2d_w, h->s2d_wp, h->s2d_off_w, e_x, d.n_in); break;
  }
  if (pe != cudaSuccess) return fail(QCONV_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(pe));
  return run_layer(h, h->d_pack, d_residual, d_y, n_run, cuda_stream, true);
}

// One native loop instead of one call from the host language per layer: a pass of 55 launches costs the host about
// 2.5 us each here against 13 us each through the binding.
int qnet_run(const qnet_step* steps, int count, const float* d_input, void* cuda_stream) {
  if (!steps || count < 0) return fail(QCONV_ERR_BAD_ARG, "NULL steps or negative count");
  for (int i = 0; i < count; ++i) {
    const qnet_step& s = steps[i];
    const float* in = reinterpret_cast<const float*>(reinterpret_cast<const char*>(d_input) + s.input_offset);
    int rc;
    switch (s.op) {
      case QNET_CONV: rc = qconv_run(s.handle, s.d_x, s.d_residual, s.d_y, s.n, cuda_stream); break;
      case QNET_CONV_F32:
        rc = d_input ? qconv_run_f32(s.handle, in, s.e_x, s.d_residual, s.d_y, s.n, cuda_stream)
                     : fail(QCONV_ERR_BAD_ARG, "step %d reads the float input, which is NULL", i);
        break;
      case QNET_QUANTIZE:
        rc = d_input ? qquantize_f32(in, s.count, s.e_x, s.n_bits, s.d_y, cuda_stream)
                     : fail(QCONV_ERR_BAD_ARG, "step %d reads the float input, which is NULL", i);
        break;
      case QNET_MAXPOOL:
        rc = qmaxpool_i8(s.d_x, s.n, s.H, s.W, s.C, s.R, s.R, s.stride, s.pad, s.d_y, cuda_stream);
        break;
      default: rc = fail(QCONV_ERR_BAD_ARG, "step %d: unknown operation %d", i, s.op);
    }
    if (rc) return rc;
  }
  return QCONV_OK;
}

int qgraph_record_begin(const float* d_input, size_t bytes) {
  if (!d_input || bytes == 0) return fail(QCONV_ERR_BAD_ARG, "NULL or empty input");
  g_graph_inputs = std::make_unique<qc::GraphInputRecord>();
  g_graph_inputs->base = reinterpret_cast<const char*>(d_input);
  g_graph_inputs->bytes = bytes;
  return QCONV_OK;
}

int qgraph_record_end(qgraph_inputs** out) {
  if (!out) return fail(QCONV_ERR_BAD_ARG, "out is NULL");
  *out = nullptr;
  std::unique_ptr<qc::GraphInputRecord> rec = std::move(g_graph_inputs);
  if (!rec) return fail(QCONV_ERR_BAD_ARG, "qgraph_record_begin has not been called on this thread");
  if (!rec->complete || rec->nodes.empty())
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "the captured graph's readers of the input could not be found");
  *out = new qgraph_inputs{std::move(*rec)};
  return QCONV_OK;
}

int qgraph_set_input(qgraph_inputs* g, void* graph_exec, const float* d_input) {
  if (!g || !graph_exec || !d_input) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  // (the kernels chose between vector and scalar loads from the recorded pointer's alignment)
  if ((reinterpret_cast<uintptr_t>(d_input) ^ reinterpret_cast<uintptr_t>(g->rec.base)) & 15)
    return fail(QCONV_ERR_ALIGNMENT, "d_input must be aligned as the recorded input");
  for (auto& node : g->rec.nodes) CUDA_TRY(node->set(static_cast<cudaGraphExec_t>(graph_exec), d_input));
  return QCONV_OK;
}

int qgraph_inputs_destroy(qgraph_inputs* g) {
  if (!g) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  delete g;
  return QCONV_OK;
}

int qconv_status(qconv_handle* h) {
  if (!h) return fail(QCONV_ERR_BAD_ARG, "NULL handle");
  CUDA_TRY(cudaStreamSynchronize(h->last_stream));
  int st = 0;
  CUDA_TRY(cudaMemcpy(&st, h->d_status, sizeof(int), cudaMemcpyDeviceToHost));
  if (st != 0) {
    CUDA_TRY(cudaMemset(h->d_status, 0, sizeof(int)));
    return fail(st, "a bounded device-side wait expired (status %d)", st);
  }
  return QCONV_OK;
}

int qconv_set_wait_limit(qconv_handle* h, unsigned int polls) {
  if (!h) return fail(QCONV_ERR_BAD_ARG, "NULL handle");
  h->wait_limit = polls;
  return QCONV_OK;
}

int qconv_describe(const qconv_handle* h, char* buf, size_t buf_len) {
  if (!h || !buf || buf_len == 0) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  if (h->algo == QCONV_ALGO_IGEMM || h->dw_mma) {
    static const char* names[] = {"flat", "view", "box", "stem", "s2d", "wrow"};
    const qc::IgemmParams& p = h->prm;
    snprintf(buf, buf_len, "%s/%s box=%dx%dx%d BN=%d tiles_k=%d BKC=%d chunks=%d taps=%dx%d stages=%d smem=%zu "
             "ctas/sm=%d fast=%d uni=%d flt=%d fold=%d tma_store=%d b_res=%d halo=%d grp=%d pair=%d pool=%d%s",
             h->dw_mma ? "depthwise3x3/mma" : "igemm", names[h->mode], p.tq, p.tp, p.tn, p.BN, p.tiles_k, p.BKC, p.nchunks, p.R, p.S, p.stages,
             h->smem_bytes, h->ctas_per_sm, p.fast_epilogue, h->uniform_shift, h->flt_epilogue && p.fast_epilogue, h->fold,
             p.out_stage_bytes ? p.out_stage_bufs : 0, p.b_resident, p.tap_boxes || h->patch ? 0 : p.halo_s, p.tap_boxes ? p.halo_s : 0, h->pair, h->d.pool, h->patch ? " patch=1" : "");
    const size_t used = std::strlen(buf);
    if (h->split > 1) snprintf(buf + used, buf_len - used, " split=%d", h->split);
    else if (h->np3) snprintf(buf + used, buf_len - used, " sums=32");
    else if (p.out_stage_bytes && !p.out_stage_bufs) snprintf(buf + used, buf_len - used, " ring=1");
  } else {
    snprintf(buf, buf_len, "%s", h->algo == QCONV_ALGO_DEPTHWISE ? (h->dw_warp ? "depthwise3x3/mma+tma" : h->dw_tma ? "depthwise3x3/tap-packed+tma" : h->dw_tap ? "depthwise3x3/tap-packed" : "depthwise3x3/dp4a")
                                                                  : "direct");
  }
  return QCONV_OK;
}

int qconv_destroy(qconv_handle* h) {
  if (!h) return fail(QCONV_ERR_BAD_ARG, "NULL handle");
  free_handle(h);
  return QCONV_OK;
}

// --------------------------------------------------------------------------- calibration
}  // extern "C"

// Scratch of qcalib_collect_static: lives in the library image, about 64 KB on every GPU that loads
// the library, until the process exits.  Its name below is only a host-side handle for the symbol;
// the device address comes from cudaGetSymbolAddress, once per device.
static __device__ __align__(256) unsigned char g_calib_static_scratch[sizeof(qc::CalibScratch)];

namespace {
// Device scratch of qcalib_collect and pinned memory its results land in, both made on first use per device and kept.
struct CalibDevice {
  // One collection at a time on each scratch, to its end: a collection relies on the accumulators that the one before left
  // at zero, so two that overlapped would spoil not only each other but every later one.
  std::mutex mu, built_in_mu;
  qc::CalibScratch* scratch = nullptr;
  qc::CalibScratch* built_in = nullptr;                    // device address of the array in the library image
  qc::CalibResult* landing = nullptr;
};
CalibDevice g_calib[64];

// The statistics passes shared by both entry points: maximum + sums, histogram, results.  `sc` is device scratch whose
// accumulators are zero (every collection leaves them so); `landing`: pinned host memory the second pass writes the
// results to, or NULL to copy them to pageable memory.
int calib_run(const float* d_x, size_t count, int nbins, float range_hi, qcalib_stats* host_out,
              cudaStream_t st, qc::CalibScratch* sc, qc::CalibResult* landing) {
  const int vec_ok = (reinterpret_cast<uintptr_t>(d_x) & 15) == 0;
  const size_t vecs = (count + 3) / 4;
  CUDA_TRY(launch_chained(qc::calib_pass1_kernel, dim3(grid_for(vecs, 256, 148 * qc::kCalibBlocksPerSm)), dim3(256), 0, st, d_x, count, sc,
                          nbins, vec_ok));
  cudaError_t e = launch_chained(qc::calib_hist_kernel, dim3(grid_for(vecs, qc::kCalibHistThreads, 148 * 2)), dim3(qc::kCalibHistThreads),
                                 nbins * sizeof(unsigned int), st, d_x, count, sc, nbins, range_hi, vec_ok, landing);
  qc::CalibResult pageable;
  if (e == cudaSuccess && !landing) {
    e = cudaMemcpyAsync(&pageable, &sc->res, offsetof(qc::CalibResult, hist) + sizeof(uint64_t) * nbins, cudaMemcpyDeviceToHost, st);
    landing = &pageable;
  }
  const cudaError_t done = cudaStreamSynchronize(st);      // (after a failure too: the scratch is the next call's from here on)
  CUDA_TRY(e);
  CUDA_TRY(done);
  const qc::CalibHead head = landing->head;
  std::memcpy(host_out->hist, landing->hist, sizeof(uint64_t) * nbins);
  std::memcpy(&host_out->maxabs, &head.maxabs_bits, sizeof(float));
  host_out->range_hi = range_hi > 0.0f ? range_hi : host_out->maxabs;
  host_out->count = head.finite;
  host_out->nonfinite = head.nonfinite;
  host_out->sum = head.sum;
  host_out->sumsq = head.sumsq;
  return QCONV_OK;
}
}  // namespace

extern "C" {

int qcalib_collect(const float* d_x, size_t count, int nbins, float range_hi, qcalib_stats* host_out,
                   void* cuda_stream) {
  if (!d_x || !host_out || !host_out->hist) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  if (count == 0 || nbins < 1 || nbins > qc::kCalibMaxBins)
    return fail(QCONV_ERR_BAD_ARG, "count must be > 0 and nbins in [1, %d]", qc::kCalibMaxBins);
  if (reinterpret_cast<uintptr_t>(d_x) & 3) return fail(QCONV_ERR_ALIGNMENT, "d_x must be 4-byte aligned");
  int dev = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(QCONV_ERR_CUDA, "device index %d out of range", dev);
  CalibDevice& d = g_calib[dev];
  std::lock_guard<std::mutex> lock(d.mu);
  if (!d.landing) CUDA_TRY(cudaHostAlloc(&d.landing, sizeof(qc::CalibResult), cudaHostAllocPortable));
  if (!d.scratch) {
    qc::CalibScratch* sc = nullptr;
    CUDA_TRY(DevicePool::pool().plain(&sc, sizeof(qc::CalibScratch)));
    const cudaError_t e = cudaMemset(sc, 0, sizeof(qc::CalibScratch));
    if (e != cudaSuccess) {
      cudaFree(sc);
      return fail(QCONV_ERR_CUDA, "calibration scratch: %s", cudaGetErrorString(e));
    }
    d.scratch = sc;
    CUDA_TRY(cudaDeviceSynchronize());                     // (the caller's stream may not wait for the legacy stream)
  }
  return calib_run(d_x, count, nbins, range_hi, host_out, static_cast<cudaStream_t>(cuda_stream), d.scratch, d.landing);
}

// ----------------------------------------------------------- calibration without allocation
int qcalib_collect_static(const float* d_x, size_t count, int nbins, float range_hi, qcalib_stats* host_out,
                          void* cuda_stream) {
  if (!d_x || !host_out || !host_out->hist) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  if (nbins < 1 || nbins > QCALIB_STATIC_MAX_BINS)
    return fail(QCONV_ERR_BAD_ARG, "qcalib_collect_static: nbins %d is outside [1, %d], the size of its built-in "
                "scratch", nbins, QCALIB_STATIC_MAX_BINS);
  if (count == 0 || count > QCALIB_STATIC_MAX_COUNT)
    return fail(QCONV_ERR_BAD_ARG, "qcalib_collect_static: count %zu is outside [1, 2^40], the most its built-in "
                "scratch is sized for", count);
  if (reinterpret_cast<uintptr_t>(d_x) & 3) return fail(QCONV_ERR_ALIGNMENT, "d_x must be 4-byte aligned");
  int dev = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(QCONV_ERR_CUDA, "device index %d out of range", dev);
  CalibDevice& d = g_calib[dev];
  std::lock_guard<std::mutex> lock(d.built_in_mu);
  if (!d.built_in) {
    // first call on this device: translate the symbol into this device's address (no allocation)
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_calib_static_scratch);
    if (e != cudaSuccess || !ptr)
      return fail(QCONV_ERR_CUDA, "cudaGetSymbolAddress(built-in calibration scratch): %s", cudaGetErrorString(e));
    d.built_in = static_cast<qc::CalibScratch*>(ptr);
  }
  // the array starts out zero with the library image, and every collection leaves its accumulators so
  return calib_run(d_x, count, nbins, range_hi, host_out, static_cast<cudaStream_t>(cuda_stream), d.built_in, nullptr);
}

int qquantize_f32(const float* d_x, size_t count, int e, int n, int8_t* d_y, void* cuda_stream) {
  if (!d_x || !d_y) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  if (n < 2 || n > 8 || e < -126 || e > 126) return fail(QCONV_ERR_BAD_ARG, "n in [2, 8], e in [-126, 126]");
  if (count == 0) return QCONV_OK;
  const int vec_ok = ((reinterpret_cast<uintptr_t>(d_x) | reinterpret_cast<uintptr_t>(d_y)) & 15) == 0;
  CUDA_TRY(launch_input(qc::quantize_f32_kernel, dim3(grid_for((count + 3) / 4, 256, 148 * 6)), dim3(256),
                        static_cast<cudaStream_t>(cuda_stream), d_x, d_y, count, e, n, vec_ok));
  CUDA_TRY(cudaGetLastError());
  return QCONV_OK;
}

int qmaxpool_i8(const int8_t* d_x, int N, int H, int W, int C, int R, int S, int stride, int pad,
                int8_t* d_y, void* cuda_stream) {
  if (!d_x || !d_y) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  if (N <= 0 || H <= 0 || W <= 0 || C <= 0 || R <= 0 || S <= 0 || stride <= 0 || pad < 0 || pad >= R || pad >= S)
    return fail(QCONV_ERR_BAD_ARG, "bad pooling geometry");
  const int P = (H + 2 * pad - R) / stride + 1, Q = (W + 2 * pad - S) / stride + 1;
  if (P <= 0 || Q <= 0) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "window larger than padded input");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const bool vec = C % 16 == 0 && ((reinterpret_cast<uintptr_t>(d_x) | reinterpret_cast<uintptr_t>(d_y)) & 15) == 0;
  const size_t pix = static_cast<size_t>(N) * P * Q;
  const bool strip_ok = vec && R == S && ((R == 3 && (stride == 1 || stride == 2)) || (R == 2 && stride == 2));
  if (strip_ok) {
    // strips as long as still leaves every SM several hundred threads
    // 3 x 3 at stride 1: two output columns a thread from about two warps' worth of such threads an SM on, one below, where the
    // longer chain of a thread counts (us, one / two: 2 x 2 x 39 x 336 1.63 / 1.83, 3 x 70 x 30 x 80 1.84 / 2.03, 16 x 7 x 7 x 832 2.34 / 2.14,
    // 16 x 28 x 28 x 192 3.8 / 2.3)
    const bool two = R == 3 && stride == 1 && Q > 1 && static_cast<size_t>(N) * ceil_div(P, 2) * ceil_div(Q, 2) * (C / 16) >= 148u * 72u;
    const int columns = ceil_div(Q, two ? 2 : 1);
    int rows = 16;
    while (rows > 2 && static_cast<size_t>(N) * ceil_div(P, rows) * columns * (C / 16) < 148u * 1024u) rows /= 2;
    const int strips = ceil_div(P, rows);
    const size_t threads = static_cast<size_t>(N) * strips * columns * (C / 16);
    if (threads > 2147483647ull) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "pooling: tensor too large");
    const dim3 grid(static_cast<unsigned int>((threads + 127) / 128));
    if (R == 3 && stride == 1 && !two)
      CUDA_TRY(launch_chained(qc::maxpool_i8_strip_kernel<3, 3, 1, 1>, grid, dim3(128), 0, st, d_x, d_y, N, H, W, C, pad, P, Q, rows, strips));
    else if (two)
      CUDA_TRY(launch_chained(qc::maxpool_i8_strip_kernel<3, 3, 1, 2>, grid, dim3(128), 0, st, d_x, d_y, N, H, W, C, pad, P, Q, rows, strips));
    else if (R == 3)
      CUDA_TRY(launch_chained(qc::maxpool_i8_strip_kernel<3, 3, 2, 1>, grid, dim3(128), 0, st, d_x, d_y, N, H, W, C, pad, P, Q, rows, strips));
    else
      CUDA_TRY(launch_chained(qc::maxpool_i8_strip_kernel<2, 2, 2, 1>, grid, dim3(128), 0, st, d_x, d_y, N, H, W, C, pad, P, Q, rows, strips));
  } else if (vec)
    CUDA_TRY(launch_chained(qc::maxpool_i8_vec_kernel, dim3(grid_for(pix * (C / 16), 256, 148 * 32)), dim3(256), 0, st,
                            d_x, d_y, N, H, W, C, R, S, stride, pad, P, Q));
  else
    qc::maxpool_i8_scalar_kernel<<<grid_for(pix * C, 256, 148 * 32), 256, 0, st>>>(d_x, d_y, N, H, W, C, R, S,
                                                                                   stride, pad, P, Q);
  CUDA_TRY(cudaGetLastError());
  return QCONV_OK;
}

int qeltwise_add_i8(const int8_t* const* d_inputs_host, int n_inputs, const int32_t* lshift_host, int rshift,
                    int relu, int rounding, int n_out, int symmetric, size_t count, int8_t* d_y, void* cuda_stream) {
  if (!d_inputs_host || !lshift_host || !d_y) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  if (n_inputs < 1 || n_inputs > 8 || n_out < 2 || n_out > 8 || rounding < 0 || rounding > 3)
    return fail(QCONV_ERR_BAD_ARG, "n_inputs in [1, 8], n_out in [2, 8], rounding in [0, 3]");
  if (rshift < 0 || rshift > 31) return fail(QCONV_ERR_BAD_SHIFT, "rshift %d outside [0, 31]", rshift);
  long long bound = 0;
  qc::EltwiseArgs a = {};
  int aligned = (reinterpret_cast<uintptr_t>(d_y) & 15) == 0;
  for (int i = 0; i < n_inputs; ++i) {
    if (!d_inputs_host[i]) return fail(QCONV_ERR_BAD_ARG, "input %d is NULL", i);
    if (lshift_host[i] < 0 || lshift_host[i] > 23)
      return fail(QCONV_ERR_RESIDUAL_SCALE, "lshift[%d] = %d outside [0, 23]", i, lshift_host[i]);
    bound += 128ll << lshift_host[i];
    a.in[i] = d_inputs_host[i];
    a.lshift[i] = lshift_host[i];
    aligned &= (reinterpret_cast<uintptr_t>(d_inputs_host[i]) & 15) == 0;
  }
  // Eq. 13: the widest sum must fit the 32-bit accumulator
  if (bound > 2147483647ll) return fail(QCONV_ERR_OVERFLOW_RISK, "worst-case |sum| %lld exceeds 2^31 - 1", bound);
  if (count == 0) return QCONV_OK;
  a.n_inputs = n_inputs; a.rshift = rshift; a.relu = relu; a.rounding = rounding;
  a.hi = (1 << (n_out - 1)) - 1;
  a.lo = symmetric ? -a.hi : -(1 << (n_out - 1));
  qc::eltwise_add_i8_kernel<<<grid_for((count + 15) / 16, 256, 148 * 16), 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
      a, d_y, count, aligned);
  CUDA_TRY(cudaGetLastError());
  return QCONV_OK;
}

// --------------------------------------------------------------------------- (n, p) codes
namespace {
int make_format(int n, int p, int e, qc::DynFloatFormat* f) {
  if (n < 2 || n > 8 || p < 0 || p > n - 1) return fail(QCONV_ERR_BAD_ARG, "need 2 <= n <= 8 and 0 <= p <= n-1");
  if (e < -126 || e > 126) return fail(QCONV_ERR_BAD_ARG, "scale exponent %d outside [-126, 126]", e);
  f->n = n; f->p = p;
  f->scale = std::ldexp(1.0f, -e);                         // normal for every e allowed here
  f->ke_min = static_cast<uint32_t>(127 + p) << 23;
  f->ke_up = static_cast<uint32_t>(23 - p) << 23;
  f->ke_off = f->ke_up + (static_cast<uint32_t>(127 + p) << p);
  // decoding reads the pattern as a binary32 number 2^(126 + p) too small; 2^(126 + p + e) may not be a binary32 number,
  // so the factor is split (the first product is exact, and what overflows on the way overflows in the end)
  f->up0 = std::ldexp(1.0f, 126);
  f->up1 = std::ldexp(1.0f, (p + e) / 2);
  f->up2 = std::ldexp(1.0f, p + e - (p + e) / 2);
  // Eq. 5 with equality: every pattern is a number
  f->beta_max = (p == n - 1) ? static_cast<float>((1 << (n - 1)) - 1)
                             : std::ldexp(static_cast<float>((2 << p) - 1), (1 << (n - p - 1)) - 2);
  return QCONV_OK;
}
}  // namespace

int qquantize_f32_np(const float* d_x, size_t count, int e, int n, int p, uint8_t* d_code, void* cuda_stream) {
  if (!d_x || !d_code) return fail(QCONV_ERR_BAD_ARG, "NULL tensor pointer");
  qc::DynFloatFormat f;
  int rc = make_format(n, p, e, &f);
  if (rc) return rc;
  if (count == 0) return QCONV_OK;
  const int vec_ok = ((reinterpret_cast<uintptr_t>(d_x) | reinterpret_cast<uintptr_t>(d_code)) & 15) == 0;
  const int grid = grid_for((count + 3) / 4, 256, 148 * 6);
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (p == 0) qc::dynfloat_encode_kernel<true><<<grid, 256, 0, st>>>(d_x, d_code, count, f, vec_ok);
  else qc::dynfloat_encode_kernel<false><<<grid, 256, 0, st>>>(d_x, d_code, count, f, vec_ok);
  CUDA_TRY(cudaGetLastError());
  return QCONV_OK;
}

int qdequantize_np(const uint8_t* d_code, size_t count, int e, int n, int p, float* d_y, void* cuda_stream) {
  if (!d_code || !d_y) return fail(QCONV_ERR_BAD_ARG, "NULL tensor pointer");
  qc::DynFloatFormat f;
  int rc = make_format(n, p, e, &f);
  if (rc) return rc;
  if (count == 0) return QCONV_OK;
  const int vec_ok = ((reinterpret_cast<uintptr_t>(d_y) | reinterpret_cast<uintptr_t>(d_code)) & 15) == 0;
  qc::dynfloat_decode_kernel<<<grid_for((count + 3) / 4, 256, 148 * 6), 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
      d_code, d_y, count, f, vec_ok);
  CUDA_TRY(cudaGetLastError());
  return QCONV_OK;
}

// --------------------------------------------------------------------------- convolution on (n, p) operands
}  // extern "C"

struct qconv_np_handle {
  qconv_np_desc d;
  qconv_handle* gemm = nullptr;      // tensor-core layer over the digit products, straight to the output patterns
  int digits_x = 1, digits_w = 1;
  qc::NpPlanes planes{};             // digit combinations of the input the products need
  int c_pad = 0;                     // channels of a plane (a whole number of ring-stage chunks)
  int P = 0, Q = 0;
  int8_t* d_planes = nullptr;        // [N][H][W][planes][c_pad]
};

namespace {
// beta_max of Eq. 5 (every pattern a number); -1 if it does not fit 62 bits.
long long np_beta_max(int n, int p) {
  if (p == n - 1) return (1ll << (n - 1)) - 1;
  const int e_max = (1 << (n - p - 1)) - 1;
  if (e_max - 1 + p + 1 > 61) return -1;
  return ((2ll << p) - 1) << (e_max - 1);
}
// 7-bit digit planes needed: the last digit may use the whole int8 range.
int np_planes(long long bmax) {
  if (bmax <= 127) return 1;
  if (bmax <= 127ll * 128 + 63) return 2;
  if (bmax <= (127ll * 128 + 63) * 128 + 63) return 3;
  return 0;
}
int np_host_decode(int code, int n, int p) {
  const int c = code & ((1 << (n - 1)) - 1);
  int v;
  if (p == n - 1) v = c;
  else {
    const int E = c >> p, m = c & ((1 << p) - 1);
    v = E == 0 ? m : ((1 << p) + m) << (E - 1);
  }
  return ((code >> (n - 1)) & 1) ? -v : v;
}
// Sum of those of beta's balanced digits that the mask names.
int np_digit_sum(int beta, int digits, int mask) {
  int sum = 0;
  for (int j = 0; j < digits; ++j) {
    const int dig = j + 1 < digits ? ((beta + 64) & 127) - 64 : beta;
    beta = (beta - dig) >> 7;
    if ((mask >> j) & 1) sum += dig;
  }
  return sum;
}
void free_np(qconv_np_handle* h) {
  if (!h) return;
  if (h->gemm) free_handle(h->gemm);
  cudaFree(h->d_planes);
  delete h;
}

// The digit products of x = sum x_i 128^i and w = sum w_j 128^j that give x w with the fewest multiplications
// (Karatsuba): with P_S = (sum of x_i, i in S) (sum of w_i, i in S) over single digits and pairs,
//   x_i w_j + x_j w_i = P_ij - P_ii - P_jj,
// three products for two digits and six for three, where the digit-by-digit schoolbook form takes four and nine.  The
// balanced digits (-64 ... 63; where there are several, the last one is at most 16) leave room for a sum of two in an int8.  Operands of different
// lengths are padded with zero digits, and products with a zero factor drop out.
struct NpProduct { int mask; long long coef; };
std::vector<NpProduct> np_products(int digits_x, int digits_w) {
  const int n = std::max(digits_x, digits_w);
  std::vector<NpProduct> all;
  for (int i = 0; i < n; ++i) {
    long long c = 1ll << (14 * i);
    for (int j = 0; j < n; ++j)
      if (j != i) c -= 1ll << (7 * (i + j));
    all.push_back({1 << i, c});
  }
  for (int i = 0; i < n; ++i)
    for (int j = i + 1; j < n; ++j) all.push_back({(1 << i) | (1 << j), 1ll << (7 * (i + j))});
  std::vector<NpProduct> kept;
  for (const NpProduct& p : all)
    if ((p.mask & ((1 << digits_x) - 1)) && (p.mask & ((1 << digits_w) - 1))) kept.push_back(p);
  return kept;
}
}  // namespace

extern "C" {

int qconv_np_create(qconv_np_handle** out, const qconv_np_desc* desc, const uint8_t* w_codes_host,
                    const int32_t* bias_host, const int32_t* shift_host) {
  if (!out) return fail(QCONV_ERR_BAD_ARG, "out is NULL");
  *out = nullptr;
  if (!desc || !w_codes_host) return fail(QCONV_ERR_BAD_ARG, "desc or w_codes_host is NULL");
  const qconv_np_desc d = *desc;
  if (d.N <= 0 || d.H <= 0 || d.W <= 0 || d.C <= 0 || d.K <= 0 || d.R <= 0 || d.S <= 0 || d.stride_h <= 0 ||
      d.stride_w <= 0 || d.pad_h < 0 || d.pad_w < 0)
    return fail(QCONV_ERR_BAD_ARG, "non-positive dimension in descriptor");
  const int fmts[3][2] = {{d.n_in, d.p_in}, {d.n_w, d.p_w}, {d.n_out, d.p_out}};
  long long bmax[3];
  for (int i = 0; i < 3; ++i) {
    if (fmts[i][0] < 2 || fmts[i][0] > 8 || fmts[i][1] < 0 || fmts[i][1] > fmts[i][0] - 1)
      return fail(QCONV_ERR_BAD_ARG, "need 2 <= n <= 8 and 0 <= p <= n-1 for every operand type");
    bmax[i] = np_beta_max(fmts[i][0], fmts[i][1]);
  }
  const int px = bmax[0] > 0 ? np_planes(bmax[0]) : 0, pw = bmax[1] > 0 ? np_planes(bmax[1]) : 0;
  if (px == 0 || pw == 0 || bmax[2] <= 0 || bmax[2] >= (1ll << 21))
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "an operand type's largest value (Eq. 5) exceeds three 7-bit digit planes (2^21)");
  if (d.C % 16) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "C must be a multiple of 16");
  const int P = (d.H + 2 * d.pad_h - d.R) / d.stride_h + 1, Q = (d.W + 2 * d.pad_w - d.S) / d.stride_w + 1;
  if (d.H + 2 * d.pad_h < d.R || d.W + 2 * d.pad_w < d.S || P <= 0 || Q <= 0)
    return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "filter larger than padded input");
  long long max_bias = 0;
  for (int k = 0; k < d.K; ++k) {
    if (shift_host && (shift_host[k] < 0 || shift_host[k] > 40))
      return fail(QCONV_ERR_BAD_SHIFT, "shift[%d] = %d outside [0, 40]", k, shift_host[k]);
    if (bias_host) max_bias = std::max<long long>(max_bias, std::llabs(static_cast<long long>(bias_host[k])));
  }
  // Eq. 9 with b = beta_max of the operand types and a 64-bit recombination (two bits of headroom)
  const long double worst = static_cast<long double>(d.R) * d.S * d.C * static_cast<long double>(bmax[0]) * bmax[1] + max_bias;
  if (worst >= 4.6e18L / 2)
    return fail(QCONV_ERR_OVERFLOW_RISK, "worst-case |sum| exceeds 2^62 (Eq. 9 with b = beta_max)");
  if (static_cast<long long>(d.R) * d.S * d.C * 128 * 128 > 2147483647ll)
    return fail(QCONV_ERR_OVERFLOW_RISK, "a digit product's sum of %lld terms does not fit a 32-bit accumulator", static_cast<long long>(d.R) * d.S * d.C);
  if (static_cast<size_t>(d.N) * P * Q * d.K >= (1ull << 38)) return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "tensor too large");

  qconv_np_handle* h = new qconv_np_handle();
  h->d = d; h->digits_x = px; h->digits_w = pw; h->P = P; h->Q = Q;
  const std::vector<NpProduct> products = np_products(px, pw);
  const size_t count = static_cast<size_t>(d.K) * d.R * d.S * d.C;
  std::vector<std::vector<int8_t>> w(products.size());
  NpSpec spec;
  spec.products = static_cast<int>(products.size());
  spec.n_out = d.n_out; spec.p_out = d.p_out; spec.top = static_cast<float>(bmax[2]);
  spec.largest_sum = static_cast<long long>(d.R) * d.S * d.C * bmax[0] * bmax[1] + max_bias;
  spec.largest_bias = max_bias;
  for (size_t m = 0; m < products.size(); ++m) {
    // the input's digit combination: one plane for each that differs
    const int x_mask = products[m].mask & ((1 << px) - 1), w_mask = products[m].mask & ((1 << pw) - 1);
    int plane = 0;
    while (plane < h->planes.count && h->planes.mask[plane] != x_mask) ++plane;
    if (plane == h->planes.count) h->planes.mask[h->planes.count++] = x_mask;
    spec.a_plane[m] = plane;
    spec.coef[m] = static_cast<int>(products[m].coef);
    w[m].resize(count);
    // one table of 256 patterns per product instead of decoding every weight
    int8_t table[256];
    for (int c = 0; c < 256; ++c) {
      const int sum = np_digit_sum(np_host_decode(c, d.n_w, d.p_w), pw, w_mask);
      const int sum_x = np_digit_sum(np_host_decode(c, d.n_in, d.p_in), px, x_mask);
      if (std::min(sum, sum_x) < -128 || std::max(sum, sum_x) > 127) {        // (no type that np_planes lets through)
        free_np(h);
        return fail(QCONV_ERR_UNSUPPORTED_SHAPE, "internal: a sum of digits does not fit an int8");
      }
      table[c] = static_cast<int8_t>(sum);
    }
    for (size_t i = 0; i < count; ++i) w[m][i] = table[w_codes_host[i]];
    spec.w[m] = w[m].data();
  }
  spec.planes = h->planes.count;
  qconv_desc g = {};
  g.N = d.N; g.H = d.H; g.W = d.W; g.C = d.C; g.K = d.K; g.R = d.R; g.S = d.S;
  g.stride_h = d.stride_h; g.stride_w = d.stride_w; g.pad_h = d.pad_h; g.pad_w = d.pad_w; g.groups = 1;
  g.n_in = 8; g.n_w = 8; g.n_out = 8; g.symmetric = 1; g.out_mode = QCONV_OUT_INT8; g.relu = d.relu; g.algo = QCONV_ALGO_IGEMM;
  int rc = create_layer(&h->gemm, &g, w[0].data(), bias_host, shift_host, nullptr, nullptr, nullptr, &spec);
  if (rc) { free_np(h); return rc; }
  h->c_pad = h->gemm->a_channels / spec.planes;
  const size_t bytes = static_cast<size_t>(d.N) * d.H * d.W * h->gemm->a_channels;
  cudaError_t e = DevicePool::pool().plain(&h->d_planes, bytes);
  if (e == cudaSuccess && h->c_pad != d.C) {
    // cleared once: the padding channels stay zero (waited for: the stream of the first run need not wait for this one)
    e = cudaMemsetAsync(h->d_planes, 0, bytes, nullptr);
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
  }
  if (e != cudaSuccess) {
    free_np(h);
    return fail(QCONV_ERR_CUDA, "qconv_np_create: %s", cudaGetErrorString(e));
  }
  *out = h;
  return QCONV_OK;
}

int qconv_np_run(qconv_np_handle* h, const uint8_t* d_x_codes, uint8_t* d_y_codes, int n_run, void* cuda_stream) {
  if (!h || !d_x_codes || !d_y_codes) return fail(QCONV_ERR_BAD_ARG, "NULL handle or tensor pointer");
  const qconv_np_desc& d = h->d;
  if (n_run <= 0 || n_run > d.N) return fail(QCONV_ERR_BAD_ARG, "n_run %d outside [1, %d]", n_run, d.N);
  if (reinterpret_cast<uintptr_t>(d_x_codes) & 15) return fail(QCONV_ERR_ALIGNMENT, "d_x_codes must be 16-byte aligned");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const size_t in_pix = static_cast<size_t>(n_run) * d.H * d.W;
  CUDA_TRY(launch_chained(qc::np_split_kernel, dim3(grid_for(in_pix * (d.C / 16), 256, 148 * 8)), dim3(256), 0, st,
                          d_x_codes, h->d_planes, in_pix, d.C, h->c_pad, d.n_in, d.p_in, h->digits_x, h->planes));
  return run_layer(h->gemm, h->d_planes, nullptr, d_y_codes, n_run, cuda_stream, false);
}

int qconv_np_status(qconv_np_handle* h) {
  if (!h) return fail(QCONV_ERR_BAD_ARG, "NULL handle");
  return qconv_status(h->gemm);
}

int qconv_np_describe(const qconv_np_handle* h, char* buf, size_t buf_len) {
  if (!h || !buf || buf_len == 0) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  char inner[400];
  qconv_describe(h->gemm, inner, sizeof(inner));
  snprintf(buf, buf_len, "np digits_x=%d digits_w=%d products=%d | %s", h->digits_x, h->digits_w, h->gemm->np_products, inner);
  return QCONV_OK;
}

int qconv_np_destroy(qconv_np_handle* h) {
  if (!h) return fail(QCONV_ERR_BAD_ARG, "NULL handle");
  free_np(h);
  return QCONV_OK;
}

// --------------------------------------------------------------------------- Algorithm 1
int qfpspace(int n, int p, double* out_host, int* count_out) {
  if (!out_host || !count_out) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  if (n < 2 || n > 8 || p < 0 || p > n - 1) return fail(QCONV_ERR_BAD_ARG, "need 2 <= n <= 8 and 0 <= p <= n-1");
  // Non-negative patterns 0 .. 2^(n-1)-1 decode (Eq. 2, exponent field per Eq. 4) to strictly
  // ascending values: subnormals are the significand itself, a normal number with exponent
  // field E is (2^p + significand) * 2^(E-1), and E = 1 continues where the subnormals end.
  const int levels = 1 << (n - 1);
  const int sig_mask = (1 << p) - 1;
  for (int b = 0; b < levels; ++b) {
    const int E = (p == n - 1) ? 0 : (b >> p);
    const int m = b & sig_mask;
    out_host[b] = E == 0 ? static_cast<double>(m) : std::ldexp(static_cast<double>((1 << p) + m), E - 1);
  }
  const double top = out_host[levels - 1];            // beta_max of Eq. 5
  for (int b = 0; b < levels; ++b) out_host[b] /= top;
  *count_out = levels;
  return QCONV_OK;
}

int qthreshold_search(const uint64_t* hist_host, int nbins, float range_hi, int n, int p, int measure,
                      double* gamma_out, double* delta_out, int* index_out, double* deltas_host, void* cuda_stream) {
  if (!hist_host || !gamma_out || !delta_out || !index_out) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  if (n < 2 || n > 8 || p < 0 || p > n - 1) return fail(QCONV_ERR_BAD_ARG, "need 2 <= n <= 8 and 0 <= p <= n-1");
  if (measure < 0 || measure > 3) return fail(QCONV_ERR_BAD_ARG, "measure in [0, 3]");
  const int first = (1 << (n - 1)) + 1;
  if (nbins < first || nbins > qc::kThrMaxBins)
    return fail(QCONV_ERR_BAD_ARG, "nbins %d outside [2^(n-1)+1 = %d, %d]", nbins, first, qc::kThrMaxBins);
  if (!(range_hi > 0.0f) || std::isinf(range_hi)) return fail(QCONV_ERR_BAD_ARG, "range_hi must be positive and finite");
  bool any = false;
  for (int j = 0; j < nbins && !any; ++j) any = hist_host[j] != 0;
  if (!any) return fail(QCONV_ERR_BAD_ARG, "empty histogram");
  double fp_host[qc::kThrMaxLevels];
  int levels = 0;
  int rc = qfpspace(n, p, fp_host, &levels);
  if (rc != QCONV_OK) return rc;

  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // device scratch sized for the largest histogram and pinned memory the operands leave from, made once per device and
  // kept; [counts | grid] go up in one copy
  struct Device {
    std::mutex mu;                                         // calls on one device share the scratch: serialised
    unsigned char* scratch = nullptr;
    unsigned char* pinned = nullptr;
    bool configured = false;                               // shared-memory limits of the kernels raised
  };
  static Device devices[64];
  int dev = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(QCONV_ERR_CUDA, "device index %d out of range", dev);
  Device& dv = devices[dev];
  const size_t off_fp = sizeof(uint64_t) * qc::kThrMaxBins;
  const size_t off_del = off_fp + sizeof(double) * qc::kThrMaxLevels;
  const size_t off_ticket = off_del + sizeof(double) * (qc::kThrMaxBins + 1);
  std::lock_guard<std::mutex> lock(dv.mu);
  if (!dv.pinned) CUDA_TRY(cudaHostAlloc(&dv.pinned, off_del + sizeof(qc::ThresholdBest), cudaHostAllocPortable));
  if (!dv.scratch) {
    unsigned char* sc = nullptr;
    CUDA_TRY(DevicePool::pool().plain(&sc, off_ticket + sizeof(unsigned int)));
    cudaError_t me = cudaMemset(sc, 0, off_ticket + sizeof(unsigned int));
    if (me == cudaSuccess) me = cudaDeviceSynchronize();
    if (me != cudaSuccess) {
      cudaFree(sc);
      return fail(QCONV_ERR_CUDA, "threshold scratch: %s", cudaGetErrorString(me));
    }
    dv.scratch = sc;
  }
  unsigned char* d = dv.scratch;
  // the levels follow the bins in memory, so that the copy is as short as the histogram
  const size_t at_fp = sizeof(uint64_t) * nbins;
  std::memcpy(dv.pinned, hist_host, at_fp);
  std::memcpy(dv.pinned + at_fp, fp_host, sizeof(double) * levels);
  auto* d_del = reinterpret_cast<double*>(d + off_del);
  // (pinned memory is mapped at the same address on the device; the kernel writes its answer there)
  qc::ThresholdBest* best_host = reinterpret_cast<qc::ThresholdBest*>(dv.pinned + off_del);
  const double top = p == n - 1 ? levels - 1.0 : std::ldexp(static_cast<double>((2 << p) - 1), (1 << (n - p - 1)) - 2);   // beta_max
  cudaError_t e = cudaMemcpyAsync(d, dv.pinned, at_fp + sizeof(double) * levels, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && deltas_host) e = cudaMemsetAsync(d_del, 0xFF, sizeof(double) * (nbins + 1), st);   // NaN outside the loop's range
  if (e == cudaSuccess) {
    using Kernel = decltype(&qc::threshold_search_kernel<0>);
    static const Kernel kernels[4] = {qc::threshold_search_kernel<qc::kMeasureL1>, qc::threshold_search_kernel<qc::kMeasureKS>,
                                      qc::threshold_search_kernel<qc::kMeasureCvM>, qc::threshold_search_kernel<qc::kMeasureKL>};
    if (!dv.configured) {
      for (Kernel k : kernels) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(qc::threshold_smem(qc::kThrMaxBins)));
        if (e != cudaSuccess) return fail(QCONV_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
      }
      dv.configured = true;
    }
    kernels[measure]<<<ceil_div(nbins - first + 1, qc::kThrCandidates), qc::kThrThreads, qc::threshold_smem(nbins), st>>>(
        reinterpret_cast<const unsigned long long*>(d), reinterpret_cast<const double*>(d + at_fp), nbins, levels, p,
        p == n - 1 ? 1 : 0, static_cast<float>(top), first, std::ldexp(1.0, -52), d_del,
        reinterpret_cast<unsigned int*>(d + off_ticket), best_host);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && deltas_host)
    e = cudaMemcpyAsync(deltas_host, d_del, sizeof(double) * (nbins + 1), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return fail(QCONV_ERR_CUDA, "qthreshold_search: %s", cudaGetErrorString(e));
  const qc::ThresholdBest best = *best_host;
  *index_out = best.index;
  *delta_out = best.delta;
  // bin_edges[i] of nbins equal bins on [0, range_hi]; the last edge is range_hi itself
  const double hi = static_cast<double>(range_hi);
  *gamma_out = best.index == nbins ? hi : static_cast<double>(best.index) * (hi / nbins);
  return QCONV_OK;
}

// --------------------------------------------------------------------------- machine measurement
int qbench_mma_i8(int bn, int mmas_per_cta, int row_bytes, int commit_every, float* ms_out, double* cycles_per_mma_out, int* ctas_out,
                  void* cuda_stream) {
  if (!ms_out || !cycles_per_mma_out || !ctas_out) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  if (bn < 16 || bn > 256 || bn % 16 || mmas_per_cta < 4 || mmas_per_cta > (1 << 20) || mmas_per_cta % 4)
    return fail(QCONV_ERR_BAD_ARG, "bn in [16, 256] multiple of 16; mmas_per_cta in [4, 2^20] multiple of 4");
  if (row_bytes != 128 && row_bytes != 64 && row_bytes != 32) return fail(QCONV_ERR_BAD_ARG, "row_bytes is 128, 64 or 32");
  if (commit_every < 0 || commit_every % 4) return fail(QCONV_ERR_BAD_ARG, "commit_every is 0 or a multiple of 4");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  int dev = 0, sms = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const size_t smem = 1024 + static_cast<size_t>(qc::kTileM + bn) * 128 + sizeof(qc::MmaPeakShared);
  CUDA_TRY(cudaFuncSetAttribute(qc::mma_peak_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  unsigned long long* d_cycles = nullptr;
  int* d_status = nullptr;
  CUDA_TRY(DevicePool::pool().plain(&d_cycles, sizeof(unsigned long long) * sms));
  cudaError_t e = DevicePool::pool().plain(&d_status, sizeof(int));
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (e == cudaSuccess) e = cudaMemsetAsync(d_status, 0, sizeof(int), st);
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  std::vector<unsigned long long> cyc(sms, 0);
  int status = 0;
  float ms = 0.0f;
  if (e == cudaSuccess) {
    // one CTA per SM (the shared-memory request above half an SM's keeps a second one out)
    const size_t smem_one = std::max<size_t>(smem, 120 * 1024);
    qc::mma_peak_kernel<<<sms, qc::kPeakThreads, smem_one, st>>>(bn, mmas_per_cta, row_bytes, commit_every, d_cycles, d_status, 1u << 26);   // warm-up
    cudaEventRecord(e0, st);
    qc::mma_peak_kernel<<<sms, qc::kPeakThreads, smem_one, st>>>(bn, mmas_per_cta, row_bytes, commit_every, d_cycles, d_status, 1u << 26);
    cudaEventRecord(e1, st);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaEventSynchronize(e1);
  if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
  if (e == cudaSuccess) e = cudaMemcpy(cyc.data(), d_cycles, sizeof(unsigned long long) * sms, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(&status, d_status, sizeof(int), cudaMemcpyDeviceToHost);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaFree(d_cycles);
  cudaFree(d_status);
  if (e != cudaSuccess) return fail(QCONV_ERR_CUDA, "qbench_mma_i8: %s", cudaGetErrorString(e));
  if (status != 0) return fail(QCONV_ERR_TIMEOUT, "qbench_mma_i8: the MMA train did not finish within the wait limit");
  double sum = 0.0;
  for (int i = 0; i < sms; ++i) sum += static_cast<double>(cyc[i]);
  *ms_out = ms;
  *cycles_per_mma_out = sum / sms / mmas_per_cta;
  *ctas_out = sms;
  return QCONV_OK;
}

// --------------------------------------------------------------------------- host helpers
int qscale_exponent(float gamma, int n, int* e_out) {
  if (!e_out || n < 2 || n > 8) return fail(QCONV_ERR_BAD_ARG, "e_out NULL or n outside [2, 8]");
  *e_out = 0;
  if (!(gamma > 0.0f) || std::isinf(gamma)) return QCONV_OK;
  // gamma = m * 2^ex with m in [0.5, 1).  beta_max * 2^e >= gamma  <=>  2^e >= gamma / beta_max.
  // Start one below the answer's lower bound and step up with exact comparisons.
  int ex;
  std::frexp(gamma, &ex);
  const double bmax = static_cast<double>((1 << (n - 1)) - 1);
  int e = ex - n;                       // beta_max * 2^(ex-n) < 2^(ex-1) <= gamma
  while (std::ldexp(bmax, e) < static_cast<double>(gamma)) ++e;
  *e_out = e;
  return QCONV_OK;
}

// Exponent bookkeeping of Section 3 (alpha = 2^e everywhere, so every factor is a shift).
int qacc_exponents(int e_x, const int32_t* e_w_host, int K, int32_t* acc_exp_host) {
  if (!e_w_host || !acc_exp_host || K <= 0) return fail(QCONV_ERR_BAD_ARG, "NULL argument or K <= 0");
  for (int k = 0; k < K; ++k) acc_exp_host[k] = e_x + e_w_host[k];
  return QCONV_OK;
}

int qrequant_shifts(int e_z, const int32_t* acc_exp_host, int K, int32_t* shift_host) {
  if (!acc_exp_host || !shift_host || K <= 0) return fail(QCONV_ERR_BAD_ARG, "NULL argument or K <= 0");
  for (int k = 0; k < K; ++k) {
    const long long sft = static_cast<long long>(e_z) - acc_exp_host[k];
    if (sft < 0 || sft > 31)
      return fail(QCONV_ERR_BAD_SHIFT, "shift[%d] = e_z - (e_x + e_w) = %lld outside [0, 31]", k, sft);
    shift_host[k] = static_cast<int32_t>(sft);
  }
  return QCONV_OK;
}

int qresidual_shifts(int e_res, const int32_t* acc_exp_host, int K, int32_t* lshift_host) {
  if (!acc_exp_host || !lshift_host || K <= 0) return fail(QCONV_ERR_BAD_ARG, "NULL argument or K <= 0");
  for (int k = 0; k < K; ++k) {
    const long long t = static_cast<long long>(e_res) - acc_exp_host[k];
    if (t < 0 || t > 23)
      return fail(QCONV_ERR_RESIDUAL_SCALE, "res_lshift[%d] = e_res - (e_x + e_w) = %lld outside [0, 23]", k, t);
    lshift_host[k] = static_cast<int32_t>(t);
  }
  return QCONV_OK;
}

int qjoin_exponent(const int32_t* e_own_host, const int32_t* const* acc_exp_hosts, const int32_t* K_host,
                   int n_branches, int* e_z_out) {
  if (!e_own_host || !acc_exp_hosts || !K_host || !e_z_out || n_branches <= 0)
    return fail(QCONV_ERR_BAD_ARG, "NULL argument or no branch");
  long long e_z = e_own_host[0];
  for (int b = 0; b < n_branches; ++b) {
    if (!acc_exp_hosts[b] || K_host[b] <= 0) return fail(QCONV_ERR_BAD_ARG, "branch %d: NULL exponents or K <= 0", b);
    e_z = std::max<long long>(e_z, e_own_host[b]);
    for (int k = 0; k < K_host[b]; ++k) e_z = std::max<long long>(e_z, acc_exp_hosts[b][k]);
  }
  *e_z_out = static_cast<int>(e_z);
  return QCONV_OK;
}

// Packed storage of n-bit betas: value i is the n-bit two's-complement field at bits [i n, (i + 1) n) of a
// little-endian bit stream.
int qpack_weights(const int8_t* wq_host, size_t count, int n, uint8_t* packed_host) {
  if (!wq_host || !packed_host || n < 2 || n > 8) return fail(QCONV_ERR_BAD_ARG, "NULL argument or n outside [2, 8]");
  const int lo = -(1 << (n - 1)), hi = (1 << (n - 1)) - 1;
  std::memset(packed_host, 0, (count * n + 7) / 8);
  for (size_t i = 0; i < count; ++i) {
    if (wq_host[i] < lo || wq_host[i] > hi) return fail(QCONV_ERR_BAD_ARG, "value %d at %zu does not fit %d bits", wq_host[i], i, n);
    const unsigned field = static_cast<unsigned>(wq_host[i]) & ((1u << n) - 1);
    const size_t bit = i * n;
    const unsigned sh = static_cast<unsigned>(bit & 7);
    packed_host[bit >> 3] |= static_cast<uint8_t>(field << sh);
    if (sh + n > 8) packed_host[(bit >> 3) + 1] |= static_cast<uint8_t>(field >> (8 - sh));
  }
  return QCONV_OK;
}

int qunpack_weights(const uint8_t* packed_host, size_t count, int n, int8_t* wq_host) {
  if (!wq_host || !packed_host || n < 2 || n > 8) return fail(QCONV_ERR_BAD_ARG, "NULL argument or n outside [2, 8]");
  const size_t nbytes = (count * n + 7) / 8;
  for (size_t i = 0; i < count; ++i) {
    const size_t bit = i * n;
    unsigned two = packed_host[bit >> 3];
    if ((bit >> 3) + 1 < nbytes) two |= static_cast<unsigned>(packed_host[(bit >> 3) + 1]) << 8;
    const unsigned field = (two >> (bit & 7)) & ((1u << n) - 1);
    wq_host[i] = static_cast<int8_t>((field >> (n - 1)) ? static_cast<int>(field) - (1 << n) : static_cast<int>(field));
  }
  return QCONV_OK;
}

int qconv_create_packed(qconv_handle** out, const qconv_desc* desc, const uint8_t* w_packed_host,
                        const int32_t* bias_host, const int32_t* shift_host, const int32_t* res_lshift_host,
                        const int32_t* acc_exp_host) {
  if (!out) return fail(QCONV_ERR_BAD_ARG, "out is NULL");
  *out = nullptr;
  if (!desc || !w_packed_host) return fail(QCONV_ERR_BAD_ARG, "desc or w_packed_host is NULL");
  if (desc->n_w < 2 || desc->n_w > 8 || desc->K <= 0 || desc->R <= 0 || desc->S <= 0 || desc->C <= 0 || desc->groups <= 0 ||
      desc->C % desc->groups)
    return fail(QCONV_ERR_BAD_ARG, "bad weight geometry or n_w outside [2, 8]");
  const size_t count = static_cast<size_t>(desc->K) * desc->R * desc->S * (desc->C / desc->groups);
  std::vector<int8_t> w(count);
  int rc = qunpack_weights(w_packed_host, count, desc->n_w, w.data());
  if (rc) return rc;
  return qconv_create(out, desc, w.data(), bias_host, shift_host, res_lshift_host, acc_exp_host);
}

int qquantize_weights(const float* w_host, int K, int R, int S, int Cg, int layout, int per_channel, int n,
                      int8_t* wq_host, int32_t* e_w_host) {
  if (!w_host || !wq_host || !e_w_host) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  if (K <= 0 || R <= 0 || S <= 0 || Cg <= 0 || n < 2 || n > 8 || layout < 0 || layout > 1)
    return fail(QCONV_ERR_BAD_ARG, "bad weight geometry");
  const size_t per_k = static_cast<size_t>(R) * S * Cg;
  if (layout == 0) {                                       // a channel's values are contiguous
    float gall = per_channel ? 0.0f : qc::host_max_abs(w_host, per_k * K);
    for (int k = 0; k < K; ++k) {
      const float* row = w_host + k * per_k;
      int e;
      qscale_exponent(per_channel ? qc::host_max_abs(row, per_k) : gall, n, &e);
      e_w_host[k] = e;
      if (per_channel) qc::host_quantize(row, per_k, e, n, wq_host + k * per_k);
    }
    if (!per_channel) qc::host_quantize(w_host, per_k * K, e_w_host[0], n, wq_host);
    return QCONV_OK;
  }
  auto at = [&](int k, size_t j) { return j * K + k; };
  auto largest = [&](int k) {
    float g = 0.0f;
    for (size_t j = 0; j < per_k; ++j) {
      const float a = std::fabs(w_host[at(k, j)]);
      if (std::isfinite(a)) g = std::max(g, a);
    }
    return g;
  };
  float gall = 0.0f;
  for (int k = 0; k < K && !per_channel; ++k) gall = std::max(gall, largest(k));
  for (int k = 0; k < K; ++k) {
    int e;
    qscale_exponent(per_channel ? largest(k) : gall, n, &e);
    e_w_host[k] = e;
    for (size_t j = 0; j < per_k; ++j) wq_host[at(k, j)] = qc::host_quantize_one(w_host[at(k, j)], e, n);
  }
  return QCONV_OK;
}

// Layers are independent: the largest first over up to eight threads.  (The conversion reads 5 bytes per value from
// memory twice; beyond eight threads the memory, not the arithmetic, sets the pace.)
int qquantize_weights_list(const qweights_job* jobs, int count) try {
  if (!jobs || count < 0) return fail(QCONV_ERR_BAD_ARG, "NULL jobs or negative count");
  std::vector<int> order(count), rc(count, QCONV_OK);
  for (int i = 0; i < count; ++i) order[i] = i;
  auto size = [&](int i) { return static_cast<long long>(jobs[i].K) * jobs[i].R * jobs[i].S * jobs[i].Cg; };
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return size(a) > size(b); });
  std::atomic<int> next{0};
  auto work = [&] {
    for (int i; (i = next.fetch_add(1)) < count;) {
      const qweights_job& j = jobs[order[i]];
      rc[order[i]] = qquantize_weights(j.w_host, j.K, j.R, j.S, j.Cg, j.layout, j.per_channel, j.n, j.wq_host, j.e_w_host);
    }
  };
  long long total = 0;
  for (int i = 0; i < count; ++i) total += size(i);
  // (a thread costs some 20 us to start: worth it from about 2^18 values each)
  const int want = static_cast<int>(std::min<long long>({8, count, total >> 18, std::max(1u, std::thread::hardware_concurrency())}));
  std::vector<std::thread> threads;
  threads.reserve(8);                                      // (nothing below may throw past a running thread)
  try {
    for (int t = 1; t < want; ++t) threads.emplace_back(work);
  } catch (const std::exception&) {                        // no more threads: the ones there are (this one at least) do it
  }
  work();
  for (std::thread& t : threads) t.join();
  for (int i = 0; i < count; ++i)
    if (rc[i]) return fail(rc[i], "weights %d: NULL argument or bad geometry", i);
  return QCONV_OK;
} catch (const std::exception& ex) {
  return fail(QCONV_ERR_BAD_ARG, "%d layers: %s", count, ex.what());
}

int qquantize_bias(const float* b_host, int K, int e_x, const int32_t* e_w_host, int32_t* bias_q_host) {
  if (!b_host || !e_w_host || !bias_q_host || K <= 0) return fail(QCONV_ERR_BAD_ARG, "NULL argument");
  int e = 0;
  double scale = 1.0;                                      // 2^-e: the product is ldexp(b, -e) wherever that is a normal number,
  for (int k = 0; k < K; ++k) {                            // and far below one half where it is not
    const int ek = e_x + e_w_host[k];
    if (ek != e) {
      e = ek;
      scale = std::ldexp(1.0, -e);
    }
    const bool plain = e >= -800 && e <= 800;
    double r = std::nearbyint(plain ? static_cast<double>(b_host[k]) * scale : std::ldexp(static_cast<double>(b_host[k]), -e));
    if (std::isnan(r)) r = 0.0;
    r = std::min(2147483647.0, std::max(-2147483648.0, r));
    bias_q_host[k] = static_cast<int32_t>(r);
  }
  return QCONV_OK;
}

}  // extern "C"
