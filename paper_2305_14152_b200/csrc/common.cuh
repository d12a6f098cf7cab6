// Shared host-side helpers of the PEQA sm_100a library: argument checks,
// CUDA error capture and the device status word.
#pragma once

#include <atomic>
#include <math.h>

#include <cuda_runtime.h>
#include <stdint.h>

#include "peqa.h"

namespace peqa {

extern thread_local int g_last_cuda_error;

inline int cuda_fail(cudaError_t e) {
  g_last_cuda_error = (int)e;
  return PEQA_ERR_CUDA;
}

#define PEQA_CUDA(expr)                                   \
  do {                                                    \
    cudaError_t _e = (expr);                              \
    if (_e != cudaSuccess) return ::peqa::cuda_fail(_e);  \
  } while (0)

#define PEQA_TRY(expr)              \
  do {                              \
    int _s = (expr);                \
    if (_s != PEQA_OK) return _s;   \
  } while (0)

// Allows `kern` its dynamic shared memory on the current device, once per device: the attribute
// stays with the function, and setting it again cost every launch 0.3 us on the host.  `done` is the kernel's
// own record (a bit per device); `bytes` is the most it is ever launched with.
template <typename Kern>
int allow_smem(Kern kern, int bytes, std::atomic<uint64_t>& done) {
  int dev = 0;
  PEQA_CUDA(cudaGetDevice(&dev));
  const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;
  if (done.load(std::memory_order_acquire) & bit) return PEQA_OK;
  PEQA_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  done.fetch_or(bit, std::memory_order_release);
  return PEQA_OK;
}

// Launches a kernel that begins with griddepcontrol.wait: its blocks stand ready when the kernel before it ends
// (a training step of one 256 x 256 layer, whose last launch adds up 256 sums: 1 us).
// Its pointer parameters are not __restrict__ (see ld_global in sm100_ptx.cuh).
template <typename... P, typename... A>
int launch_after(void (*kern)(P...), int blocks, int threads, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  PEQA_CUDA(cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...));
  return PEQA_OK;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Effective group size (per-channel when 0 or K) or 0 when invalid.
inline int effective_group(int K, int group_size) {
  if (group_size == 0 || group_size == K) return K;
  if (group_size < 0 || group_size % 32 != 0 || K % group_size != 0) return 0;
  return group_size;
}

inline int check_bits_shape(int N, int K, int bits, int group_size) {
  if (bits != 3 && bits != 4) return PEQA_ERR_BAD_BITS;
  if (N <= 0 || K <= 0 || K % 32 != 0) return PEQA_ERR_BAD_SHAPE;
  if (effective_group(K, group_size) == 0) return PEQA_ERR_BAD_SHAPE;
  return PEQA_OK;
}

// Validates a layer descriptor; fills g (effective group) and G.  With zeros_optional the
// integer zero-points may be absent (entry points that take real-valued ones).
int check_qweight(const peqa_qweight_t* w, int* g, int* G, bool zeros_optional = false);

// The current device must be compute capability 10.x (cached per device).
int check_arch();

// Device address of the status slot kernels launched on `st` report to, on the current
// device.  A slot is int[8]: [0] status code, [1..3] where, [4] bound of a single device-side
// wait in microseconds, [5] self-test knob (see peqa_selftest_configure), [6..7] unused.
// Streams get slots of their own (first come, first served; the last slot is shared by any
// further streams).  The first call on a device initialises the table with a blocking copy.
constexpr int kStatusSlots = 32;
constexpr int kStatusInts = 8;
int status_word(cudaStream_t st, int** dev_ptr);

// Multiprocessor count of the current device (cached per device); `fallback` when the query
// fails.
int sm_count_or(int fallback);

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

// One AdamW step on a scale (App. A; decoupled decay, bias-corrected moments).  The bias
// corrections 1 - b^t are formed on the host in double and passed as reciprocals, as are
// 1 - b1 and 1 - b2.  Every operation is a single rounded binary32 operation, so the
// stand-alone kernel and the kernels that apply the step where dS is produced agree bit
// for bit.
struct AdamWConsts {
  float lr, b1, b2, omb1, omb2, eps, decay, inv_c1, inv_c2;
};

inline AdamWConsts adamw_consts(float lr, float beta1, float beta2, float eps, float weight_decay,
                                long long step) {
  AdamWConsts c;
  const double c1 = pow((double)beta1, (double)step), c2 = pow((double)beta2, (double)step);
  c.lr = lr;
  c.b1 = beta1;
  c.b2 = beta2;
  c.omb1 = (float)(1.0 - (double)beta1);
  c.omb2 = (float)(1.0 - (double)beta2);
  c.eps = eps;
  c.decay = (float)(1.0 - (double)lr * (double)weight_decay);
  c.inv_c1 = (float)(1.0 / (1.0 - c1));
  c.inv_c2 = (float)(1.0 / (1.0 - c2));
  return c;
}

#ifdef __CUDACC__
__device__ __forceinline__ void adamw_update(float& s, float gr, float& m, float& v,
                                             const AdamWConsts& c) {
  const float mn = __fmaf_rn(c.b1, m, __fmul_rn(c.omb1, gr));
  const float vn = __fmaf_rn(c.b2, v, __fmul_rn(__fmul_rn(c.omb2, gr), gr));
  const float denom = __fadd_rn(sqrtf(__fmul_rn(vn, c.inv_c2)), c.eps);
  s = __fsub_rn(__fmul_rn(s, c.decay), __fdiv_rn(__fmul_rn(c.lr, __fmul_rn(mn, c.inv_c1)), denom));
  m = mn;
  v = vn;
}
#endif

// Work items of the CTA-pair kernels (forward, dX).  A tile is 512 tokens x 256 outputs held as
// two accumulators of 256 tokens.  Tiles are dealt round-robin to the pairs; when the last round
// would keep at most half of the pairs busy, its tiles are cut into two items of 256 tokens each.
// Rebuilding the weights costs the same for one block of tokens as for two, so that round takes 0.8
// to 0.9 as long (18944 x 8192, one round of 74 tiles: 256 tokens 92 us, 512 tokens 112).  Every tile must have
// two blocks to cut, the last row of tiles too (T % 512).  Items [0, full_items) are whole tiles, the rest are
// halves: item full_items + 2*i + h is half h of tile full_items + i.
struct PairItems {
  int o_tiles;       // 256-wide tiles along the output dimension
  int full_items;    // items that are whole tiles
  int total_items;
};
inline PairItems make_pair_items(int o_tiles, int t_tiles, int T, int pairs) {
  PairItems it;
  const int tiles = o_tiles * t_tiles;
  it.o_tiles = o_tiles;
  it.full_items = tiles;
  it.total_items = tiles;
  const int rem = pairs > 0 ? tiles % pairs : 0;
  if ((T % 512 == 0 || T % 512 > 256) && tiles > pairs && rem > 0 && 2 * rem <= pairs) {
    it.full_items = tiles - rem;
    it.total_items = tiles + rem;
  }
  return it;
}
#ifdef __CUDACC__
// Output tile, first token and token blocks (1 or 2) of an item.
__device__ __forceinline__ void pair_item(const PairItems& it, int item, int T, int& o_tile, int& tt0,
                                          int& blocks) {
  int tile = item, half = -1;
  if (item >= it.full_items) {
    const int h = item - it.full_items;
    tile = it.full_items + (h >> 1);
    half = h & 1;
  }
  const int t_tile = tile / it.o_tiles;
  o_tile = tile - t_tile * it.o_tiles;
  tt0 = t_tile * 512;
  if (half >= 0) {
    tt0 += half * 256;
    blocks = 1;
  } else {
    blocks = tt0 + 256 < T ? 2 : 1;
  }
}
#endif

// Contractions side by side: launched behind kernels of the same entry point whose results it does not read and whose operands it does
// not write (but AdamW, which waits for them), a contraction need not wait for them to end (kBeside) and fills the SMs they leave
// idle.  The first of them (kFollowed) lets it in only behind its own wait for what came before, so
// all of that is complete, and hands on that it is visible (let_next_in, begin_beside in sm100_ptx.cuh); and one that ran beside another does not
// end before it, so whoever waits for the last waits for all.  Training step, us, one after the other / side by side: 256 x 256
// at 64 tokens 15.2 / 10.5, 1024 x 1024 in groups of 64 at 200 24.3 / 20.2, 4096 x 4096 in groups of 128 at 2048 166 / 153; gradients
// with real zero-points 4096 x 11008 at 1001 164 / 135.
enum Side : int {
  kInOrder,     // waits for the kernel before, and whatever comes behind waits for this one
  kFollowed,    // waits; the next one is kBeside
  kBeside       // begins beside the one before, as the next one may beside this one
};

// Entry points implemented in the individual translation units.
// zeros_f != nullptr: real-valued zero-points [N, G] (App. K) replace w->zeros.  A call of T_call tokens may
// be launched in parts of T tokens from t0 on (X, Y: of the part; t0 a multiple of part_tokens(w, T_call)): every
// part takes the route of the whole call and sums in its order, so its results are the same bits.
int part_tokens(const peqa_qweight_t* w, int T_call);
int launch_fwd(const peqa_qweight_t* w, const float* zeros_f, int g, const void* X, int T, void* Y,
               cudaStream_t st, int T_call, int t0, Side side = kInOrder);
// Forward and, from its fp32 sums, the scale gradient of a layer with one scale per channel in two
// launches: the forward leaves partial sums per channel, launch_ds_channel adds them (and makes the
// AdamW step).  fwd_ds_slots: rows of N floats that takes, at most ds_workspace_bytes; 0 when the
// layer or T is not served this way.
int fwd_ds_slots(const peqa_qweight_t* w, int g, int T);
struct DsAdam;
int launch_fwd_ds(const peqa_qweight_t* w, const void* X, const void* dY, int T, void* Y, float* ds_part,
                  cudaStream_t st, Side side);
int launch_ds_channel(const peqa_qweight_t* w, const float* ds_part, int slots, float* dS, const DsAdam* adam,
                      cudaStream_t st);
bool fwd_pair_supported(const peqa_qweight_t* w);
// ds_part != nullptr (one scale per channel): sums of dY * u per channel, see fwd_pair_sm100.cu
int launch_fwd_pair(const peqa_qweight_t* w, const float* zeros_f, int g, const void* X, int T,
                    void* Y, const void* dY, float* ds_part, cudaStream_t st, Side side);
bool dx_pair_supported(const peqa_qweight_t* w);
int launch_dx_pair(const peqa_qweight_t* w, const float* zeros_f, int g, const void* dY, int T,
                   void* dX, Side side, cudaStream_t st);
int launch_dx(const peqa_qweight_t* w, const float* zeros_f, int g, const void* dY, int T, void* dX,
              cudaStream_t st, int T_call, int t0, Side side = kInOrder);
// forward (trans = false) or dX (true) for few tokens; same shapes as the pair kernels.
// channel_scales: a forward that multiplies by one scale per channel at the end
long long split_ns(const peqa_qweight_t* w, int T, bool trans);
bool split_is_faster(const peqa_qweight_t* w, int T, bool trans, bool channel_scales);
int split_ds_slots(const peqa_qweight_t* w, int T);
int split_part_tokens(const peqa_qweight_t* w, int T_call, bool trans);
int launch_split(const peqa_qweight_t* w, const float* zeros_f, int g, const void* act, int T, void* out,
                 bool trans, const void* dY, float* ds_part, cudaStream_t st, int T_call, int t0, Side side = kInOrder);
// adam != nullptr: the AdamW step on (w->scales, m, v) is applied where dS is produced
struct DsAdam {
  AdamWConsts c;
  float* scales;
  float* m;
  float* v;
};
// zeros_f != nullptr needs dZ: dS is then taken with the real-valued zero-point
int launch_ds(const peqa_qweight_t* w, const float* zeros_f, int g, const void* X, const void* dY,
              int T, float* dS, float* dZ, const DsAdam* adam, void* workspace,
              size_t workspace_bytes, cudaStream_t st, Side side = kInOrder);
size_t dsdz_workspace_bytes(const peqa_qweight_t* w, int g, int T);
size_t ds_workspace_bytes(const peqa_qweight_t* w, int g, int T);
size_t ds_from_y_workspace_bytes(const peqa_qweight_t* w, int T);
int launch_ds_from_y(const peqa_qweight_t* w, const void* dY, const void* Y, int T, float* dS,
                     void* workspace, cudaStream_t st);
// canonical weights through the kernel of the prepared decode (decode_prep.cu), up to eight tokens: one scale per
// channel, groups of 128 or 256 columns
bool decode_rows_are_faster(const peqa_qweight_t* w, int g, int M);
bool decode_rows_supported(const peqa_qweight_t* w, int g, int M);
int launch_decode_rows(const peqa_qweight_t* w, int g, const void* X, int M, void* Y, const float* scale_table,
                       int n_tasks, const int32_t* task_ids, cudaStream_t st);
bool decode_stream_supported(const peqa_qweight_t* w, int g, int M);
int launch_decode_stream(const peqa_qweight_t* w, int g, const void* X, int M, void* Y,
                         const float* scale_table, int n_tasks, const int32_t* task_ids,
                         cudaStream_t st);
int launch_decode(const peqa_qweight_t* w, int g, const void* X, int M, void* Y,
                  void* workspace, size_t workspace_bytes, cudaStream_t st);
size_t decode_workspace_bytes(const peqa_qweight_t* w, int g, int M);

}  // namespace peqa
