// Tensor-core kernels of the PEQA layer for sm_100a.
//
//   qgemm_kernel<TRANS=false>  Y[t,i]  = sum_j X[t,j]  * W_hat[i,j]     (forward, Eq. 2)
//   qgemm_kernel<TRANS=true>   dX[t,j] = sum_i dY[t,i] * W_hat[i,j]     (backward wrt input)
//   ds_kernel                  dS[i,g] = sum_{j in g} (Q-z)[i,j] * (dY^T X)[i,j]
//
// All three are persistent, warp-specialised kernels: one CTA per SM walks a
// static list of 128x256 output tiles.  Activations arrive by TMA into
// 128-byte-swizzled shared memory, tcgen05.mma accumulates fp32 in tensor
// memory (two 256-column accumulators, so the epilogue of one tile overlaps
// the main loop of the next), and every mbarrier wait is bounded.
//
// In qgemm the weight operand never exists in HBM as bf16: dedicated warps
// read the packed codes, rebuild (Q - z) [times bf16(s) when the scale varies
// along the contraction] in registers and write the bf16 tile straight into
// the swizzled layout the tensor core reads.  The weight tile is the MMA "A"
// operand (M = 128 weight rows/columns), the activation tile the "B" operand
// (N = 256 tokens), so each weight is dequantised once per 256 tokens.
//   forward : A is K-major   (row = out channel i, 64 contraction columns j)
//   dX      : A is MN-major  (row = contraction index i, 128 columns j) --
//             the same row-wise unpack, only the descriptor differs, so Q is
//             "read transposed" without any transposed copy.
//
// In ds_kernel both operands are activations (dY^T and X, MN-major straight
// from their row-major storage); the 128x256 dW tile stays in tensor memory,
// and the epilogue multiplies it by (Q - z) and sums over column pieces that
// lie inside one group.  dW never reaches HBM.
#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "dequant.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"

namespace peqa {

namespace {

using namespace ptx;

constexpr int BM = 128;      // weight rows per tile (MMA M, TMEM lanes)
constexpr int BN = 256;      // tokens (qgemm) / weight columns (ds) per tile (MMA N)
constexpr int BK = 64;       // contraction elements per pipeline stage
constexpr int UMMA_K = 16;   // contraction elements per tcgen05.mma
constexpr int STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;   // 16 KiB
constexpr int B_BYTES = BN * BK * 2;   // 32 KiB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int TMEM_COLS = 512;         // two fp32 accumulators of 256 columns
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align*/ + 512 /*barriers*/;

constexpr int kQgemmThreads = 512;     // warps: 0 TMA, 1 MMA, 2 TMEM alloc, 4-7 epilogue, 8-15 dequant
constexpr int kDequantThreads = 256;
constexpr int DQ_GROUPS = 4;           // dequant warp groups that take the stages round-robin
constexpr int kDsThreads = 384;        // warps: 0 TMA, 1 MMA, 2 TMEM alloc, 4-11 epilogue

struct Barriers {
  uint64_t full_a[STAGES];   // dequantised weight tile written (qgemm only)
  uint64_t full_b[STAGES];   // TMA bytes landed
  uint64_t empty[STAGES];    // MMAs that read the stage have completed
  uint64_t acc_full[2];      // accumulator ready for the epilogue
  uint64_t acc_empty[2];     // accumulator drained by the epilogue
  uint32_t tmem_base;
  int abort_flag;
  int wait_limit_us;    // must follow abort_flag (read by the bounded waits)
};

struct SmemView {
  uint8_t* a[STAGES];
  uint8_t* b[STAGES];
  Barriers* bars;
};

__device__ __forceinline__ SmemView carve_smem(uint8_t* raw) {
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  SmemView v;
#pragma unroll
  for (int s = 0; s < STAGES; ++s) {
    v.a[s] = base + s * STAGE_BYTES;
    v.b[s] = base + s * STAGE_BYTES + A_BYTES;
  }
  v.bars = reinterpret_cast<Barriers*>(base + STAGES * STAGE_BYTES);
  return v;
}

// After a bounded wait gave up: let copies and MMAs already in flight finish
// before shared and tensor memory are released.
__device__ __forceinline__ void drain_after_abort() {
  for (int i = 0; i < 64; ++i) __nanosleep(1000);
}

struct QGemmParams {
  const uint32_t* qw;
  const uint8_t* zeros;
  const float* zeros_f;   // real-valued zero-points (App. K) or nullptr; replaces `zeros`
  const float* scales;
  __nv_bfloat16* out;   // [T, R]
  int N, K, G, g, T;
  int g_shift;          // log2(g) when g is a power of two, else -1
  int wpr;              // packed words per weight row
  int R, C;             // output features, contraction length
  int r_tiles, t_tiles, k_blocks;
  int* status;
};

// Packed words, zero-point and scale of one 32-column unit of one weight row.
template <int BITS>
struct Unit {
  uint32_t w[BITS];
  uint32_t z;   // the bits of a real-valued zero-point (App. K)
  float s;
};

__device__ __forceinline__ int group_of(const QGemmParams& p, int col) {
  if (p.G == 1) return 0;
  return p.g_shift >= 0 ? (col >> p.g_shift) : (col / p.g);
}

// Weight row i, columns [col0, col0 + 32): packed words, zero-point and scale.
template <int BITS>
__device__ __forceinline__ Unit<BITS> load_unit(const QGemmParams& p, int i, int col0) {
  Unit<BITS> u;
#pragma unroll
  for (int q = 0; q < BITS; ++q) u.w[q] = 0u;
  if (i < p.N && col0 < p.K) {
    const uint32_t* src = p.qw + (size_t)i * p.wpr + (col0 >> 5) * BITS;
#pragma unroll
    for (int q = 0; q < BITS; ++q) u.w[q] = ld_global(src + q);
    const size_t gidx = (size_t)i * p.G + group_of(p, col0);
    u.s = ld_global(p.scales + gidx);
    u.z = p.zeros_f ? __float_as_uint(ld_global(p.zeros_f + gidx)) : ld_global(p.zeros + gidx);
  } else {
    // Outside the matrix: codes equal to the zero-point dequantise to exactly 0.
    u.z = 0u;
    u.s = 0.0f;
  }
  return u;
}

// (q - z) [* bf16(s)] of one unit; with a real-valued zero-point (zf, uniform over the
// launch, only with FOLD) the affine form (q - zi) * s + c.
template <int BITS, bool FOLD>
__device__ __forceinline__ void dequant_unit(const Unit<BITS>& u, bool zf, uint32_t (&o)[16]) {
  if (FOLD && zf) dq::unit32_affine<BITS>(u.w, u.z, u.s, o);
  else dq::unit32_natural<BITS, FOLD>(u.w, u.z, u.s, o);
}

// The fallback for packed rows whose pitch is not a multiple of 16 bytes (3-bit, K % 128 == 64): TMA
// cannot fetch their codes, so the dequant threads read them from global memory.
template <int BITS, bool TRANS, bool FOLD>
__global__ void __launch_bounds__(kQgemmThreads, 1)
qgemm_kernel(const __grid_constant__ CUtensorMap tmap_act, const QGemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  SmemView sm = carve_smem(smem_raw);
  Barriers* bars = sm.bars;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  volatile int* abort_flag = &bars->abort_flag;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&bars->full_a[s]), kDequantThreads / DQ_GROUPS);   // the threads of one dequant group
      mbar_init(smem_u32(&bars->full_b[s]), 1);
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bars->acc_full[b]), 1);
      mbar_init(smem_u32(&bars->acc_empty[b]), 128);
    }
    bars->abort_flag = 0;
    bars->wait_limit_us = p.status[4];
    fence_mbar_init();
    prefetch_tmap(&tmap_act);
  }
  if (warp == 2) {
    tmem_alloc(smem_u32(&bars->tmem_base), TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = bars->tmem_base;

  const int total_tiles = p.r_tiles * p.t_tiles;

  if (warp == 0) {
    // ------------------------------------------------ TMA producer (one lane)
    if (const uint32_t lane = elect_lane(); lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int tile = blockIdx.x; ok && tile < total_tiles; tile += gridDim.x) {
        const int t0 = (tile / p.r_tiles) * BN;
        for (int kb = 0; kb < p.k_blocks; ++kb, ++it) {
          const int s = it % STAGES;
          const uint32_t ph = (it / STAGES) & 1u;
          if (!mbar_wait(smem_u32(&bars->empty[s]), ph ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t bar = smem_u32(&bars->full_b[s]);
          mbar_arrive_expect_tx(bar, B_BYTES);
          tma_load_2d(smem_u32(sm.b[s]), &tmap_act, bar, kb * BK, t0);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------- MMA issuer (one lane)
    if (const uint32_t lane = elect_lane(); lane == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(BM, BN, TRANS ? 1 : 0, 0);
      uint32_t it = 0;
      int local = 0;
      bool ok = true;
      for (int tile = blockIdx.x; ok && tile < total_tiles; tile += gridDim.x, ++local) {
        const int buf = local & 1;
        const uint32_t acc_ph = (local >> 1) & 1u;
        if (!mbar_wait(smem_u32(&bars->acc_empty[buf]), acc_ph ^ 1u, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + buf * BN;
        for (int kb = 0; kb < p.k_blocks; ++kb, ++it) {
          const int s = it % STAGES;
          const uint32_t ph = (it / STAGES) & 1u;
          if (!mbar_wait(smem_u32(&bars->full_a[s]), ph, abort_flag) ||
              !mbar_wait(smem_u32(&bars->full_b[s]), ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t a_addr = smem_u32(sm.a[s]);
          const uint32_t b_addr = smem_u32(sm.b[s]);
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) {
            const uint64_t adesc = TRANS
                ? smem_desc_sw128(a_addr + k * (UMMA_K * 128), 64 * 128, 1024)
                : smem_desc_sw128(a_addr + k * (UMMA_K * 2), 16, 1024);
            const uint64_t bdesc = smem_desc_sw128(b_addr + k * (UMMA_K * 2), 16, 1024);
            mma_bf16_ss(d_tmem, adesc, bdesc, idesc, (kb | k) != 0 ? 1u : 0u);
          }
          mma_commit(smem_u32(&bars->empty[s]));
        }
        if (ok) mma_commit(smem_u32(&bars->acc_full[buf]));
      }
    }
  } else if (warp >= 4 && warp < 8) {
    // ------------------------------------------------------------- epilogue
    const int ew = warp - 4;  // == warp % 4: the TMEM lane quarter this warp may read
    int local = 0;
    bool ok = true;
    for (int tile = blockIdx.x; ok && tile < total_tiles; tile += gridDim.x, ++local) {
      const int r0 = (tile % p.r_tiles) * BM;
      const int t0 = (tile / p.r_tiles) * BN;
      const int buf = local & 1;
      const uint32_t acc_ph = (local >> 1) & 1u;
      if (!warp_wait(smem_u32(&bars->acc_full[buf]), acc_ph, abort_flag)) { ok = false; break; }
      tc_fence_after();
      const int r = r0 + ew * 32 + lane;
      float scale = 1.0f;
      if (!FOLD && r < p.R) scale = ld_global(p.scales + r);  // per-channel forward: s[i] applied here
#pragma unroll 1
      for (int cc = 0; cc < BN / 32; ++cc) {
        const int tc0 = t0 + cc * 32;
        if (tc0 >= p.T) break;
        uint32_t v[32];
        tmem_ld_32x32(tmem_base + ((uint32_t)(ew * 32) << 16) + buf * BN + cc * 32, v);
        tmem_ld_wait();
        if (r < p.R) {
          __nv_bfloat16* dst = p.out + (size_t)tc0 * p.R + r;
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            if (tc0 + j < p.T) dst[(size_t)j * p.R] = __float2bfloat16_rn(__uint_as_float(v[j]) * scale);
          }
        }
      }
      tc_fence_before();
      mbar_arrive(smem_u32(&bars->acc_empty[buf]));
    }
  } else if (warp >= 8) {
    // ------------------------------------------------------- weight dequant
    // DQ_GROUPS groups of warps take the stages round-robin, so that one group's
    // wait -> read -> convert -> store -> signal chain overlaps the other groups';
    // a thread converts UPT units (32 columns each) of its group's stage, all of
    // them into registers before it waits for the stage buffer to be released.
    constexpr int UPT = DQ_GROUPS;                      // 256 units per stage / threads per group
    constexpr int GW = (kDequantThreads / 32) / DQ_GROUPS;   // warps per group
    const int dw = warp - 8;
    const int grp = dw / GW;
    const int gw = dw % GW;
    const int my_tiles = (total_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    const uint32_t total_it = (uint32_t)my_tiles * (uint32_t)p.k_blocks;
    // forward: stage = 128 weight rows x 2 units; lanes = 32 consecutive rows; the
    //          thread's units are (row, 0), (row, 1), (row + 32*GW, 0), ...
    // dX:      stage = 64 weight rows x 4 units; lanes = 8 rows x 4 units; further
    //          units of the thread are the same columns 8*GW rows further down.
    const int u4 = lane >> 3;
    int rowl[UPT], col_off[UPT], chunk0[UPT], row_off[UPT];
#pragma unroll
    for (int k = 0; k < UPT; ++k) {
      if constexpr (!TRANS) {
        rowl[k] = gw * 32 + lane + (k >> 1) * (32 * GW);
        col_off[k] = 32 * (k & 1);
        chunk0[k] = 4 * (k & 1);
        row_off[k] = rowl[k] * 128;
      } else {
        rowl[k] = gw * 8 + (lane & 7) + k * (8 * GW);
        col_off[k] = 32 * u4;
        chunk0[k] = (u4 & 1) * 4;
        row_off[k] = (u4 >> 1) * (64 * 128) + rowl[k] * 128;
      }
    }
    const int swz = rowl[0] & 7;            // all rows of a thread agree modulo 8
    // cursor of the stage being prefetched (this group's next stage), no divisions
    int pf_tile = blockIdx.x, pf_kb = grp;
    while (pf_kb >= p.k_blocks) { pf_kb -= p.k_blocks; pf_tile += gridDim.x; }
    int pf_w0 = (pf_tile % p.r_tiles) * BM;
    auto load_next = [&](Unit<BITS> (&u)[UPT]) {
#pragma unroll
      for (int k = 0; k < UPT; ++k) {
        if constexpr (!TRANS) u[k] = load_unit<BITS>(p, pf_w0 + rowl[k], pf_kb * BK + col_off[k]);
        else u[k] = load_unit<BITS>(p, pf_kb * BK + rowl[k], pf_w0 + col_off[k]);
      }
      pf_kb += DQ_GROUPS;
      while (pf_kb >= p.k_blocks) {
        pf_kb -= p.k_blocks;
        pf_tile += gridDim.x;
        pf_w0 = (pf_tile % p.r_tiles) * BM;
      }
    };
    Unit<BITS> cur[UPT], nxt[UPT];
    if ((uint32_t)grp < total_it) load_next(cur);
    for (uint32_t it = grp; it < total_it; it += DQ_GROUPS) {
      if (it + DQ_GROUPS < total_it) load_next(nxt);
      const int s = it % STAGES;
      const uint32_t ph = (it / STAGES) & 1u;
      uint32_t o[UPT][16];
#pragma unroll
      for (int k = 0; k < UPT; ++k) dequant_unit<BITS, FOLD>(cur[k], p.zeros_f != nullptr, o[k]);
      if (!warp_wait(smem_u32(&bars->empty[s]), ph ^ 1u, abort_flag)) break;
#pragma unroll
      for (int k = 0; k < UPT; ++k) {
        uint8_t* row_ptr = sm.a[s] + row_off[k];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<uint4*>(row_ptr + (((chunk0[k] + q) ^ swz) << 4)) =
              make_uint4(o[k][4 * q], o[k][4 * q + 1], o[k][4 * q + 2], o[k][4 * q + 3]);
      }
      fence_proxy_async_smem();
      mbar_arrive(smem_u32(&bars->full_a[s]));
#pragma unroll
      for (int k = 0; k < UPT; ++k) cur[k] = nxt[k];
    }
  }

  // ---------------------------------------------------------------- teardown
  if (*abort_flag) drain_after_abort();
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
  if (threadIdx.x == 0 && bars->abort_flag) {
    atomicExch(p.status, (int)PEQA_ERR_DEVICE_TIMEOUT);
    p.status[1] = (int)blockIdx.x;
  }
}

// ------------------------------------------------------------------- dS ---
struct DsParams {
  const uint32_t* qw;
  const uint8_t* zeros;
  const float* zeros_f;   // real-valued zero-points (App. K) or nullptr; only with DZ
  float* out;        // [N, K / piece]: dS itself when piece == g, else partial sums
  float* out_z;      // same shape: dZ (or its partial sums of dW); only read by ds_kernel<.., true>
  const float* scales;
  // ds_kernel<.., ADAM = true> and the reduction kernel: AdamW applied where dS is final
  AdamWConsts adam;
  float* adam_s;
  float* adam_m;
  float* adam_v;
  int N, K, G, g, T;
  int wpr;
  int piece;         // columns per output piece: 32, 64 or 128; divides g
  int vec_ok;        // out, out_z, adam_s, adam_m, adam_v are 16-byte aligned
  int i_tiles, j_tiles, k_blocks;
  int band, band_rows;   // tile order: tiles per band and which dimension is banded (see ds_tile)
  Side side;           // see common.cuh
  int* status;
};

// Tile order of the dS kernel.  One of the two tile dimensions is taken in bands of `band`
// tiles (row tiles of dY^T when band_rows, else column tiles of X); within a band the other
// dimension moves slowest.  The pairs that run at the same time then share a band of operand
// rows (band x 2 MiB at T = 4096) that stays in L2 while the other operand is swept once per
// band; with the plain order (all row tiles for one column tile) dY was re-read from HBM for
// every few column tiles: 4x the algorithmic bytes on the 8192 x 8192 layer.
__device__ __forceinline__ void ds_tile(const DsParams& p, int tile, int& it, int& jt) {
  const int banded = p.band_rows ? p.i_tiles : p.j_tiles;   // tiles along the banded dimension
  const int other = p.band_rows ? p.j_tiles : p.i_tiles;
  const int per_band = p.band * other;
  const int b = tile / per_band;
  const int r = tile - b * per_band;
  const int width = min(p.band, banded - b * p.band);
  const int o = r / width;
  const int w = b * p.band + (r - o * width);
  it = p.band_rows ? w : o;
  jt = p.band_rows ? o : w;
}

// A CTA pair (cta_group::2) owns a 256 x 256 tile of dW: CTA `rank` holds rows
// [i0 + 128*rank, +128) of dY^T as its A operand and accumulator, and loads the
// 128 columns [j0 + 128*rank, +128) of X as its half of the shared B operand.
// The leader CTA (rank 0) issues every MMA; both CTAs' TMA loads credit the
// leader's "full" barrier and tcgen05.commit releases the stage in both CTAs.
constexpr int DS_STAGES = 6;
constexpr int DS_NEXT = 2;                                               // tiles asked for ahead (dynamic)
constexpr int DS_STAGE_BYTES = 2 * (BM * BK * 2);                      // A 16 KiB + B half 16 KiB
constexpr int DS_PK_BYTES = BM * 128;                                    // packed codes of a CTA's 128 x 256 half tile
constexpr int DS_SMEM_BYTES = DS_STAGES * DS_STAGE_BYTES + 2 * DS_PK_BYTES + 1024 + 512;

struct DsBarriers {
  uint64_t full[DS_STAGES];     // leader: bytes of both CTAs landed
  uint64_t empty[DS_STAGES];    // each CTA: MMAs that read the stage completed
  uint64_t acc_full[2];         // each CTA: accumulator ready
  uint64_t acc_empty[2];        // leader: both CTAs' epilogues drained the accumulator
  uint64_t pk_full[2];          // each CTA: packed codes of a tile landed
  uint64_t pk_empty[2];         // each CTA: its epilogue warps have read them
  uint4 response;               // leader: answer to a request for another tile (dynamic)
  uint64_t wanted;              // leader: one is wanted
  uint64_t answered;            // leader: the answer has arrived
  uint64_t next_full[DS_NEXT];  // each CTA: the number of a further tile stands in next_tile
  uint64_t next_empty[DS_NEXT]; // leader: every role of both CTAs has read it
  int next_tile[DS_NEXT];       // -1: no more
  uint32_t tmem_base;
  int abort_flag;
  int wait_limit_us;    // must follow abort_flag (read by the bounded waits)
};

// A thread's pieces of one row (n <= 4 adjacent floats): one vector access when they are whole and
// aligned.  The rows of a warp's lanes lie far apart, so every access touches 32 sectors and
// their number is what counts.
__device__ __forceinline__ void load_pieces(const float* src, int n, bool vec, float (&v)[4]) {
  if (n == 4 && vec) {
    const float4 t = *reinterpret_cast<const float4*>(src);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else if (n == 2 && vec) {
    const float2 t = *reinterpret_cast<const float2*>(src);
    v[0] = t.x; v[1] = t.y;
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < n) v[k] = src[k];
  }
}
__device__ __forceinline__ void store_pieces(float* dst, int n, bool vec, const float (&v)[4]) {
  if (n == 4 && vec) *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
  else if (n == 2 && vec) *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
  else {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < n) dst[k] = v[k];
  }
}

// PKTMA: the packed codes of a tile arrive by TMA (needs a 16-byte row pitch of the packed matrix);
// otherwise the epilogue threads read them from global memory.  With few tokens the epilogue sets
// the pace (a 256 x 256 tile has only T / 64 stages of MMAs), and what it cost was some thirty
// accesses of 32 sectors per warp and tile -- codes, optimizer state and results, read row by row
// after the accumulator was ready.  Codes by TMA a tile ahead, the rest as vectors requested before
// the wait (gradient and AdamW, before -> after): 22016 x 8192 in groups of 64 at 40 tokens
// 235 -> 122 us, 4096 x 4096 in groups of 32 at 77 tokens 42 -> 18 us, 4096 x 11008 per channel at
// 77 tokens 44 -> 31 us; 8192 x 8192 in groups of 64 at 4096 tokens 427 -> 406 us.
//
// DYNAMIC (beside another contraction, see common.cuh): the grid has a CTA pair per tile.  Pairs start on the SMs that the other kernel
// leaves idle, take over tiles that have not been started (cluster launch control), and those that start late find so
// many fewer left (us, dealt / taken over: dX, dS and dZ of 4096 x 11008 at 1001 tokens 158 / 135).
template <int BITS, bool DZ, bool ADAM, bool PKTMA, bool DYNAMIC>
__global__ void __launch_bounds__(kDsThreads, 1)
ds_kernel(const __grid_constant__ CUtensorMap tmap_dy, const __grid_constant__ CUtensorMap tmap_x,
          const __grid_constant__ CUtensorMap tmap_pk, const DsParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sm_pk = base + DS_STAGES * DS_STAGE_BYTES;
  DsBarriers* bars = reinterpret_cast<DsBarriers*>(sm_pk + 2 * DS_PK_BYTES);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  volatile int* abort_flag = &bars->abort_flag;
  const bool beside = p.side == kBeside;
  begin_beside(beside);

  if (threadIdx.x == 0) {
    for (int s = 0; s < DS_STAGES; ++s) {
      mbar_init(smem_u32(&bars->full[s]), 1);
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bars->acc_full[b]), 1);
      mbar_init(smem_u32(&bars->acc_empty[b]), 16);   // 8 epilogue warps in each of the 2 CTAs
      mbar_init(smem_u32(&bars->pk_full[b]), 1);
      mbar_init(smem_u32(&bars->pk_empty[b]), 8);
    }
    if (DYNAMIC) {
      for (int b = 0; b < DS_NEXT; ++b) {
        mbar_init(smem_u32(&bars->next_full[b]), 1);
        // two copying lanes and eight epilogue warps in each CTA, the leader's issuing lane
        mbar_init(smem_u32(&bars->next_empty[b]), 2 * 10 + 1);
      }
      mbar_init(smem_u32(&bars->wanted), 1);
      mbar_init(smem_u32(&bars->answered), 1);
    }
    bars->abort_flag = 0;
    bars->wait_limit_us = p.status[4];
    fence_mbar_init();
    prefetch_tmap(&tmap_dy);
    prefetch_tmap(&tmap_x);
    if (PKTMA) prefetch_tmap(&tmap_pk);
  }
  if (warp == 2) {
    tmem_alloc_pair(smem_u32(&bars->tmem_base), TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();          // barriers of both CTAs initialised before any remote arrive
  tc_fence_after();
  // Set-up is done.  Everything below touches memory that the preceding kernel may still be writing, unless this one was
  // launched beside it (common.cuh).
  if (!beside) asm volatile("griddepcontrol.wait;" ::: "memory");
  let_next_in(p.side == kFollowed);
  const uint32_t tmem_base = bars->tmem_base;
  const int total_tiles = p.i_tiles * p.j_tiles;   // pair tiles (256 x 256)
  const int pair = blockIdx.x >> 1;
  const int n_pairs = gridDim.x >> 1;
  // The tile behind `tile`, -1 if there is none: dealt round-robin, or (dynamic) the n-th that warp 2 got hold of.  A role
  // that reads it in one lane hands in that lane (0), a warp that goes on together reads it together.
  auto dealt = [&](int tile) { return tile + n_pairs < total_tiles ? tile + n_pairs : -1; };
  auto taken = [&](uint32_t n) { return *reinterpret_cast<volatile int*>(&bars->next_tile[n % DS_NEXT]); };
  auto release = [&](uint32_t n) { mbar_arrive_cluster_release(mapa_shared(smem_u32(&bars->next_empty[n % DS_NEXT]), 0)); };
  auto next_of_lane = [&](uint32_t lane, int tile, uint32_t n) {
    if (!DYNAMIC) return dealt(tile);
    if (lane == 0) {
      if (!mbar_wait_cluster(smem_u32(&bars->next_full[n % DS_NEXT]), (n / DS_NEXT) & 1u, abort_flag)) return -1;
    }
    const int next = taken(n);
    release(n);
    return next;
  };
  auto next_of_warp = [&](int tile, uint32_t n) {
    if (!DYNAMIC) return dealt(tile);
    if (!warp_wait_cluster(smem_u32(&bars->next_full[n % DS_NEXT]), (n / DS_NEXT) & 1u, abort_flag)) return -1;
    const int next = taken(n);
    __syncwarp();
    if (lane == 0) release(n);
    return next;
  };

  if (warp == 0) {
    if (const uint32_t lane = elect_lane(); lane == 0) {
      uint32_t it = 0, n = 0;
      bool ok = true;
      const int ask_at = DYNAMIC ? max(p.k_blocks - 6, 0) : -1;
      for (int tile = pair; ok && tile >= 0; tile = next_of_lane(lane, tile, n++)) {
        int ti, tj;
        ds_tile(p, tile, ti, tj);
        const int i0 = ti * (2 * BM) + (int)rank * BM;
        const int j0 = tj * BN + (int)rank * (BN / 2);
        for (int kb = 0; kb < p.k_blocks; ++kb, ++it) {
          const int s = it % DS_STAGES;
          const uint32_t ph = (it / DS_STAGES) & 1u;
          if (!mbar_wait_cluster(smem_u32(&bars->empty[s]), ph ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t bar = mapa_shared(smem_u32(&bars->full[s]), 0);
          if (leader) mbar_arrive_expect_tx(smem_u32(&bars->full[s]), 2 * DS_STAGE_BYTES);
          if (leader && kb == ask_at) mbar_arrive(smem_u32(&bars->wanted));
          uint8_t* st = base + s * DS_STAGE_BYTES;
          // Each box is 64 contiguous features x 64 tokens = one 8 KiB MN-major chunk.
#pragma unroll
          for (int m = 0; m < 2; ++m)
            tma_load_2d_pair(smem_u32(st) + m * 8192, &tmap_dy, bar, i0 + 64 * m, kb * BK);
#pragma unroll
          for (int m = 0; m < 2; ++m)
            tma_load_2d_pair(smem_u32(st) + 16384 + m * 8192, &tmap_x, bar, j0 + 64 * m, kb * BK);
        }
      }
    }
  } else if (warp == 1) {
    if (leader) if (const uint32_t lane = elect_lane(); lane == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(2 * BM, BN, 1, 1);
      const uint64_t adesc0 = smem_desc_sw128(smem_u32(base), 8192, 1024);
      const uint64_t bdesc0 = smem_desc_sw128(smem_u32(base) + 16384, 8192, 1024);
      const uint32_t full0 = smem_u32(&bars->full[0]), empty0 = smem_u32(&bars->empty[0]);
      uint32_t s = 0, ph = 0;
      int local = 0;
      bool ok = true;
      for (int tile = pair; ok && tile >= 0; tile = next_of_lane(lane, tile, (uint32_t)local++)) {
        const int buf = local & 1;
        const uint32_t acc_ph = (local >> 1) & 1u;
        if (!mbar_wait_cluster(smem_u32(&bars->acc_empty[buf]), acc_ph ^ 1u, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + buf * BN;
        for (int kb = 0; kb < p.k_blocks; ++kb) {
          if (!mbar_wait_cluster(full0 + s * 8, ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint64_t adesc = adesc0 + s * (DS_STAGE_BYTES >> 4), bdesc = bdesc0 + s * (DS_STAGE_BYTES >> 4);
          const uint32_t at = s;
          if (++s == DS_STAGES) {
            s = 0;
            ph ^= 1u;
          }
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k)
            mma_bf16_ss_pair(d_tmem, adesc + k * (UMMA_K * 128 / 16), bdesc + k * (UMMA_K * 128 / 16), idesc, (kb | k) != 0 ? 1u : 0u);
          mma_commit_pair(empty0 + at * 8, 3);
        }
        if (ok) mma_commit_pair(smem_u32(&bars->acc_full[buf]), 3);
      }
    }
  } else if (warp == 3) {
    // packed codes of this CTA's 128 rows x 256 columns, a tile ahead of the epilogue (one lane)
    if (PKTMA) if (const uint32_t lane = elect_lane(); lane == 0) {
      int local = 0;
      for (int tile = pair; tile >= 0; tile = next_of_lane(lane, tile, (uint32_t)local++)) {
        int ti, tj;
        ds_tile(p, tile, ti, tj);
        const int ps = local & 1;
        if (!mbar_wait(smem_u32(&bars->pk_empty[ps]), ((local >> 1) & 1u) ^ 1u, abort_flag)) break;
        const uint32_t bar = smem_u32(&bars->pk_full[ps]);
        mbar_arrive_expect_tx(bar, BM * 32 * BITS);
        tma_load_2d(smem_u32(sm_pk + ps * DS_PK_BYTES), &tmap_pk, bar, tj * (8 * BITS), ti * (2 * BM) + (int)rank * BM);
      }
    }
  } else if (warp == 2) {
    // DYNAMIC: takes over a tile that no CTA pair has been started for and tells all roles of both CTAs.  Late in the tile
    // before: what a pair holds is not there for one that becomes idle.
    if (DYNAMIC && leader) if (const uint32_t lane = elect_lane(); lane == 0) {
      const uint32_t answered = smem_u32(&bars->answered), response = smem_u32(&bars->response);
      for (uint32_t n = 0;; ++n) {
        const uint32_t q = n % DS_NEXT;
        if (!mbar_wait(smem_u32(&bars->wanted), n & 1u, abort_flag)) break;
        if (!mbar_wait_cluster(smem_u32(&bars->next_empty[q]), ((n / DS_NEXT) & 1u) ^ 1u, abort_flag)) break;
        mbar_arrive_expect_tx(answered, 16);
        launch_try_cancel(response, answered);
        if (!mbar_wait(answered, n & 1u, abort_flag)) break;
        uint32_t first_cta;
        const int tile = launch_cancelled(response, first_cta) ? (int)(first_cta >> 1) : -1;
        fence_proxy_async_smem();                      // it has been read: the next answer may be written over it
        bars->next_tile[q] = tile;
        st_cluster_u32(mapa_shared(smem_u32(&bars->next_tile[q]), 1), (uint32_t)tile);
        mbar_arrive(smem_u32(&bars->next_full[q]));
        mbar_arrive_cluster_release_all(mapa_shared(smem_u32(&bars->next_full[q]), 1));
        if (tile < 0) break;
      }
    }
  } else if (warp >= 4) {
    // Epilogue: thread = one weight row i (TMEM lane) and one 128-column half.
    const int quarter = warp & 3;
    const int half = (warp - 4) >> 2;
    const int npieces = p.K / p.piece;
    const int cpp = p.piece >> 5;                    // 32-column chunks per piece: 1, 2 or 4
    const uint32_t acc_empty_leader0 = mapa_shared(smem_u32(&bars->acc_empty[0]), 0);
    const uint32_t acc_empty_leader1 = mapa_shared(smem_u32(&bars->acc_empty[1]), 0);
    int local = 0;
    bool ok = true;
    for (int tile = pair; ok && tile >= 0; tile = next_of_warp(tile, (uint32_t)local++)) {
      int ti, tj;
      ds_tile(p, tile, ti, tj);
      const int i0 = ti * (2 * BM) + (int)rank * BM;
      const int c0 = tj * BN + half * 128;             // this thread's columns [c0, c0 + 128)
      const int buf = local & 1;
      const uint32_t acc_ph = (local >> 1) & 1u;
      const int i = i0 + quarter * 32 + lane;
      const bool row_ok = i < p.N;
      // Zero-points and optimizer state of the tile do not depend on the accumulator: they are
      // requested before the wait for it, one vector of the thread's pieces per array.
      const bool live = row_ok && c0 < p.K;
      const int n_pieces = live ? min(4 / cpp, (p.K - c0) / p.piece) : 0;
      // the pieces of a thread are one aligned vector (m and v may have any 4-byte address)
      const bool vec = p.vec_ok && (npieces & (4 / cpp - 1)) == 0;
      const size_t e0 = (size_t)i * npieces + c0 / p.piece;  // first piece
      uint32_t z[4] = {0u, 0u, 0u, 0u};
      float zreal[4], sc[4], ms[4], mm[4], mv[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        zreal[k] = sc[k] = ms[k] = mm[k] = mv[k] = 0.0f;
        if (k < n_pieces) {
          const size_t gi = (size_t)i * p.G + (p.G == 1 ? 0 : (c0 + k * p.piece) / p.g);
          if (DZ && p.zeros_f) zreal[k] = ld_global(p.zeros_f + gi);
          else z[k] = ld_global(p.zeros + gi);
          if (DZ && p.piece == p.g) sc[k] = ld_global(p.scales + gi);
        }
      }
      if (ADAM) {
        load_pieces(p.adam_s + e0, n_pieces, vec, ms);
        load_pieces(p.adam_m + e0, n_pieces, vec, mm);
        load_pieces(p.adam_v + e0, n_pieces, vec, mv);
      }
      // the packed codes of the tile (see warp 3)
      uint32_t w[4][BITS];
      if (PKTMA) {
        const int ps = local & 1;
        if (!warp_wait(smem_u32(&bars->pk_full[ps]), acc_ph, abort_flag)) { ok = false; break; }
        const uint8_t* src = sm_pk + ps * DS_PK_BYTES;
        const int row = quarter * 32 + lane;
        if constexpr (BITS == 4) {
          // rows of 128 bytes, 16-byte chunk c at c ^ (row % 8): the code map's swizzle
#pragma unroll
          for (int cc = 0; cc < 4; ++cc) {
            const uint4 v = *reinterpret_cast<const uint4*>(src + row * 128 + (((half * 4 + cc) ^ (row & 7)) << 4));
            w[cc][0] = v.x; w[cc][1] = v.y; w[cc][2] = v.z; w[cc][3] = v.w;
          }
        } else {
          const uint4* at = reinterpret_cast<const uint4*>(src + row * 96 + half * 48);
          const uint4 a = at[0], b = at[1], c = at[2];
          const uint32_t f[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
#pragma unroll
          for (int cc = 0; cc < 4; ++cc)
#pragma unroll
            for (int q = 0; q < 3; ++q) w[cc][q] = f[3 * cc + q];
        }
      } else {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
#pragma unroll
          for (int q = 0; q < BITS; ++q)
            w[cc][q] = row_ok && c0 + cc * 32 < p.K ? ld_global(p.qw + (size_t)i * p.wpr + ((c0 >> 5) + cc) * BITS + q) : 0u;
        }
      }
      if (!warp_wait_cluster(smem_u32(&bars->acc_full[buf]), acc_ph, abort_flag)) { ok = false; break; }
      tc_fence_after();
      float acc = 0.0f, accz = 0.0f;
      float r[4] = {0.f, 0.f, 0.f, 0.f}, rz[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        if (c0 + cc * 32 >= p.K) break;
        const uint32_t zc = cpp == 1 ? z[cc] : cpp == 2 ? z[cc >> 1] : z[0];
        const float zr = cpp == 1 ? zreal[cc] : cpp == 2 ? zreal[cc >> 1] : zreal[0];
        uint32_t v[32];
        tmem_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + buf * BN + half * 128 + cc * 32, v);
        uint32_t zi = zc;
        float delta = 0.0f;   // real-valued zero-point = zi + delta
        if (DZ && p.zeros_f) dq::split_zero_point<BITS>(zr, zi, delta);
        uint32_t o[16];
        dq::unit32_natural<BITS, false>(w[cc], zi, 0.0f, o);
        tmem_ld_wait();   // warp-wide: every lane executes it, ragged rows included
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          acc = fmaf(__uint_as_float(v[2 * q]), __uint_as_float(o[q] << 16), acc);
          acc = fmaf(__uint_as_float(v[2 * q + 1]), __uint_as_float(o[q] & 0xFFFF0000u), acc);
          if (DZ) accz += __uint_as_float(v[2 * q]) + __uint_as_float(v[2 * q + 1]);
        }
        if (((cc + 1) & (cpp - 1)) == 0) {
          // with a real-valued zero-point, sum (q - z) dW = sum (q - zi) dW - delta * sum dW;
          // partial pieces are stored raw and corrected after they have been added
          if (DZ && p.zeros_f && p.piece == p.g) acc = fmaf(-delta, accz, acc);
          if (cpp == 1) { r[cc] = acc; rz[cc] = accz; }
          else if (cpp == 2) { r[cc >> 1] = acc; rz[cc >> 1] = accz; }
          else { r[0] = acc; rz[0] = accz; }
          acc = 0.0f;
          accz = 0.0f;
        }
      }
      store_pieces(p.out + e0, n_pieces, vec, r);
      if (ADAM) {
        // pieces are whole groups here (the launcher only asks for this then): r holds the final
        // dS of this row's scales, owned by this thread alone
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k < n_pieces) adamw_update(ms[k], r[k], mm[k], mv[k], p.adam);
        // the kernels this one runs beside read the scales
        if (beside && local == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
        store_pieces(p.adam_s + e0, n_pieces, vec, ms);
        store_pieces(p.adam_m + e0, n_pieces, vec, mm);
        store_pieces(p.adam_v + e0, n_pieces, vec, mv);
      }
      if (DZ) {
        // a piece that is a whole group is dZ itself: -s * sum of dW; otherwise the reduction
        // kernel applies -s after adding the pieces
#pragma unroll
        for (int k = 0; k < 4; ++k) rz[k] *= p.piece == p.g ? -sc[k] : 1.0f;
        store_pieces(p.out_z + e0, n_pieces, vec, rz);
      }
      tc_fence_before();
      if (PKTMA) fence_proxy_async_smem();           // the codes have been read: their slot goes back
      __syncwarp();
      if (PKTMA && lane == 0) mbar_arrive(smem_u32(&bars->pk_empty[local & 1]));
      if (lane == 0) mbar_arrive_cluster(buf ? acc_empty_leader1 : acc_empty_leader0);
    }
  }

  if (*abort_flag) drain_after_abort();
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // no CTA leaves while its peer may still signal its barriers
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, TMEM_COLS);
  }
  if (threadIdx.x == 0 && bars->abort_flag) {
    atomicExch(p.status, (int)PEQA_ERR_DEVICE_TIMEOUT);
    p.status[1] = (int)blockIdx.x;
  }
  // beside another kernel: this one has not ended before that one has (any CTA but the running ones may have been taken over)
  if (beside && threadIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// An output's pieces lie side by side.  A thread that adds up its own reads every line of memory as often as the
// line has pieces, out of L1; launched programmatically these kernels find their SM laid out for the contraction
// before them, with next to no L1, so from 25 pieces on a block of 128 threads reads the pieces of 32 outputs row by row
// into shared memory and its first warp adds them up, in index order all the same.  us, contraction and
// reduction, a thread each / this: 456 x 9600 at 60 tokens (75 pieces) 17.8 / 11.3, 1128 x 6016 at 56 16.8 / 10.6,
// 6800 x 13440 at 75 62 / 50; with fewer pieces a thread each is faster (10048 x 1280 at 53 tokens 11.1 / 11.9, 2304 columns
// 7.2 / 7.7).
constexpr int kWidePieces = 25, kWideThreads = 128, kWideRows = 32;
__device__ __forceinline__ float sum_pieces_wide(const float* partial, long long n_out, int pieces) {
  __shared__ float tile[kWideRows][33];
  const long long e0 = (long long)blockIdx.x * kWideRows;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float acc = 0.0f;
  for (int q0 = 0; q0 < pieces; q0 += 32) {
#pragma unroll
    for (int k = 0; k < kWideRows / (kWideThreads / 32); ++k) {
      const int row = warp + k * (kWideThreads / 32);
      if (e0 + row < n_out && q0 + lane < pieces) tile[row][lane] = partial[(e0 + row) * pieces + q0 + lane];
    }
    __syncthreads();
    if (warp == 0) {
      const int n = min(32, pieces - q0);
      for (int q = 0; q < n; ++q) acc += tile[lane][q];     // (of rows beyond the last one: never stored)
    }
    __syncthreads();
  }
  return acc;
}

// Real-valued zero-point, groups wider than a piece: dS = sum(pieces) - delta * sum(dW pieces)
// and dZ = -s * sum(dW pieces).
template <bool WIDE>
__global__ void ds_reduce_zf_kernel(const float* partial_s, const float* partial_w,
                                    float* dS, float* dZ, long long n_out,
                                    int pieces_per_group, const float* zeros_f,
                                    const float* scales, int bits) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  long long e = (long long)blockIdx.x * (WIDE ? kWideRows : blockDim.x) + threadIdx.x;
  float acc_s = 0.0f, acc_w = 0.0f;
  if constexpr (WIDE) {
    acc_s = sum_pieces_wide(partial_s, n_out, pieces_per_group);
    acc_w = sum_pieces_wide(partial_w, n_out, pieces_per_group);
    if (threadIdx.x >= kWideRows) return;
  }
  if (e >= n_out) return;
  if constexpr (!WIDE) {
    for (int q = 0; q < pieces_per_group; ++q) {
      acc_s += partial_s[e * pieces_per_group + q];
      acc_w += partial_w[e * pieces_per_group + q];
    }
  }
  uint32_t zi;
  float delta;
  if (bits == 3) dq::split_zero_point<3>(zeros_f[e], zi, delta);
  else dq::split_zero_point<4>(zeros_f[e], zi, delta);
  dS[e] = fmaf(-delta, acc_w, acc_s);
  dZ[e] = -scales[e] * acc_w;
}

// dS[i, gi] = sum of the group's partial pieces, in index order (deterministic); with
// neg_scales the sum is multiplied by -s[i, gi] (the zero-point gradient); with adam_s the
// AdamW step on scale e follows at once.
template <bool WIDE>
__global__ void ds_reduce_kernel(const float* partial, float* dS,
                                 long long n_out, int pieces_per_group,
                                 const float* neg_scales, AdamWConsts adam,
                                 float* adam_s, float* adam_m,
                                 float* adam_v) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  long long e = (long long)blockIdx.x * (WIDE ? kWideRows : blockDim.x) + threadIdx.x;
  float acc = 0.0f;
  if constexpr (WIDE) {
    acc = sum_pieces_wide(partial, n_out, pieces_per_group);
    if (threadIdx.x >= kWideRows) return;
  }
  if (e >= n_out) return;
  if constexpr (!WIDE) {
    const float* src = partial + e * pieces_per_group;
    for (int q = 0; q < pieces_per_group; ++q) acc += src[q];
  }
  dS[e] = neg_scales ? -neg_scales[e] * acc : acc;
  if (adam_s) {
    float sv = adam_s[e], mv = adam_m[e], vv = adam_v[e];
    adamw_update(sv, acc, mv, vv, adam);
    adam_s[e] = sv;
    adam_m[e] = mv;
    adam_v[e] = vv;
  }
}

// dS[i] = sum over the token blocks' partial sums, in a fixed order (eight interleaved chains, then
// these in order), and the AdamW step on scale i with adam_s.
__global__ void ds_channel_kernel(const float* part, float* dS, int N, int slots,
                                  AdamWConsts adam, float* adam_s, float* adam_m,
                                  float* adam_v) {
  // Launched programmatically: its blocks stand ready when the kernel before (dX) ends (LLaMA-7B MLP, 66
  // tokens, 1.5 us a linear).  The next kernel, which reads the scales written here, is not let in early.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ float sums[8][33];
  const int i = blockIdx.x * 32 + threadIdx.x;
  float acc = 0.0f;
  if (i < N)
    for (int q = threadIdx.y; q < slots; q += 8) acc += __ldcg(part + (size_t)q * N + i);
  sums[threadIdx.y][threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.y != 0 || i >= N) return;
  for (int y = 1; y < 8; ++y) acc += sums[y][threadIdx.x];
  dS[i] = acc;
  if (adam_s) {
    float sv = adam_s[i], mv = adam_m[i], vv = adam_v[i];
    adamw_update(sv, acc, mv, vv, adam);
    adam_s[i] = sv;
    adam_m[i] = mv;
    adam_v[i] = vv;
  }
}

// --------------------------------------------------------------- host side

// bf16 row-major [outer, inner] tensor, box = [box_outer rows, 64 elements], 128B swizzle,
// out-of-bounds elements read as zero.
int make_tmap_bf16(CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer,
                   uint32_t box_outer) {
  EncodeTiledFn enc = nullptr;
  PEQA_TRY(tensor_map_encoder(&enc));
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {inner * 2};
  cuuint32_t box[2] = {64, box_outer};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                   box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return cuda_fail(cudaErrorInvalidValue);
  return PEQA_OK;
}

int sm_count(int* n) {
  static thread_local int cached_dev = -1, cached_n = 0;
  int dev = 0;
  PEQA_CUDA(cudaGetDevice(&dev));
  if (dev != cached_dev) {
    PEQA_CUDA(cudaDeviceGetAttribute(&cached_n, cudaDevAttrMultiProcessorCount, dev));
    cached_dev = dev;
  }
  *n = cached_n;
  return PEQA_OK;
}

template <int BITS, bool TRANS, bool FOLD>
int launch_qgemm_t(const CUtensorMap& tmap, const QGemmParams& p, int grid, cudaStream_t st) {
  auto kern = qgemm_kernel<BITS, TRANS, FOLD>;
  static std::atomic<uint64_t> done{0};
  PEQA_TRY(allow_smem(kern, SMEM_BYTES, done));
  kern<<<grid, kQgemmThreads, SMEM_BYTES, st>>>(tmap, p);
  PEQA_CUDA(cudaGetLastError());
  return PEQA_OK;
}

int launch_qgemm(const peqa_qweight_t* w, const float* zeros_f, int g, const void* act, int T,
                 void* out, bool trans, cudaStream_t st) {
  QGemmParams p;
  p.qw = w->qweight;
  p.zeros = w->zeros;
  p.zeros_f = zeros_f;
  p.scales = w->scales;
  p.out = static_cast<__nv_bfloat16*>(out);
  p.N = w->out_features;
  p.K = w->in_features;
  p.g = g;
  p.G = p.K / g;
  p.g_shift = -1;
  for (int b = 5; b < 31; ++b)
    if ((1 << b) == g) p.g_shift = b;
  p.T = T;
  p.wpr = p.K * w->bits / 32;
  p.R = trans ? p.K : p.N;
  p.C = trans ? p.N : p.K;
  p.r_tiles = (p.R + BM - 1) / BM;
  p.t_tiles = (T + BN - 1) / BN;
  p.k_blocks = (p.C + BK - 1) / BK;
  PEQA_TRY(status_word(st, &p.status));
  CUtensorMap tmap;
  PEQA_TRY(make_tmap_bf16(&tmap, act, (uint64_t)p.C, (uint64_t)T, BN));
  int sms = 0;
  PEQA_TRY(sm_count(&sms));
  const int tiles = p.r_tiles * p.t_tiles;
  const int grid = tiles < sms ? tiles : sms;
  const bool fold = trans || p.G > 1 || zeros_f != nullptr;
  // only 3-bit rows have such a pitch: K is a multiple of 64
  if (trans) return launch_qgemm_t<3, true, true>(tmap, p, grid, st);
  return fold ? launch_qgemm_t<3, false, true>(tmap, p, grid, st)
              : launch_qgemm_t<3, false, false>(tmap, p, grid, st);
}

int gcd_int(int a, int b) { return b == 0 ? a : gcd_int(b, a % b); }

// Columns per dS output piece: the largest of {32, 64, 128} that divides g, so
// that a piece never crosses a group or a 128-column epilogue half.
int ds_piece(int g) { return gcd_int(g, 128); }

}  // namespace

int part_tokens(const peqa_qweight_t* w, int T_call) {
  const bool channel_scales = effective_group(w->in_features, w->group_size) == w->in_features;
  int unit = 8;     // 16-byte aligned slices
  for (int trans = 0; trans < 2; ++trans)
    if (fwd_pair_supported(w) && split_is_faster(w, T_call, trans, channel_scales && !trans)) {
      const int part = split_part_tokens(w, T_call, trans);
      unit = unit / gcd_int(unit, part) * part;
    }
  return unit;
}

int launch_fwd(const peqa_qweight_t* w, const float* zeros_f, int g, const void* X, int T, void* Y,
               cudaStream_t st, int T_call, int t0, Side side) {
  const bool channel_scales = g == w->in_features && !zeros_f;
  if (fwd_pair_supported(w) && split_is_faster(w, T_call, false, channel_scales))
    return launch_split(w, zeros_f, g, X, T, Y, false, nullptr, nullptr, st, T_call, t0, side);
  if (fwd_pair_supported(w)) return launch_fwd_pair(w, zeros_f, g, X, T, Y, nullptr, nullptr, st, side);
  return launch_qgemm(w, zeros_f, g, X, T, Y, false, st);
}

int launch_dx(const peqa_qweight_t* w, const float* zeros_f, int g, const void* dY, int T, void* dX,
              cudaStream_t st, int T_call, int t0, Side side) {
  if (dx_pair_supported(w) && split_is_faster(w, T_call, true, false))
    return launch_split(w, zeros_f, g, dY, T, dX, true, nullptr, nullptr, st, T_call, t0, side);
  if (dx_pair_supported(w)) return launch_dx_pair(w, zeros_f, g, dY, T, dX, side, st);
  return launch_qgemm(w, zeros_f, g, dY, T, dX, true, st);
}

int fwd_ds_slots(const peqa_qweight_t* w, int g, int T) {
  if (g != w->in_features || !fwd_pair_supported(w)) return 0;
  // dS = sum_t dY * u from the forward's fp32 sums instead of a contraction of its own (training
  // step of one linear, before -> after in us, and error of dS against binary64): 11008 x 4096 at
  // 4096 tokens 742 -> 611, 4.4e-6 -> 1.4e-7; 22016 x 8192 at 2048 tokens 1406 -> 1040; 4096 x 4096
  // at 16 tokens (2^28 products) 39 -> 25, 2048 x 2048 at 64 (2^28) 26 -> 20.5.  Below 2^28 it would
  // save 3 to 6 us of a step too (1024 x 1024 at 128 tokens 25 -> 21, 256 x 256 at 64 19.5 -> 16.5); there
  // the call stays the exact composition of the single calls, whose dS differs from this one in its
  // last bits.
  if ((double)T * w->out_features * w->in_features < (double)(1 << 28)) return 0;
  const int slots = split_is_faster(w, T, false, true) ? split_ds_slots(w, T) : 2 * ((T + 255) / 256);
  // The partial sums go to the workspace the caller was asked for, whose size does not depend on
  // T (about T <= K fits).  Held against that size and not against the one that was given, so that
  // the bits of dS depend on the shape and T alone and a pointer that is not needed is not used.
  return (size_t)slots * w->out_features * sizeof(float) <= ds_workspace_bytes(w, g, T) ? slots : 0;
}

int launch_fwd_ds(const peqa_qweight_t* w, const void* X, const void* dY, int T, void* Y, float* ds_part,
                  cudaStream_t st, Side side) {
  const int g = w->in_features;
  if (split_is_faster(w, T, false, true)) return launch_split(w, nullptr, g, X, T, Y, false, dY, ds_part, st, T, 0, side);
  return launch_fwd_pair(w, nullptr, g, X, T, Y, dY, ds_part, st, side);
}

int launch_ds_channel(const peqa_qweight_t* w, const float* ds_part, int slots, float* dS, const DsAdam* adam,
                      cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((w->out_features + 31) / 32, 1, 1);
  cfg.blockDim = dim3(32, 8, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  PEQA_CUDA(cudaLaunchKernelEx(&cfg, ds_channel_kernel, ds_part, dS, (int)w->out_features, slots, adam ? adam->c : AdamWConsts{},
                               adam ? adam->scales : nullptr, adam ? adam->m : nullptr, adam ? adam->v : nullptr));
  return PEQA_OK;
}

size_t ds_workspace_bytes(const peqa_qweight_t* w, int g, int T) {
  (void)T;
  const int piece = ds_piece(g);
  if (piece == g) return 0;
  return (size_t)w->out_features * (size_t)(w->in_features / piece) * sizeof(float);
}

// with dZ: a second array of partial sums behind the first
size_t dsdz_workspace_bytes(const peqa_qweight_t* w, int g, int T) {
  return 2 * ds_workspace_bytes(w, g, T);
}

int launch_ds(const peqa_qweight_t* w, const float* zeros_f, int g, const void* X, const void* dY,
              int T, float* dS, float* dZ, const DsAdam* adam, void* workspace,
              size_t workspace_bytes, cudaStream_t st, Side side) {
  if (adam && dZ) return PEQA_ERR_BAD_SHAPE;   // dZ reads the scales the step would be rewriting
  if (zeros_f && !dZ) return PEQA_ERR_NULL;    // the correction needs the sums dZ is made of
  (void)workspace_bytes;
  DsParams p;
  p.side = side;
  p.qw = w->qweight;
  p.zeros = w->zeros;
  p.zeros_f = zeros_f;
  p.N = w->out_features;
  p.K = w->in_features;
  p.g = g;
  p.G = p.K / g;
  p.T = T;
  p.wpr = p.K * w->bits / 32;
  p.piece = ds_piece(g);
  const bool direct = (p.piece == g);
  p.out = direct ? dS : static_cast<float*>(workspace);
  p.scales = w->scales;
  const size_t n_pieces = (size_t)p.N * (size_t)(p.K / p.piece);
  p.out_z = dZ ? (direct ? dZ : static_cast<float*>(workspace) + n_pieces) : nullptr;
  p.adam = adam ? adam->c : AdamWConsts{};
  p.adam_s = adam ? adam->scales : nullptr;
  p.adam_m = adam ? adam->m : nullptr;
  p.adam_v = adam ? adam->v : nullptr;
  const bool adam_in_kernel = adam && direct;
  p.vec_ok = aligned16(p.out) && aligned16(p.out_z) && aligned16(p.adam_s) && aligned16(p.adam_m) && aligned16(p.adam_v);
  p.i_tiles = (p.N + 2 * BM - 1) / (2 * BM);   // 256-row pair tiles
  p.j_tiles = (p.K + BN - 1) / BN;
  p.k_blocks = (T + BK - 1) / BK;
  {
    // a band of about 32 MiB of one operand; band the dimension that gives less HBM traffic:
    // rows: dY once + X once per band of rows; columns: X once + dY once per band of columns
    int band = (int)((32u << 20) / ((size_t)512 * (size_t)T));
    band = band < 1 ? 1 : band;
    const double by_rows = (double)p.N + (double)p.K * ((p.i_tiles + band - 1) / band);
    const double by_cols = (double)p.K + (double)p.N * ((p.j_tiles + band - 1) / band);
    p.band_rows = by_rows <= by_cols ? 1 : 0;
    const int dim = p.band_rows ? p.i_tiles : p.j_tiles;
    p.band = band < dim ? band : dim;
  }
  PEQA_TRY(status_word(st, &p.status));
  CUtensorMap tmap_dy, tmap_x;
  PEQA_TRY(make_tmap_bf16(&tmap_dy, dY, (uint64_t)p.N, (uint64_t)T, BK));
  PEQA_TRY(make_tmap_bf16(&tmap_x, X, (uint64_t)p.K, (uint64_t)T, BK));
  int sms = 0;
  PEQA_TRY(sm_count(&sms));
  const int tiles = p.i_tiles * p.j_tiles;
  const int max_pairs = sms / 2;
  // Taking tiles over pays but for short tiles of a step with AdamW in the kernel, where the store of a pair's first tile waits for the
  // kernels beside: there from where shapes that lose and shapes that gain come to the same.  us, dealt / taken over, steps with AdamW here: 8192 x 8192 in groups of 64 at 64 tokens 99 / 102, at 256 134.7 /
  // 136.5, at 384 187.5 / 190.3, at 512 215.5 / 215.8, at 2048 633 / 609; 2304 x 2304 in groups of 64 at 64 22.3 / 21.5, at 256
  // 31.4 / 33.8, at 384 39.6 / 41.4, at 512 45.2 / 46.3, at 1000 47.3 / 45.7; 4096 x 4096 in groups of 128 at 384 59.0 / 57.6, at
  // 700 87.2 / 87.5, at 2048 174 / 164; five shapes lose 1.8 % at 256, seven 0.3 % at 384, five 0.2 % at 512, nine gain 2.1 % at 1000.  Without AdamW here: real
  // zero-points, 2304 x 2304 in groups of 64 at 64 14.8 / 12.8, at 200 20.5 / 14.4, 4096 x 4096 per channel at 64 27.5 / 27.8, at 384 39.7 /
  // 38.6, 4096 x 11008 in groups of 128 at 40 47.6 / 45.3, at 256 67.3 / 61.9; step in groups of 256, 4096 x 4096 at 64 34.4 / 34.7, at 384 53.9 / 51.1.
  const bool pktma = ((size_t)p.wpr * 4) % 16 == 0;   // 4-bit: always; 3-bit: K % 128 == 0
  const bool dynamic = side == kBeside && pktma && tiles > max_pairs && (!adam_in_kernel || p.k_blocks >= 6);
  const int pairs = tiles < max_pairs || dynamic ? tiles : max_pairs;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs, 1, 1);
  cfg.blockDim = dim3(kDsThreads, 1, 1);
  cfg.dynamicSmemBytes = DS_SMEM_BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  // barrier set-up and the tensor-memory allocation may overlap the tail of the kernel before
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  CUtensorMap tmap_pk = tmap_x;
  if (pktma) {
    EncodeTiledFn enc = nullptr;
    PEQA_TRY(tensor_map_encoder(&enc));
    cuuint64_t dims[2] = {(cuuint64_t)p.wpr, (cuuint64_t)p.N};
    cuuint64_t strides[1] = {(cuuint64_t)p.wpr * 4};
    cuuint32_t box[2] = {8u * w->bits, (cuuint32_t)BM};
    cuuint32_t estr[2] = {1, 1};
    if (enc(&tmap_pk, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<uint32_t*>(w->qweight), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            w->bits == 4 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cuda_fail(cudaErrorInvalidValue);
  }
#define PEQA_DS_LAUNCH_T(B, Z, A, P, D)                                                               \
  do {                                                                                               \
    auto kern = ds_kernel<B, Z, A, P, D>;                                                            \
    static std::atomic<uint64_t> done{0};                                                            \
    PEQA_TRY(allow_smem(kern, DS_SMEM_BYTES, done));                                                 \
    PEQA_CUDA(cudaLaunchKernelEx(&cfg, kern, tmap_dy, tmap_x, tmap_pk, p));                          \
  } while (0)
#define PEQA_DS_LAUNCH(B, Z, A)                     \
  do {                                              \
    if (B == 4 || pktma) {                          \
      if (dynamic) PEQA_DS_LAUNCH_T(B, Z, A, true, true); \
      else PEQA_DS_LAUNCH_T(B, Z, A, true, false);  \
    } else {                                        \
      PEQA_DS_LAUNCH_T(B, Z, A, (B == 4), false);   \
    }                                               \
  } while (0)
  if (w->bits == 4) {
    if (dZ) PEQA_DS_LAUNCH(4, true, false);
    else if (adam_in_kernel) PEQA_DS_LAUNCH(4, false, true);
    else PEQA_DS_LAUNCH(4, false, false);
  } else {
    if (dZ) PEQA_DS_LAUNCH(3, true, false);
    else if (adam_in_kernel) PEQA_DS_LAUNCH(3, false, true);
    else PEQA_DS_LAUNCH(3, false, false);
  }
#undef PEQA_DS_LAUNCH
#undef PEQA_DS_LAUNCH_T
  if (!direct) {
    const long long n_out = (long long)p.N * p.G;
    const int ppg = g / p.piece;
    const bool wide = ppg >= kWidePieces;
    const int threads = wide ? kWideThreads : 256;
    const int blocks = (int)((n_out + (wide ? kWideRows : 256) - 1) / (wide ? kWideRows : 256));
    if (zeros_f)
      return launch_after(wide ? ds_reduce_zf_kernel<true> : ds_reduce_zf_kernel<false>, blocks, threads, st, p.out, p.out_z, dS,
                          dZ, n_out, ppg, zeros_f, w->scales, (int)w->bits);
    auto reduce = wide ? ds_reduce_kernel<true> : ds_reduce_kernel<false>;
    PEQA_TRY(launch_after(reduce, blocks, threads, st, p.out, dS, n_out, ppg, nullptr, p.adam, p.adam_s, p.adam_m, p.adam_v));
    if (dZ)
      PEQA_TRY(launch_after(reduce, blocks, threads, st, p.out_z, dZ, n_out, ppg, w->scales, AdamWConsts{}, nullptr, nullptr,
                            nullptr));
  }
  return PEQA_OK;
}

}  // namespace peqa
