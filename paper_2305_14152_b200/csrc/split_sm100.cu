// Forward and dX of the PEQA layer for few tokens:
//
//   TRANS = false   Y[t,i]  = sum_j X[t,j]  * W_hat[i,j]     (Eq. 2)
//   TRANS = true    dX[t,j] = sum_i dY[t,i] * W_hat[i,j]
//
// With a few hundred tokens the CTA-pair kernels (512 tokens x 256 outputs per tile) keep a
// handful of SMs busy and multiply mostly padding.  What bounds such a call is rebuilding the
// weights, so this kernel spreads exactly that over the whole chip: a tile is 128 outputs x up to
// 256 tokens (the token side is the MMA "N" and is cut to a multiple of 16, so padding costs
// nothing), and the contraction of a tile is cut across the CTAs of a thread-block cluster.
//
// A cluster of `csize` CTAs owns `q` <= csize tiles.  Their q * k_blocks stages, tile-major, are
// cut into csize equal contiguous ranges, one per CTA; a range is never longer than a tile, so a
// CTA works on at most two tiles and holds their partial sums in two tensor-memory accumulators.
// When its stages are done a CTA copies its partial sums to its own shared memory (over the stage
// buffers), the cluster synchronises, and every CTA adds up one slice of the rows of each tile,
// reading the contributors' shared memory in rank order: no workspace, no atomics, and the result
// does not depend on timing.
//
// Warps: 0 activation TMA, 1 MMA issuer, 2 tensor memory, 3 code TMA, 4-19 dequant.  The weights
// are the MMA "A" operand (M = 128).  Forward: a dequant thread is a row of them, and stores its half stage
// into its lane of TENSOR MEMORY (32 columns), beside the accumulators: shared memory, which carried the
// weights twice, is left to the activations, and a tile of 256 tokens keeps as many stages as one of 80.
// us before / after: 22016 x 8192 at 256 tokens 124 / 109, 8192 x 8192 at 512 68 / 55, 4096 x 11008 at 1001
// 89 / 77, 2048 x 5504 at 150 17.8 / 14.4, 4096 x 4096 at 77 12.8 / 12.4 (an MMA of 80 tokens takes 40 cycles so, 52 with A in
// shared memory, behind an elected lane).  dX: thread and contraction run the other way, so the weights are rebuilt in shared
// memory, MN-major, as in the single-CTA kernel of gemm_sm100.cu.  Four groups
// of four warps take the half stages round-robin; scales and zero-points are fetched one turn ahead.
#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "dequant.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"

namespace peqa {

namespace {

using namespace ptx;

constexpr int SM_ROWS = 128;                  // outputs per tile (MMA M, TMEM lanes)
constexpr int SM_BK = 128;                    // contraction elements per stage: two halves of 64
constexpr int SM_HALF = 64;                   // (the reach of the 128-byte swizzle)
constexpr int SM_MAX_NT = 256;                // tokens per tile
constexpr int SM_A_BYTES = SM_ROWS * SM_HALF * 2;   // weights of one half
constexpr int SM_PK_BYTES = 8192;             // packed codes of one stage
constexpr int SM_PK_SLOTS = 4;
constexpr int SM_MAX_STAGES = 4;
constexpr int kSplitThreads = 640;
constexpr int kSplitWorkers = 512;            // threads of the dequant warps
constexpr int SM_DUMP_TOK = 128;              // tokens reduced per pass
constexpr int SM_SMEM_LIMIT = 227 * 1024;
constexpr int SM_SMEM_FIXED = SM_PK_SLOTS * SM_PK_BYTES + 1024 /*align*/ + 512 /*barriers*/;

struct SplitBarriers {
  uint64_t full[SM_MAX_STAGES];       // weight tile written and activation bytes landed
  uint64_t empty[SM_MAX_STAGES];      // MMAs that read the stage completed
  uint64_t full_pk[SM_PK_SLOTS];
  uint64_t empty_pk[SM_PK_SLOTS];
  uint64_t acc_full;                  // every MMA of this CTA completed
  uint32_t tmem_base;
  int abort_flag;
  int wait_limit_us;    // must follow abort_flag (read by the bounded waits)
};

struct SplitParams {
  const uint8_t* zeros;
  const float* zeros_f;   // real-valued zero-points (App. K) or nullptr; replaces `zeros`
  const float* scales;
  __nv_bfloat16* out;     // [T, R]
  int N, K, G, g, g_shift, T;
  int R;                  // output features
  int r_tiles, tiles;     // row tiles, row tiles * token tiles (of the whole call)
  int tile0, tile1;       // tiles of this launch, see launch_split
  int first, t_first;     // tile its first cluster begins with, its first token tile
  int k_blocks;
  int nt;                 // tokens per tile, a multiple of 16
  int stages;
  int region;             // bytes of the stage buffers, which the partial sums take over
  int acc2, a_col;        // tensor-memory columns of the second accumulator and of the weights (forward)
  int q, cshift;          // tiles per cluster, log2 of the CTAs per cluster (q <= 1 << cshift)
  const __nv_bfloat16* dY;   // DS: [T, N]
  float* ds_part;            // DS: [token tiles * passes][N]
  Side side;                 // see common.cuh
  int* status;
};

__device__ __forceinline__ int split_group_of(const SplitParams& p, int col) {
  if (p.G == 1) return 0;
  return p.g_shift >= 0 ? (col >> p.g_shift) : (col / p.g);
}

// (Without a memory clobber: it stays behind the cluster's barrier as one volatile statement behind another,
// and the outputs of one turn of a loop need not be stored before the sums of the next are read.)
__device__ __forceinline__ float4 ld_cluster_f4(uint32_t cluster_addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(cluster_addr));
  return v;
}

// Zero-point (its bits, if real-valued) and scale of one 32-column unit.  Nothing is made of them where they are loaded, a turn
// ahead of their use: an operation on one would wait for it.
struct UnitZS {
  uint32_t z;
  float s;
};

template <bool ZF>
__device__ __forceinline__ UnitZS split_load_zs(const SplitParams& p, int i, int col) {
  UnitZS u;
  u.z = 0u;
  u.s = 0.0f;       // outside the matrix: code 0, zero-point 0, scale 0
  if (i < p.N && col < p.K) {
    const size_t gi = (size_t)i * p.G + split_group_of(p, col);
    u.s = ld_global(p.scales + gi);
    u.z = ZF ? __float_as_uint(ld_global(p.zeros_f + gi)) : ld_global(p.zeros + gi);
  }
  return u;
}

// DS (forward with one scale per channel): where the fp32 sums of a tile are complete they are also
// multiplied by dY and summed over the tile's tokens, dS[i] = sum_t dY[t,i] * u[t,i] (see the
// pair kernel).
template <int BITS, bool TRANS, bool FOLD, bool ZF, bool DS>
__global__ void __launch_bounds__(kSplitThreads, 1)
qsplit_kernel(const __grid_constant__ CUtensorMap tmap_act, const __grid_constant__ CUtensorMap tmap_pk,
              const SplitParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  constexpr int kWBytes = TRANS ? SM_A_BYTES : 0;               // forward: the weights are in tensor memory
  const int half_bytes = kWBytes + p.nt * (SM_HALF * 2);        // weights, then activations
  const int stage_bytes = 2 * half_bytes;
  uint8_t* sm_pk = base + p.region;
  SplitBarriers* bars = reinterpret_cast<SplitBarriers*>(sm_pk + SM_PK_SLOTS * SM_PK_BYTES);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  volatile int* abort_flag = &bars->abort_flag;

  // ---- this CTA's stages: [lo, hi) of the cluster's list, its first tile's, then the next tile's.  The
  // list is cut as in the whole call; a part of a call leaves out the stages of tiles that are not its own.
  const int csize = 1 << p.cshift;
  const int rank = (int)(blockIdx.x & (csize - 1));
  const int first_tile = p.first + (int)(blockIdx.x >> p.cshift) * p.q;
  const int L = min(p.q, p.tiles - first_tile) * p.k_blocks;
  auto range_lo = [&](int r) { return (r * L) >> p.cshift; };
  const int j_lo = max(0, p.tile0 - first_tile), j_hi = min(p.q, p.tile1 - first_tile);   // its own tiles
  const int lo = min(max(range_lo(rank), j_lo * p.k_blocks), j_hi * p.k_blocks);
  const int hi = min(max(range_lo(rank + 1), lo), j_hi * p.k_blocks);
  const int n_it = hi - lo;
  const int j0 = lo / p.k_blocks;                            // first tile of the range
  const int split_at = (j0 + 1) * p.k_blocks - lo;           // local stages of the first tile
  const int kb0 = lo - j0 * p.k_blocks;
  // local stage -> k-block; row and token tile of the segment
  auto kb_of = [&](int it) { return it < split_at ? kb0 + it : it - split_at; };
  auto r0_of = [&](int it) { return ((first_tile + j0 + (it < split_at ? 0 : 1)) % p.r_tiles) * SM_ROWS; };
  auto t0_of = [&](int it) { return ((first_tile + j0 + (it < split_at ? 0 : 1)) / p.r_tiles - p.t_first) * p.nt; };

  const bool beside = TRANS && p.side == kBeside;     // (a forward is the first of its call)
  begin_beside(beside);
  // Forward: the first codes, scales and zero-points are asked for in L2 at once.  (Nothing is read: the preceding
  // kernel may still be writing them, and L2 is where it writes.)  us before / after: 256 x 256 at 64 tokens 5.8 / 5.4,
  // 4096 x 4096 at 77 12.55 / 12.3; dX gained nothing (13.0 / 13.2).
  if constexpr (!TRANS) {
    if (n_it > 0 && warp == 3 && lane < min(n_it, SM_PK_SLOTS)) {
      prefetch_tile_2d(&tmap_pk, kb_of(lane) * (4 * BITS), r0_of(lane));
    } else if (n_it > 0 && warp >= 4 && warp < 8) {
      const int i = r0_of(0) + (int)threadIdx.x - 128, col = kb_of(0) * SM_BK;
      if (i < p.N && col < p.K) {
        const size_t gi = (size_t)i * p.G + split_group_of(p, col);
        prefetch_l2(p.scales + gi);
        if (ZF) prefetch_l2(p.zeros_f + gi);
        else prefetch_l2(p.zeros + gi);
      }
    }
  }

  if (threadIdx.x == 0) {
#pragma unroll 1
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&bars->full[s]), 8 + 1);     // the warps of two dequant groups, the TMA lane
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
#pragma unroll 1
    for (int s = 0; s < SM_PK_SLOTS; ++s) {
      mbar_init(smem_u32(&bars->full_pk[s]), 1);
      mbar_init(smem_u32(&bars->empty_pk[s]), 8);
    }
    mbar_init(smem_u32(&bars->acc_full), 1);
    bars->abort_flag = 0;
    bars->wait_limit_us = p.status[4];
    fence_mbar_init();
    prefetch_tmap(&tmap_act);
    prefetch_tmap(&tmap_pk);
  }
  if (warp == 2) {
    tmem_alloc(smem_u32(&bars->tmem_base), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // Set-up is done.  Everything below touches memory that the preceding kernel may still be writing, unless this one was
  // launched beside it (common.cuh).
  if (!beside) asm volatile("griddepcontrol.wait;" ::: "memory");
  let_next_in(p.side == kFollowed);
  const uint32_t tmem_base = bars->tmem_base;

  if (warp == 0) {
    // ------------------------------------------------ activation TMA (one lane)
    if (const uint32_t lane = elect_lane(); lane == 0) {
      const int ta = t0_of(0), tb = t0_of(split_at);
      // self-test knob (peqa_selftest_configure): announce one byte more than will arrive, so
      // that the stage never fills and the bounded waits have to end the kernel
      const uint32_t starve = !TRANS && p.status[5] != 0 ? 1u : 0u;
      int s = 0;
      uint32_t ph = 1;
#pragma unroll 1
      for (int it = 0; it < n_it; ++it) {
        if (!mbar_wait(smem_u32(&bars->empty[s]), ph, abort_flag)) break;
        const uint32_t bar = smem_u32(&bars->full[s]);
        mbar_arrive_expect_tx(bar, p.nt * (SM_BK * 2) + starve);
        const uint32_t dst = smem_u32(base + s * stage_bytes + kWBytes);
        const int t0 = it < split_at ? ta : tb, col = kb_of(it) * SM_BK;
        tma_load_2d(dst, &tmap_act, bar, col, t0);
        tma_load_2d(dst + half_bytes, &tmap_act, bar, col + SM_HALF, t0);
        if (++s == p.stages) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 3) {
    // ------------------------------------------ packed-code TMA (one lane)
    // 128 rows x 128 columns of codes: the tile's rows and the stage's columns (forward), or the
    // stage's rows and the tile's columns (dX)
    if (const uint32_t lane = elect_lane(); lane == 0) {
      const int ra = r0_of(0), rb = r0_of(split_at);
#pragma unroll 1
      for (int it = 0; it < n_it; ++it) {
        const int s = it % SM_PK_SLOTS;
        if (!mbar_wait(smem_u32(&bars->empty_pk[s]), ((it / SM_PK_SLOTS) & 1u) ^ 1u, abort_flag)) break;
        const uint32_t bar = smem_u32(&bars->full_pk[s]);
        const int kb = kb_of(it), r0 = it < split_at ? ra : rb;
        mbar_arrive_expect_tx(bar, 128 * 16 * BITS);
        const uint32_t dst = smem_u32(sm_pk + s * SM_PK_BYTES);
        if (!TRANS) tma_load_2d(dst, &tmap_pk, bar, kb * (4 * BITS), r0);
        else tma_load_2d(dst, &tmap_pk, bar, (r0 >> 5) * BITS, kb * SM_BK);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------- MMA issuer (one lane)
    if (const uint32_t lane = elect_lane(); lane == 0) {
      const uint32_t idesc = idesc_bf16_f32(SM_ROWS, 16, TRANS ? 1 : 0, 0) +
                             ((uint32_t)((p.nt - 16) >> 3) << 17);
      // Descriptors are advanced by additions (the address field counts 16-byte units).
      const uint32_t a0 = smem_u32(base);
      const uint64_t adesc0 = smem_desc_sw128(a0, TRANS ? 64 * 128 : 16, 1024);
      const uint64_t bdesc0 = smem_desc_sw128(a0 + kWBytes, 16, 1024);
      const uint64_t stage_inc = (uint64_t)(stage_bytes >> 4), half_inc = (uint64_t)(half_bytes >> 4);
      const uint32_t full0 = smem_u32(&bars->full[0]), empty0 = smem_u32(&bars->empty[0]);
      uint64_t adesc = adesc0, bdesc = bdesc0;
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
#pragma unroll 1
      for (int it = 0; it < n_it; ++it) {
        if (!mbar_wait(full0 + s * 8, ph, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d = tmem_base + (it < split_at ? 0u : (uint32_t)p.acc2);
        const bool fresh = it == 0 || it == split_at;
        if constexpr (TRANS) {
#pragma unroll
          for (int k = 0; k < SM_HALF / 16; ++k)
            mma_bf16_ss(d, adesc + k * (16 * 128 / 16), bdesc + k * (32 / 16), idesc, (fresh && k == 0) ? 0u : 1u);
#pragma unroll
          for (int k = 0; k < SM_HALF / 16; ++k)
            mma_bf16_ss(d, adesc + half_inc + k * (16 * 128 / 16), bdesc + half_inc + k * (32 / 16), idesc, 1u);
        } else {
          const uint32_t a = tmem_base + (uint32_t)(p.a_col + s * (SM_BK / 2));
#pragma unroll
          for (int k = 0; k < SM_HALF / 16; ++k)
            mma_bf16_ts(d, a + k * 8, bdesc + k * (32 / 16), idesc, (fresh && k == 0) ? 0u : 1u);
#pragma unroll
          for (int k = 0; k < SM_HALF / 16; ++k)
            mma_bf16_ts(d, a + SM_HALF / 2 + k * 8, bdesc + half_inc + k * (32 / 16), idesc, 1u);
        }
        mma_commit(empty0 + s * 8);
        adesc += stage_inc;
        bdesc += stage_inc;
        if (++s == p.stages) {
          s = 0;
          ph ^= 1u;
          adesc = adesc0;
          bdesc = bdesc0;
        }
      }
      if (ok) mma_commit(smem_u32(&bars->acc_full));
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------- weight dequant
    // A group takes every fourth half stage.  Forward: a thread is one weight row and both 32-column
    // units of the half.  dX: lanes are 8 rows x 4 units; the thread's second unit is 32 rows
    // further down.
    const int grp = (warp - 4) >> 2;
    const int half = grp & 1;
    const int gw = (warp - 4) & 3;
    const int u4 = lane >> 3;
    const int rowl = TRANS ? gw * 8 + (lane & 7) : gw * 32 + lane;
    const int swz = rowl & 7;                          // rows of a thread agree modulo 8
    const int ra = r0_of(0), rb = r0_of(split_at);
    // (forward) the second unit shares the first one's group unless groups are not multiples of 64 columns
    const bool one_group = !TRANS && (p.G == 1 || (p.g & 63) == 0);
    auto load_zs = [&](int it, UnitZS (&u)[2]) {
      if (it >= n_it) { u[0] = UnitZS{0u, 0.f}; u[1] = u[0]; return; }
      const int c0 = kb_of(it) * SM_BK + half * SM_HALF, r0 = it < split_at ? ra : rb;
      if (TRANS) {
        u[0] = split_load_zs<ZF>(p, c0 + rowl, r0 + 32 * u4);
        u[1] = split_load_zs<ZF>(p, c0 + rowl + 32, r0 + 32 * u4);
      } else {
        u[0] = split_load_zs<ZF>(p, r0 + rowl, c0);
        if (!one_group) u[1] = split_load_zs<ZF>(p, r0 + rowl, c0 + 32);
      }
    };
    auto turn = [&](int it, const UnitZS (&cur)[2], UnitZS (&next)[2]) -> bool {
      load_zs(it + 2, next);
      const int pq = it % SM_PK_SLOTS;
      if (!warp_wait(smem_u32(&bars->full_pk[pq]), (it / SM_PK_SLOTS) & 1u, abort_flag)) return false;
      const uint8_t* src = sm_pk + pq * SM_PK_BYTES;
      uint32_t w[2][BITS];
      if constexpr (!TRANS) {
        if constexpr (BITS == 4) {
          // 64-byte rows, 16-byte chunk c of row r at c ^ ((r >> 1) & 3): the code map's swizzle
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const uint4 v = *reinterpret_cast<const uint4*>(src + rowl * 64 + (((2 * half + k) ^ ((rowl >> 1) & 3)) << 4));
            w[k][0] = v.x; w[k][1] = v.y; w[k][2] = v.z; w[k][3] = v.w;
          }
        } else {
          // 48-byte rows, read whole (consecutive rows fall into different banks)
          const uint4 a = *reinterpret_cast<const uint4*>(src + rowl * 48 + 16 * half);
          const uint4 b = *reinterpret_cast<const uint4*>(src + rowl * 48 + 16 * half + 16);
          const uint32_t w8[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            w[0][e] = half ? w8[2 + e] : w8[e];
            w[1][e] = half ? w8[5 + e] : w8[3 + e];
          }
        }
      } else {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const uint8_t* at = src + (half * SM_HALF + rowl + 32 * k) * (16 * BITS) + u4 * (4 * BITS);
          if constexpr (BITS == 4) {
            const uint4 v = *reinterpret_cast<const uint4*>(at);
            w[k][0] = v.x; w[k][1] = v.y; w[k][2] = v.z; w[k][3] = v.w;
          } else {
#pragma unroll
            for (int e = 0; e < BITS; ++e) w[k][e] = reinterpret_cast<const uint32_t*>(at)[e];
          }
        }
      }
      uint32_t o[2][16];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const uint32_t z = one_group ? cur[0].z : cur[k].z;
        const float sc = one_group ? cur[0].s : cur[k].s;
        if constexpr (ZF) dq::unit32_affine<BITS>(w[k], z, sc, o[k]);
        else dq::unit32_natural<BITS, FOLD>(w[k], z, sc, o[k]);
      }
      const int s = it % p.stages;
      if (!warp_wait(smem_u32(&bars->empty[s]), ((it / p.stages) & 1u) ^ 1u, abort_flag)) return false;
      if constexpr (TRANS) {
        uint8_t* tile = base + s * stage_bytes + half * half_bytes;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          uint8_t* row_ptr = tile + (u4 >> 1) * (64 * 128) + (rowl + 32 * k) * 128;
          const int chunk0 = (u4 & 1) * 4;
#pragma unroll
          for (int c = 0; c < 4; ++c)
            *reinterpret_cast<uint4*>(row_ptr + (((chunk0 + c) ^ swz) << 4)) =
                make_uint4(o[k][4 * c], o[k][4 * c + 1], o[k][4 * c + 2], o[k][4 * c + 3]);
        }
      } else {
        // the row's 64 elements of the half stage: 32 columns of its lane
        tc_fence_after();
        tmem_st_32x32(tmem_base + ((uint32_t)(gw * 32) << 16) + (uint32_t)(p.a_col + s * (SM_BK / 2) + half * (SM_HALF / 2)),
                      o[0], o[1]);
        tmem_st_wait();
        tc_fence_before();
      }
      fence_proxy_async_smem();       // the weights are written, the codes have been read
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(smem_u32(&bars->full[s]));
        mbar_arrive(smem_u32(&bars->empty_pk[pq]));
      }
      return true;
    };
    // Two turns per loop, so that the values fetched ahead stay in the registers they were loaded
    // into: a copy at the end of a turn would wait for the load.
    UnitZS za[2], zb[2];
    const int it0 = grp >> 1;
    load_zs(it0, za);
#pragma unroll 1
    for (int it = it0; it < n_it; it += 4) {
      if (!turn(it, za, zb)) break;
      if (it + 2 >= n_it || !turn(it + 2, zb, za)) break;
    }
  }

  // ------------------------------------------------- partial sums -> outputs
  // Passes of SM_DUMP_TOK tokens.  dump[seg][token][row], fp32, over the stage buffers (every MMA
  // that read them has completed: acc_full).
  const bool worker = warp >= 4;
  bool ok = n_it > 0;
  if (worker && ok) {
    ok = warp_wait(smem_u32(&bars->acc_full), 0, abort_flag);
    tc_fence_after();
  }
  __syncwarp();
  float* dump = reinterpret_cast<float*>(base);
  const int tok_pass = min(p.nt, SM_DUMP_TOK);
  const int seg_floats = tok_pass * SM_ROWS;
  const int wtid = (int)threadIdx.x - 128;                   // worker thread index
  const int rows_per = SM_ROWS / csize;                      // rows of a tile this CTA finishes
  const int vec_shift = 5 - p.cshift, vec_per = 1 << vec_shift;
  const uint32_t dump_addr = smem_u32(dump);
#pragma unroll 1
  for (int tp = 0; tp < p.nt; tp += SM_DUMP_TOK) {
    if (worker && ok) {
      const int quarter = warp & 3;
      const int col = ((warp - 4) >> 2) * 32;                // tokens of the pass this warp copies
      if (tp + col < p.nt) {
#pragma unroll 1
        for (int seg = 0; seg < 2; ++seg) {
          if (seg == 1 && n_it <= split_at) break;
          uint32_t v[32];
          tmem_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + seg * p.acc2 + tp + col, v);
          tmem_ld_wait();
          float* d = dump + seg * seg_floats + col * SM_ROWS + quarter * 32 + lane;
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if (tp + col + e < p.nt) d[e * SM_ROWS] = __uint_as_float(v[e]);
        }
      }
    }
    __syncwarp();
    cluster_sync_shared();
    if (worker) {
      const int toks = min(tok_pass, p.nt - tp);
#pragma unroll 1
      for (int j = j_lo; j < j_hi; ++j) {
        const int tile = first_tile + j;
        const int r0 = (tile % p.r_tiles) * SM_ROWS + rank * rows_per;
        const int t0 = (tile / p.r_tiles - p.t_first) * p.nt + tp;
        // contributors: the CTAs whose ranges meet [j * k_blocks, (j + 1) * k_blocks)
        const int b0 = j * p.k_blocks, b1 = b0 + p.k_blocks;
        uint32_t from = 0, second = 0;     // contributing ranks; those that hold it as second segment
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int rl = range_lo(r), rh = range_lo(r + 1);
          if (r < csize && rl < b1 && rh > b0 && rh > rl) from |= 1u << r;
          if (rl < b0 && j > j_lo) second |= 1u << r;
        }
        float4 ds = make_float4(0.f, 0.f, 0.f, 0.f);   // vec_per divides kSplitWorkers: a thread keeps its rows
        // One vector per thread and turn, the sums of four CTAs requested before the first is used.  (Two vectors a
        // turn were twice the code for a launch to fetch, us, one / two: forward 2672 x 1856 at 142 tokens 11.8 / 12.6, 1096 x
        // 768 at 32 5.7 / 6.0, 2.1 % over 180 forwards; dX 8192 x 8192 at 45 28.2 / 28.9.)
#pragma unroll 1
        for (int idx = wtid; idx < toks * vec_per; idx += kSplitWorkers) {
          const int t = idx >> vec_shift, rv = (idx & (vec_per - 1)) * 4;
          const int row = r0 + rv;
          if (t0 + t >= p.T || row >= p.R) continue;
          const uint32_t off = dump_addr + (uint32_t)(t * SM_ROWS + rank * rows_per + rv) * 4u;
          uint2 y = make_uint2(0u, 0u);
          if (DS) y = ld_global(reinterpret_cast<const uint2*>(p.dY + (size_t)(t0 + t) * p.R + row));
          float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int rh = 0; rh < 8; rh += 4) {
            if (rh >= csize) break;
            float4 v[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              v[r] = make_float4(0.f, 0.f, 0.f, 0.f);
              if (from >> (rh + r) & 1u)
                v[r] = ld_cluster_f4(mapa_shared(off + (second >> (rh + r) & 1u ? (uint32_t)seg_floats * 4u : 0u), (uint32_t)(rh + r)));
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              a.x += v[r].x; a.y += v[r].y; a.z += v[r].z; a.w += v[r].w;
            }
          }
          if (DS) {
            ds.x = fmaf(a.x, __uint_as_float(y.x << 16), ds.x);
            ds.y = fmaf(a.y, __uint_as_float(y.x & 0xFFFF0000u), ds.y);
            ds.z = fmaf(a.z, __uint_as_float(y.y << 16), ds.z);
            ds.w = fmaf(a.w, __uint_as_float(y.y & 0xFFFF0000u), ds.w);
          }
          if (!FOLD) {
            const float4 sc = ld_global(reinterpret_cast<const float4*>(p.scales + row));   // one scale per channel
            a.x *= sc.x; a.y *= sc.y; a.z *= sc.z; a.w *= sc.w;
          }
          __nv_bfloat162 h0 = __floats2bfloat162_rn(a.x, a.y), h1 = __floats2bfloat162_rn(a.z, a.w);
          uint2 o;
          o.x = *reinterpret_cast<uint32_t*>(&h0);
          o.y = *reinterpret_cast<uint32_t*>(&h1);
          *reinterpret_cast<uint2*>(p.out + (size_t)(t0 + t) * p.R + row) = o;
        }
        if (DS) {
          // lanes that share rows, then the warps in order (over the code slots, which are done with)
#pragma unroll 1
          for (int o = 16; o >= vec_per; o >>= 1) {
            ds.x += __shfl_xor_sync(0xffffffffu, ds.x, o);
            ds.y += __shfl_xor_sync(0xffffffffu, ds.y, o);
            ds.z += __shfl_xor_sync(0xffffffffu, ds.z, o);
            ds.w += __shfl_xor_sync(0xffffffffu, ds.w, o);
          }
          float4* sums = reinterpret_cast<float4*>(sm_pk);
          if (lane < vec_per) sums[(warp - 4) * 32 + lane] = ds;
          named_barrier_sync(1, kSplitWorkers);
          if (wtid < vec_per && r0 + wtid * 4 < p.R) {
            float4 s = sums[wtid];
#pragma unroll 1
            for (int w = 1; w < kSplitWorkers / 32; ++w) {
              const float4 v = sums[w * 32 + wtid];
              s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
            }
            const int passes = (p.nt + SM_DUMP_TOK - 1) / SM_DUMP_TOK;
            const size_t slot = (size_t)(tile / p.r_tiles) * passes + tp / SM_DUMP_TOK;
            *reinterpret_cast<float4*>(p.ds_part + slot * p.R + r0 + wtid * 4) = s;
          }
          named_barrier_sync(1, kSplitWorkers);
        }
      }
    }
    __syncwarp();
    cluster_sync_reads();   // the buffers are read by the whole cluster until here
  }

  if (*abort_flag)        // let copies and MMAs already in flight finish before memory is released
#pragma unroll 1
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  if (threadIdx.x == 0 && bars->abort_flag) {
    atomicExch(p.status, (int)PEQA_ERR_DEVICE_TIMEOUT);
    p.status[1] = (int)blockIdx.x;
  }
  // beside another kernel: this one has not ended before that one has
  if (beside && blockIdx.x == 0 && threadIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int BITS, bool TRANS, bool FOLD, bool ZF, bool DS = false>
int launch_split_t(const CUtensorMap& ta, const CUtensorMap& tp, const SplitParams& p, size_t smem,
                   cudaStream_t st) {
  auto kern = qsplit_kernel<BITS, TRANS, FOLD, ZF, DS>;
  static std::atomic<uint64_t> done{0};
  PEQA_TRY(allow_smem(kern, SM_SMEM_LIMIT, done));
  cudaLaunchConfig_t cfg = {};
  const int clusters = (p.tile1 - p.first + p.q - 1) / p.q;
  cfg.gridDim = dim3(clusters << p.cshift, 1, 1);
  cfg.blockDim = dim3(kSplitThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1 << p.cshift;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  PEQA_CUDA(cudaLaunchKernelEx(&cfg, kern, ta, tp, p));
  return PEQA_OK;
}

// Token tile, tiles per cluster and CTAs per cluster with the smallest estimated time.
//
// Measured on this part (4096 x 4096 and 4096 x 11008, 17 to 1024 tokens): a stage of 128
// contraction elements takes 0.60 us + 1.8 ns per token of the tile (the weights of a stage cost
// the same however many tokens multiply them; past 80 tokens the MMAs show), a wave of CTAs
// another 7 us (launch, first copies, the exchange of the sums).  Good enough to choose among cluster
// shapes; against the other kernels split_ns is held.
struct SplitPlan {
  int nt, t_tiles, q, cshift;
  int waves, stages;   // waves of clusters, stages of a CTA in each
  long long ns;
};
// Forward: stages of weights (64 columns each) that fit in tensor memory beside the accumulators.
int split_tmem_stages(int nt, int q) {
  const int s = (512 - (q > 1 ? 2 : 1) * ((nt + 31) & ~31)) / (SM_BK / 2);
  return s < SM_MAX_STAGES ? s : SM_MAX_STAGES;
}
// Forward: time of a plan in ns.  Fitted to 150 calls (17 to 4096 tokens, 256 to 22016 rows and columns; nine of
// ten within 0.89 to 1.13, since the exchange takes one vector per thread 0.94 to 1.14): 4.7 us a wave, 0.65 us + 0.28 ns per token a stage, and for the sums and their
// exchange 28 ns per token of the tile, 54 where a CTA may hold two tiles'.
long long split_fwd_ns(long long waves, long long stages, int nt, int q) {
  return waves * (4700 + stages * (649 + nt * 28 / 100) + nt * (q > 1 ? 54 : 28));
}
SplitPlan plan_split(int r_tiles, int C, int T, int sms, bool trans) {
  SplitPlan plans[2] = {};             // whole and halved token tiles
  plans[0].ns = plans[1].ns = -1;
  const long long k_blocks = (C + SM_BK - 1) / SM_BK;
  // clusters of 1, 2, 4, 8 CTAs that run at once (cudaOccupancyMaxActiveClusters on this part: 148,
  // 74, 33, 15 -- the larger ones leave SMs of a GPC idle)
  const int active[4] = {sms, sms / 2, sms * 33 / 148, sms * 15 / 148};
  const int t_min = (T + SM_MAX_NT - 1) / SM_MAX_NT;
  // Token tiles as wide as they can be, or half as wide: a forward whose CTAs hold two accumulators has no room
  // for its weights beside two wide ones, and where one round of CTAs leaves SMs idle the halves share the
  // exchange (us, whole / halved: 1480 x 384 at 183 tokens 10.6 / 7.0, 4216 x 1664 at 173 13.5 / 11.5).  Halves of 16 tokens gain
  // nothing (six calls, 0.96 to 1.24 of the time: 4728 x 512 at 18 6.1 / 7.5), and at less than 64 the estimate does not tell
  // 3 % (2136 x 1024 at 85 7.3 / 7.8).
  for (int halved = 0; halved < (trans ? 1 : 2); ++halved) {
    const int tt = t_min << halved;
    const int nt = ((T + tt - 1) / tt + 15) & ~15;
    if (halved && nt < 32) break;
    SplitPlan& best = plans[halved];
    const int t_tiles = (T + nt - 1) / nt;
    const long long tiles = (long long)r_tiles * t_tiles;
    for (int ci = 0; ci < 4; ++ci) {
      if (active[ci] < 1) continue;
      for (int q = 1; q <= (1 << ci); ++q) {
        if (!trans && split_tmem_stages(nt, q) < 3) continue;
        const long long clusters = (tiles + q - 1) / q;
        const long long waves = (clusters + active[ci] - 1) / active[ci];
        const long long stages = (q * k_blocks + (1 << ci) - 1) >> ci;
        const long long ns = trans ? waves * (stages * (600 + nt * 9 / 5) + 7000 + (ci ? 500 : 0) + 50 * ci)
                                   : split_fwd_ns(waves, stages, nt, q) + 50 * ci;
        if (best.ns < 0 || ns < best.ns) {
          best.t_tiles = t_tiles;
          best.nt = nt;
          best.q = q;
          best.cshift = ci;
          best.waves = (int)waves;
          best.stages = (int)stages;
          best.ns = ns;
        }
      }
    }
  }
  return plans[1].ns >= 0 && plans[1].ns * (plans[1].nt < 64 ? 103 : 100) < plans[0].ns * 100 ? plans[1] : plans[0];
}

// The pair kernels on the same call: rounds of 512 x 256 tiles over the pairs of SMs.  dX, fitted to 400
// random calls, launches back to back (256 to 22016 rows and columns, 17 to 2600 tokens): a stage of 64
// takes 0.58 us, with two blocks of tokens in the tile 0.67; a round 3.3 us more, with two blocks
// 4.3; the launch 3.2.  The forward, fitted to 150: 0.55 / 0.62 us, 1.85 / 3.45, 4.4 and 4.95 where its epilogue multiplies by
// the channels' scales.  Nine of ten estimates are 0.88 to 1.09 of what was measured.  The shorter last round of
// items of one block (make_pair_items) is left out: it saves a sixth of one round.
long long pair_ns(int R, int C, int T, bool trans, bool channel_scales, int sms) {
  const long long tiles = (long long)((R + 255) / 256) * ((T + 511) / 512);
  const int pairs = sms / 2 > 0 ? sms / 2 : 1;
  const long long rounds = (tiles + pairs - 1) / pairs, stages = (C + 63) / 64;
  if (trans) return rounds * (T > 256 ? 4300 + stages * 666 : 3300 + stages * 580) + 3200;
  return rounds * (T > 256 ? 3450 + stages * 618 : 1850 + stages * 550) + (channel_scales ? 4950 : 4400);
}

}  // namespace

// Estimated time of this kernel on a call of T tokens, in ns.  dX, fitted to the 400 calls: 3.6 us a wave,
// 0.72 us + 0.83 ns per token a stage, and 34 ns per token of the tile for the exchange of the sums, 43
// where no cluster shares it and 61 where a cluster owns several tiles.  Nine of ten estimates are 0.87
// to 1.11 of what was measured.
long long split_ns(const peqa_qweight_t* w, int T, bool trans) {
  const int R = trans ? w->in_features : w->out_features, C = trans ? w->out_features : w->in_features;
  const SplitPlan p = plan_split((R + SM_ROWS - 1) / SM_ROWS, C, T, sm_count_or(148), trans);
  if (!trans) return split_fwd_ns(p.waves, p.stages, p.nt, p.q);
  return (long long)p.waves * (3600 + p.stages * (720 + p.nt * 5 / 6) + p.nt * (34 + (p.cshift ? 0 : 9) + (p.q > 1 ? 27 : 0)));
}

// Whether a call is served faster by this kernel than by the pair kernels; 3 % in doubt go to those.  The estimates of both were fitted before MMAs
// were issued by an elected lane and weights published by a restricted release, which made both kernels a tenth faster.  Over
// 140 random calls (40 to 2600 tokens) the choice costs 0.3 % on average; it is a third off at worst, dX 7560 x 14848 in groups of 64 at 254
// tokens (us, pair / here 67 / 89).  Over 60 (17 to 300) the choice of cluster shapes costs 0.3 %.  Pair / here, in us, before that:
// 4096 x 11008 forward at 1001 tokens 116 / 77, its dX (86 row tiles: three waves) 90 / 124; 4096 x 4096
// forward at 77 tokens 42 / 12.5, at 2048 52 / 71; 22016 x 8192 at 256 tokens forward 174 / 109, dX 217 / 91;
// 2360 x 256 forward at 1134 tokens 10.0 / 13.0.
bool split_is_faster(const peqa_qweight_t* w, int T, bool trans, bool channel_scales) {
  const int R = trans ? w->in_features : w->out_features, C = trans ? w->out_features : w->in_features;
  return split_ns(w, T, trans) * 100 < pair_ns(R, C, T, trans, channel_scales, sm_count_or(148)) * 97;
}

// Partial sums per channel that a forward with dS writes.
int split_ds_slots(const peqa_qweight_t* w, int T) {
  const SplitPlan plan = plan_split((w->out_features + SM_ROWS - 1) / SM_ROWS, w->in_features, T, sm_count_or(148), false);
  return plan.t_tiles * ((plan.nt + SM_DUMP_TOK - 1) / SM_DUMP_TOK);
}

// A part of a call begins at a multiple of this: whole token tiles.
int split_part_tokens(const peqa_qweight_t* w, int T_call, bool trans) {
  const int r_tiles = ((trans ? w->in_features : w->out_features) + SM_ROWS - 1) / SM_ROWS;
  return plan_split(r_tiles, trans ? w->out_features : w->in_features, T_call, sm_count_or(148), trans).nt;
}

// The T tokens from t0 on of a call of T_call tokens (act, out: of the part).  Plan and cut are those of the
// whole call, so a token's sums are added in the same order in whichever part it comes.
int launch_split(const peqa_qweight_t* w, const float* zeros_f, int g, const void* act, int T, void* out,
                 bool trans, const void* dY, float* ds_part, cudaStream_t st, int T_call, int t0, Side side) {
  SplitParams p;
  p.side = side;
  p.zeros = w->zeros;
  p.zeros_f = zeros_f;
  p.scales = w->scales;
  p.out = static_cast<__nv_bfloat16*>(out);
  p.dY = static_cast<const __nv_bfloat16*>(dY);
  p.ds_part = ds_part;
  p.N = w->out_features;
  p.K = w->in_features;
  p.g = g;
  p.G = p.K / g;
  p.g_shift = -1;
  for (int b = 5; b < 31; ++b)
    if ((1 << b) == g) p.g_shift = b;
  p.T = T;
  p.R = trans ? p.K : p.N;
  const int C = trans ? p.N : p.K;
  p.r_tiles = (p.R + SM_ROWS - 1) / SM_ROWS;
  const SplitPlan plan = plan_split(p.r_tiles, C, T_call, sm_count_or(148), trans);
  p.nt = plan.nt;
  p.q = plan.q;
  p.cshift = plan.cshift;
  p.tiles = p.r_tiles * plan.t_tiles;
  p.tile0 = p.r_tiles * (t0 / plan.nt);
  p.tile1 = p.r_tiles * ((t0 + T + plan.nt - 1) / plan.nt);
  p.first = p.tile0 / p.q * p.q;
  p.t_first = t0 / plan.nt;
  p.k_blocks = (C + SM_BK - 1) / SM_BK;
  const int stage_bytes = 2 * ((trans ? SM_A_BYTES : 0) + p.nt * (SM_HALF * 2));
  p.stages = (SM_SMEM_LIMIT - SM_SMEM_FIXED) / stage_bytes;
  if (p.stages > SM_MAX_STAGES) p.stages = SM_MAX_STAGES;
  const int segs = p.q > 1 ? 2 : 1;          // partial sums a CTA may hold
  if (trans) {
    p.acc2 = SM_MAX_NT;
    p.a_col = 0;
  } else {
    p.acc2 = (p.nt + 31) & ~31;
    p.stages = p.stages < split_tmem_stages(p.nt, p.q) ? p.stages : split_tmem_stages(p.nt, p.q);
    p.a_col = 512 - p.stages * (SM_BK / 2);
  }
  const int dump = segs * (p.nt < SM_DUMP_TOK ? p.nt : SM_DUMP_TOK) * SM_ROWS * 4;
  p.region = p.stages * stage_bytes > dump ? p.stages * stage_bytes : dump;
  const size_t smem = (size_t)p.region + SM_SMEM_FIXED;
  PEQA_TRY(status_word(st, &p.status));
  EncodeTiledFn enc = nullptr;
  PEQA_TRY(tensor_map_encoder(&enc));
  CUtensorMap ta, tp;
  {
    cuuint64_t dims[2] = {(cuuint64_t)C, (cuuint64_t)T};
    cuuint64_t strides[1] = {(cuuint64_t)C * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)p.nt};
    cuuint32_t estr[2] = {1, 1};
    if (enc(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(act), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cuda_fail(cudaErrorInvalidValue);
  }
  {
    const int wpr = p.K * w->bits / 32;
    cuuint64_t dims[2] = {(cuuint64_t)wpr, (cuuint64_t)p.N};
    cuuint64_t strides[1] = {(cuuint64_t)wpr * 4};
    cuuint32_t box[2] = {(cuuint32_t)(4 * w->bits), 128u};
    cuuint32_t estr[2] = {1, 1};
    if (enc(&tp, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<uint32_t*>(w->qweight), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            !trans && w->bits == 4 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cuda_fail(cudaErrorInvalidValue);
  }
  const bool b4 = w->bits == 4;
  if (trans) {
    if (zeros_f) return b4 ? launch_split_t<4, true, true, true>(ta, tp, p, smem, st)
                           : launch_split_t<3, true, true, true>(ta, tp, p, smem, st);
    return b4 ? launch_split_t<4, true, true, false>(ta, tp, p, smem, st)
              : launch_split_t<3, true, true, false>(ta, tp, p, smem, st);
  }
  if (zeros_f) return b4 ? launch_split_t<4, false, true, true>(ta, tp, p, smem, st)
                         : launch_split_t<3, false, true, true>(ta, tp, p, smem, st);
  if (p.G > 1) return b4 ? launch_split_t<4, false, true, false>(ta, tp, p, smem, st)
                         : launch_split_t<3, false, true, false>(ta, tp, p, smem, st);
  if (ds_part) return b4 ? launch_split_t<4, false, false, false, true>(ta, tp, p, smem, st)
                         : launch_split_t<3, false, false, false, true>(ta, tp, p, smem, st);
  return b4 ? launch_split_t<4, false, false, false>(ta, tp, p, smem, st)
            : launch_split_t<3, false, false, false>(ta, tp, p, smem, st);
}

}  // namespace peqa
