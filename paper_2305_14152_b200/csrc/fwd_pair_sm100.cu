// Forward of the PEQA layer, Y = X * W_hat^T (Eq. 2), on CTA pairs.
//
// A pair of CTAs (cta_group::2) owns a tile of 512 tokens x 256 output channels,
// held as two 256 x 256 accumulators that fill tensor memory.  The tokens are
// the MMA "M" side: CTA `rank` TMA-loads two blocks of 128 tokens of X per
// 64-deep stage (A operands, K-major).  The weights are the "N" side, split
// between the two CTAs: each rebuilds (Q - z) [* bf16(s)] of its 128 channels
// [n0 + 128*rank, +128) as bf16 in its own shared memory, K-major with the
// 128-byte swizzle the tensor core expects, and both token blocks multiply the
// same weight stage.  A weight element is therefore rebuilt once per 512
// tokens, which brings the conversion work per stage (8192 elements per CTA)
// under the time the tensor cores need for it (two 256x256x64 products), and
// the accumulator is token-major, so an epilogue thread writes contiguous runs
// of Y.
//
// Packed codes reach the dequant warps through their own TMA ring (one box =
// 128 channels x 64 columns of codes).  Four groups of four dequant warps take
// the stages round-robin, so that one group's wait -> read -> convert -> store
// -> signal chain overlaps the others'.  A tile whose second token block lies
// wholly beyond T runs with one block.
//
// With one scale per channel (G == 1) the weights stay the exact integers
// Q - z and the fp32 scale multiplies the accumulator columns in the epilogue;
// with grouped scales the product (Q - z) * bf16(s) is formed before the MMA.
#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "dequant.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"

namespace peqa {

namespace {

using namespace ptx;

constexpr int PK = 64;                       // contraction elements per stage
constexpr int PSTAGES = 4;
constexpr int PBLK_BYTES = 128 * PK * 2;     // one block of 128 tokens of X: 16 KiB
constexpr int PA_BYTES = 2 * PBLK_BYTES;     // this CTA's two token blocks
constexpr int PB_BYTES = 128 * PK * 2;       // this CTA's 128 channels: 16 KiB
constexpr int PSTAGE_BYTES = PA_BYTES + PB_BYTES;
constexpr int PQ_SLOTS = 4;
constexpr int PE_BYTES = 32 * 64;            // one epilogue warp's staging tile: 32 tokens x 32 channels
constexpr int PQ_BYTES = 128 * 32;           // packed codes of one stage: 128 rows x 8 words
constexpr int P_TMEM_COLS = 512;
constexpr int P_SMEM_BYTES = PSTAGES * PSTAGE_BYTES + PQ_SLOTS * PQ_BYTES + 8 * PE_BYTES + 1024 + 512;
constexpr int P_GROUPS = 4;        // dequant groups (four warps each)
constexpr int kPairThreads = 896;  // warps: 0 act TMA, 1 MMA, 2 TMEM alloc, 3 code TMA, 4-11 epilogue, 12-27 dequant

struct PairBarriers {
  uint64_t full[PSTAGES];       // leader: both CTAs' X landed and weights written
  uint64_t empty[PSTAGES];      // each CTA: MMAs that read the stage completed
  uint64_t pk_full[PQ_SLOTS];   // each CTA: packed codes landed
  uint64_t pk_empty[PQ_SLOTS];  // each CTA: the group that owns the slot has read it
  uint64_t acc_full;            // each CTA: both accumulators ready
  uint64_t acc_empty;           // leader: both CTAs' epilogues drained them
  uint64_t ds_full, ds_free;    // each CTA (DS): the epilogue warps' sums of a tile lie ready / have been read
  uint32_t tmem_base;
  int abort_flag;
  int wait_limit_us;    // must follow abort_flag (read by the bounded waits)
};

struct PairParams {
  const uint8_t* zeros;
  const float* zeros_f;   // real-valued zero-points (App. K) or nullptr; replaces `zeros`
  const float* scales;
  __nv_bfloat16* out;   // Y [T, N]
  int N, K, G, g, g_shift, T;
  int n_tiles, t_tiles, k_blocks;   // 256-channel tiles, 512-token tiles, 64-deep stages
  PairItems items;
  Side side;            // see common.cuh
  const __nv_bfloat16* dY;   // DS: [T, N]
  float* ds_part;            // DS: [2 * ceil(T / 256)][N]
  int* status;
};

__device__ __forceinline__ int pair_group_of(const PairParams& p, int col) {
  if (p.G == 1) return 0;
  return p.g_shift >= 0 ? (col >> p.g_shift) : (col / p.g);
}

// DS (one scale per channel): the epilogue also takes the scale gradient's sums.  Eq. 2 reads
// Y[t,i] = s[i] * u[t,i] with u = sum_j X (Q - z), so dS[i] = sum_t dY[t,i] * u[t,i], and u is
// what the accumulator holds, in fp32: a product per output replaces the third contraction
// (2 T N K flop).  A warp multiplies its 32 tokens x 32 channels by dY and folds them over its
// lanes; the four warps of a token block are added through their staging tiles in warp order and
// stored to ds_part; ds_channel_kernel adds the blocks.
template <int BITS, bool FOLD, bool ZF, bool DS>
__global__ void __launch_bounds__(kPairThreads, 1)
qfwd_pair_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_q,
                 const __grid_constant__ CUtensorMap tmap_y, const PairParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sm_q = base + PSTAGES * PSTAGE_BYTES;          // PQ_SLOTS x 4 KiB, plain 32-byte rows
  uint8_t* sm_e = sm_q + PQ_SLOTS * PQ_BYTES;             // 8 epilogue warps x 2 KiB, 64-byte swizzle
  PairBarriers* bars = reinterpret_cast<PairBarriers*>(sm_e + 8 * PE_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  volatile int* abort_flag = &bars->abort_flag;

  if (threadIdx.x == 0) {
    for (int s = 0; s < PSTAGES; ++s) {
      mbar_init(smem_u32(&bars->full[s]), 1 + 8);         // the X copies, 4 warps of one group in each CTA
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
    for (int q = 0; q < PQ_SLOTS; ++q) {
      mbar_init(smem_u32(&bars->pk_full[q]), 1);
      mbar_init(smem_u32(&bars->pk_empty[q]), 4);         // 4 warps of the owning group
    }
    mbar_init(smem_u32(&bars->acc_full), 1);
    mbar_init(smem_u32(&bars->acc_empty), 16);            // 8 epilogue warps in each CTA
    mbar_init(smem_u32(&bars->ds_full), 8);
    mbar_init(smem_u32(&bars->ds_free), 8);
    bars->abort_flag = 0;
    bars->wait_limit_us = p.status[4];
    fence_mbar_init();
    prefetch_tmap(&tmap_x);
    prefetch_tmap(&tmap_q);
    prefetch_tmap(&tmap_y);
  }
  if (warp == 2) {
    tmem_alloc_pair(smem_u32(&bars->tmem_base), P_TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  tc_fence_after();
  // Set-up is done.  Everything below touches memory that the preceding kernel may still be writing.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  let_next_in(p.side == kFollowed);
  const uint32_t tmem_base = bars->tmem_base;
  const int total_tiles = p.items.total_items;      // work items: whole tiles, then halves
  const int pair = blockIdx.x >> 1;
  const int n_pairs = gridDim.x >> 1;
  const int my_tiles = (total_tiles - pair + n_pairs - 1) / n_pairs;

  if (warp == 0) {
    // ------------------------------------------ activation TMA (one lane)
    if (const uint32_t lane = elect_lane(); lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      // self-test knob (peqa_selftest_configure): announce one byte more than will arrive, so
      // that the stage never fills and the bounded waits have to end the kernel
      const uint32_t starve = p.status[5] != 0 ? 1u : 0u;
      for (int tile = pair; ok && tile < total_tiles; tile += n_pairs) {
        int n_tile, tt0, blocks;
        pair_item(p.items, tile, p.T, n_tile, tt0, blocks);
        const int t0 = tt0 + (int)rank * 128;
        for (int kb = 0; kb < p.k_blocks; ++kb, ++it) {
          const int s = it % PSTAGES;
          const uint32_t ph = (it / PSTAGES) & 1u;
          if (!mbar_wait_cluster(smem_u32(&bars->empty[s]), ph ^ 1u, abort_flag)) { ok = false; break; }
          if (leader) mbar_arrive_expect_tx(smem_u32(&bars->full[s]), 2 * blocks * PBLK_BYTES + starve);
          const uint32_t bar = mapa_shared(smem_u32(&bars->full[s]), 0);
          tma_load_2d_pair(smem_u32(base + s * PSTAGE_BYTES), &tmap_x, bar, kb * PK, t0);
          if (blocks == 2)
            tma_load_2d_pair(smem_u32(base + s * PSTAGE_BYTES + PBLK_BYTES), &tmap_x, bar, kb * PK, t0 + 256);
        }
      }
    }
  } else if (warp == 3) {
    // ------------------------------------------ packed-code TMA (one lane)
    // A box is 128 rows x 8 words holding the stage's 64 columns; for 3-bit codes the 6
    // words start 2 words into the box on odd k-blocks, which keeps the box start
    // 16-byte aligned.
    if (const uint32_t lane = elect_lane(); lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int tile = pair; ok && tile < total_tiles; tile += n_pairs) {
        int n_tile, tt0, blocks;
        pair_item(p.items, tile, p.T, n_tile, tt0, blocks);
        const int r0 = n_tile * 256 + (int)rank * 128;
        for (int kb = 0; kb < p.k_blocks; ++kb, ++it) {
          const int q = it % PQ_SLOTS;
          const uint32_t ph = (it / PQ_SLOTS) & 1u;
          if (!mbar_wait(smem_u32(&bars->pk_empty[q]), ph ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t bar = smem_u32(&bars->pk_full[q]);
          mbar_arrive_expect_tx(bar, PQ_BYTES);
          tma_load_2d(smem_u32(sm_q + q * PQ_BYTES), &tmap_q, bar,
                      BITS == 3 ? 6 * kb - 2 * (kb & 1) : 8 * kb, r0);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------ MMA issuer (leader CTA, one lane)
    if (leader) if (const uint32_t lane = elect_lane(); lane == 0) {
      // One thread issues everything, the MMAs of a stage in a few cycles each (see elect_lane), so the tensor pipe has work
      // while this thread waits for the next stage.  Weights and activations share a barrier, and descriptors are advanced
      // by additions (the address field counts 16-byte units).
      constexpr uint32_t idesc = idesc_bf16_f32(256, 256, 0, 0);
      const uint32_t a0 = smem_u32(base);
      const uint64_t adesc0 = smem_desc_sw128(a0, 16, 1024);
      const uint64_t bdesc0 = smem_desc_sw128(a0 + PA_BYTES, 16, 1024);
      const uint32_t full0 = smem_u32(&bars->full[0]), empty0 = smem_u32(&bars->empty[0]);
      uint32_t s = 0, ph = 0;
      int local = 0;
      bool ok = true;
      for (int tile = pair; ok && tile < total_tiles; tile += n_pairs, ++local) {
        int n_tile, tt0, blocks;
        pair_item(p.items, tile, p.T, n_tile, tt0, blocks);
        if (!mbar_wait_cluster(smem_u32(&bars->acc_empty), (uint32_t)(local & 1) ^ 1u, abort_flag)) { ok = false; break; }
        tc_fence_after();
        for (int kb = 0; kb < p.k_blocks; ++kb) {
          if (!mbar_wait_cluster(full0 + s * 8, ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint64_t adesc = adesc0 + s * (PSTAGE_BYTES >> 4), bdesc = bdesc0 + s * (PSTAGE_BYTES >> 4);
          const uint32_t at = s;
          if (++s == PSTAGES) {
            s = 0;
            ph ^= 1u;
          }
          if (blocks == 2) {
#pragma unroll
            for (int k = 0; k < PK / 16; ++k)
              mma_bf16_ss_pair(tmem_base, adesc + k * (32 / 16), bdesc + k * (32 / 16), idesc, (kb | k) != 0 ? 1u : 0u);
          }
          const uint64_t alast = blocks == 2 ? adesc + (PBLK_BYTES >> 4) : adesc;
          const uint32_t dlast = blocks == 2 ? tmem_base + 256 : tmem_base;
#pragma unroll
          for (int k = 0; k < PK / 16; ++k)
            mma_bf16_ss_pair(dlast, alast + k * (32 / 16), bdesc + k * (32 / 16), idesc, (kb | k) != 0 ? 1u : 0u);
          mma_commit_pair(empty0 + at * 8, 3);
        }
        if (ok) mma_commit_pair(smem_u32(&bars->acc_full), 3);
      }
    }
  } else if (warp >= 4 && warp < 12) {
    // ------------------------------------------ epilogue: thread = token, 256 channels
    // A warp drains 32 tokens x 32 channels at a time: tensor memory -> registers -> bf16 ->
    // its 2 KiB staging tile (rows of 64 bytes, 16-byte chunk c of row r at c ^ ((r >> 1) & 3):
    // the 64-byte swizzle of the output tensor map, which also keeps the stores free of bank
    // conflicts) -> one tiled bulk store.  The copy engine writes whole sectors of Y; a
    // thread-per-row store by the warp itself cost 32 half-filled sectors per instruction and
    // made the drain take ~11,000 cycles a tile.  The accumulators are released as soon as the
    // last chunk has left tensor memory.
    const int quarter = warp & 3;
    const int m = (warp - 4) >> 2;                 // token block = accumulator
    const uint32_t acc_empty_leader = mapa_shared(smem_u32(&bars->acc_empty), 0);
    uint8_t* stage = sm_e + (warp - 4) * PE_BYTES;
    uint8_t* srow = stage + lane * 64;
    const int sw = (lane >> 1) & 3;
    int local = 0;
    bool ok = true;
    for (int tile = pair; ok && tile < total_tiles; tile += n_pairs, ++local) {
      int n_tile, tt0, blocks;
      pair_item(p.items, tile, p.T, n_tile, tt0, blocks);
      const int n0 = n_tile * 256;
      const int row0 = tt0 + m * 256 + (int)rank * 128 + quarter * 32;   // first token of this warp
      const __nv_bfloat16* dy_row = p.dY + (size_t)(row0 + lane) * p.N + n0;
      float ds_sum[8];
      if (DS) {
#pragma unroll
        for (int k = 0; k < 8; ++k) ds_sum[k] = 0.0f;
        // this token's 256 channels of dY on their way into L2 while the accumulators fill
        if (m < blocks && row0 + lane < p.T)
          for (int c = 0; c < 256 && n0 + c < p.N; c += 64)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(dy_row + c));
      }
      // Scales and dY are asked for ahead: a lane holds the scale of one channel of the chunk and hands it
      // round, and the dY of its token's next 16 channels.  Loaded where they were used (32 scales, one
      // after the other, by every lane) a chunk took 7000 cycles, 3500 for the scales and 2600 for dY.
      // With dY (DS) a chunk is worked through in two halves of 16 channels, which leaves registers for that.
      constexpr int W = DS ? 16 : 32;              // channels at a time
      auto chunk_scale = [&](int c) { return !FOLD && c + lane < p.N ? ld_global(p.scales + c + lane) : 0.0f; };
      uint4 dy[2];
      auto load_dy = [&](int c) {                  // tokens and channels beyond the matrix count zero
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          dy[q] = make_uint4(0u, 0u, 0u, 0u);
          if (m < blocks && row0 + lane < p.T && n0 + c + 8 * q < p.N) dy[q] = ld_global(reinterpret_cast<const uint4*>(dy_row + c + 8 * q));
        }
      };
      float next_scale = chunk_scale(n0);
      if (DS) load_dy(0);
      if (!warp_wait_cluster(smem_u32(&bars->acc_full), (uint32_t)(local & 1), abort_flag)) { ok = false; break; }
      tc_fence_after();
      int chunks = m < blocks ? (p.N - n0 + 31) / 32 : 0;
      chunks = chunks > 8 ? 8 : chunks;
      // the sums of the last tile must have been read before the staging tiles are written again
      if (DS && local > 0 && !warp_wait(smem_u32(&bars->ds_free), (uint32_t)(local - 1) & 1u, abort_flag)) { ok = false; break; }
#pragma unroll 1
      for (int cc = 0; cc < chunks; ++cc) {
        const int c0 = n0 + cc * 32;
        const float scale = next_scale;
        if (!FOLD && cc + 1 < chunks) next_scale = chunk_scale(c0 + 32);
        float half_sum[2] = {0.0f, 0.0f};
#pragma unroll
        for (int h = 0; h < 32 / W; ++h) {
          uint32_t v[W];
          const uint32_t at = tmem_base + ((uint32_t)(quarter * 32) << 16) + m * 256 + cc * 32 + h * W;
          if constexpr (DS) tmem_ld_32x16(at, v);
          else tmem_ld_32x32(at, v);
          tmem_ld_wait();
          if (cc + 1 == chunks && h + 1 == 32 / W) {
            // nothing of this tile is left in tensor memory for this warp
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(acc_empty_leader);
          }
          auto scaled = [&](int j) {
            const float u = __uint_as_float(v[j]);
            return FOLD ? u : u * __shfl_sync(0xffffffffu, scale, h * W + j);
          };
          // the previous store must have finished reading the staging tile
          if (h == 0) {
            if (lane == 0) bulk_wait_group_read0();
            __syncwarp();
          }
#pragma unroll
          for (int q = 0; q < W / 8; ++q) {
            uint4 o;
            __nv_bfloat162 b;
            b = __floats2bfloat162_rn(scaled(8 * q + 0), scaled(8 * q + 1)); o.x = *reinterpret_cast<uint32_t*>(&b);
            b = __floats2bfloat162_rn(scaled(8 * q + 2), scaled(8 * q + 3)); o.y = *reinterpret_cast<uint32_t*>(&b);
            b = __floats2bfloat162_rn(scaled(8 * q + 4), scaled(8 * q + 5)); o.z = *reinterpret_cast<uint32_t*>(&b);
            b = __floats2bfloat162_rn(scaled(8 * q + 6), scaled(8 * q + 7)); o.w = *reinterpret_cast<uint32_t*>(&b);
            *reinterpret_cast<uint4*>(srow + (((h * (W / 8) + q) ^ sw) << 4)) = o;
          }
          if constexpr (DS) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const uint32_t w4[4] = {dy[q].x, dy[q].y, dy[q].z, dy[q].w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                v[8 * q + 2 * e] = __float_as_uint(__uint_as_float(v[8 * q + 2 * e]) * __uint_as_float(w4[e] << 16));
                v[8 * q + 2 * e + 1] = __float_as_uint(__uint_as_float(v[8 * q + 2 * e + 1]) * __uint_as_float(w4[e] & 0xFFFF0000u));
              }
            }
            if (cc + 1 < chunks || h == 0) load_dy(cc * 32 + h * W + W);
            // fold 32 tokens: at distance o a lane keeps the channels that agree with it in bit o and
            // hands the others over; lanes j and j + 16 end with channel c0 + 16 * h + j
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
              const bool up = lane & o;
#pragma unroll
              for (int j = 0; j < o; ++j) {
                const float keep = __uint_as_float(up ? v[j + o] : v[j]), give = __uint_as_float(up ? v[j] : v[j + o]);
                v[j] = __float_as_uint(keep + __shfl_xor_sync(0xffffffffu, give, o));
              }
            }
            half_sum[h] = __uint_as_float(v[0]) + __shfl_xor_sync(0xffffffffu, __uint_as_float(v[0]), 16);
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0 && row0 < p.T) {
          tma_store_2d(&tmap_y, smem_u32(stage), c0, row0);
          bulk_commit_group();
        }
        if (DS) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (k == cc) ds_sum[k] = lane < 16 ? half_sum[0] : half_sum[1];
        }
      }
      if (chunks == 0) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc_empty_leader);
      }
      if (DS) {
        if (lane == 0) bulk_wait_group_read0();
        __syncwarp();
        float* mine = reinterpret_cast<float*>(stage);
#pragma unroll
        for (int k = 0; k < 8; ++k) mine[k * 32 + lane] = ds_sum[k];
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars->ds_full));
        if (!warp_wait(smem_u32(&bars->ds_full), (uint32_t)(local & 1), abort_flag)) { ok = false; break; }
        // thread = channel: the four warps of a token block, in order
        const int ch = (warp - 4) * 32 + lane;
        const float* all = reinterpret_cast<const float*>(sm_e);
        for (int mb = 0; mb < blocks; ++mb) {
          float sum = 0.0f;
#pragma unroll
          for (int w = 0; w < 4; ++w) sum += all[(mb * 4 + w) * (PE_BYTES / 4) + ch];
          if (n0 + ch < p.N) p.ds_part[(size_t)(((tt0 >> 8) + mb) * 2 + (int)rank) * p.N + n0 + ch] = sum;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars->ds_free));   // behind the stores that used what was read
      }
    }
    if (lane == 0) bulk_wait_group0();             // every store has left shared memory and landed
  } else if (warp >= 12) {
    // ------------------------------------------ weight dequant (this CTA's 128 channels)
    // Group g (four warps) serves the stages with it % 4 == g.  A thread is one channel:
    // it converts the 64 contraction elements of the stage (two units of 32 columns)
    // and writes them as the channel's 128-byte row, 16-byte chunk c at position
    // c ^ (row % 8) (the 128-byte swizzle).
    const int grp = (warp - 12) >> 2;
    const int row = ((warp - 12) & 3) * 32 + lane;
    const int swz = row & 7;
    const uint32_t full_leader0 = mapa_shared(smem_u32(&bars->full[0]), 0);
    const uint32_t total_it = (uint32_t)my_tiles * (uint32_t)p.k_blocks;
    // cursor of the stage whose (s, z) is being prefetched, walked without divisions
    int pf_tile = pair, pf_kb = grp;
    while (pf_kb >= p.k_blocks) { pf_kb -= p.k_blocks; pf_tile += n_pairs; }
    auto item_row = [&](int item) {
      int n_tile, tt0, blocks;
      pair_item(p.items, item, p.T, n_tile, tt0, blocks);
      return n_tile * 256 + (int)rank * 128 + row;
    };
    int pf_r = item_row(pf_tile);
    // every lane reads another row, so each load of a warp touches 32 sectors: the two
    // units of a stage share one load when they share a group (g >= 64, or one scale per
    // channel), and one 2-byte / 8-byte load when the groups are 32 columns wide
    const bool one_group = p.G == 1 || (p.g & 63) == 0;
    const bool pair_load = !one_group && p.g == 32 && (p.G & 1) == 0;
    // Nothing is made of the values here: they are used a turn later, and an operation on one would wait for it.  z: zero-point,
    // its bits if real-valued (ZF), both units' with pair_load; a unit that shares the first one's group has none.
    auto load_zs = [&](uint32_t (&z)[2], float (&sc)[2]) {
      z[0] = z[1] = 0u;
      sc[0] = sc[1] = 0.0f;
      const int col = pf_kb * PK;
      if (pf_r < p.N && col < p.K) {
        const size_t gi = (size_t)pf_r * p.G + pair_group_of(p, col);
        if (!ZF && pair_load) {
          z[0] = ld_global(reinterpret_cast<const unsigned short*>(p.zeros + gi));
          if (FOLD) {
            const float2 s2 = ld_global(reinterpret_cast<const float2*>(p.scales + gi));
            sc[0] = s2.x;
            sc[1] = s2.y;
          }
        } else {
          z[0] = ZF ? __float_as_uint(ld_global(p.zeros_f + gi)) : ld_global(p.zeros + gi);
          if (FOLD) sc[0] = ld_global(p.scales + gi);
          if (!one_group && col + 32 < p.K) {
            const size_t g1 = (size_t)pf_r * p.G + pair_group_of(p, col + 32);
            z[1] = ZF ? __float_as_uint(ld_global(p.zeros_f + g1)) : ld_global(p.zeros + g1);
            if (FOLD) sc[1] = ld_global(p.scales + g1);
          }
        }
      }
      pf_kb += P_GROUPS;
      while (pf_kb >= p.k_blocks) {
        pf_kb -= p.k_blocks;
        pf_tile += n_pairs;
        pf_r = item_row(pf_tile);
      }
    };
    uint32_t z[2], zn[2];
    float sc[2], scn[2];
    int cur_kb = pf_kb;
    if ((uint32_t)grp < total_it) load_zs(z, sc);
    for (uint32_t it = grp; it < total_it; it += P_GROUPS) {
      const int next_kb = pf_kb;
      if (it + P_GROUPS < total_it) load_zs(zn, scn);
      const int s = it % PSTAGES;
      const int q = it % PQ_SLOTS;
      if (!warp_wait(smem_u32(&bars->pk_full[q]), (it / PQ_SLOTS) & 1u, abort_flag)) break;
      uint32_t w[2][BITS];
      {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(sm_q + q * PQ_BYTES) + row * 8;
        const uint4 lo = *reinterpret_cast<const uint4*>(src);
        const uint4 hi = *reinterpret_cast<const uint4*>(src + 4);
        const uint32_t w8[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        if constexpr (BITS == 4) {
#pragma unroll
          for (int e = 0; e < 4; ++e) { w[0][e] = w8[e]; w[1][e] = w8[4 + e]; }
        } else {
          const bool odd = (cur_kb & 1) != 0;
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            w[0][e] = odd ? w8[2 + e] : w8[e];
            w[1][e] = odd ? w8[5 + e] : w8[3 + e];
          }
        }
      }
      uint32_t o0[16], o1[16];
      const float s1 = one_group ? sc[0] : sc[1];
      if constexpr (ZF) {
        dq::unit32_affine<BITS>(w[0], z[0], sc[0], o0);
        dq::unit32_affine<BITS>(w[1], one_group ? z[0] : z[1], s1, o1);
      } else {
        dq::unit32_natural<BITS, FOLD>(w[0], pair_load ? z[0] & 0xFFu : z[0], sc[0], o0);
        dq::unit32_natural<BITS, FOLD>(w[1], one_group ? z[0] : pair_load ? z[0] >> 8 : z[1], s1, o1);
      }
      fence_proxy_async_smem();                                   // the codes have been read
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->pk_empty[q]));   // slot free
      if (!warp_wait_cluster(smem_u32(&bars->empty[s]), ((it / PSTAGES) & 1u) ^ 1u, abort_flag)) break;
      uint8_t* wrow = base + s * PSTAGE_BYTES + PA_BYTES + row * 128;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        *reinterpret_cast<uint4*>(wrow + ((c ^ swz) << 4)) =
            make_uint4(o0[4 * c], o0[4 * c + 1], o0[4 * c + 2], o0[4 * c + 3]);
        *reinterpret_cast<uint4*>(wrow + (((4 + c) ^ swz) << 4)) =
            make_uint4(o1[4 * c], o1[4 * c + 1], o1[4 * c + 2], o1[4 * c + 3]);
      }
      // make the rows visible to the tensor cores of both CTAs, then tell the leader
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster_release(full_leader0 + s * 8);
      z[0] = zn[0]; z[1] = zn[1];
      sc[0] = scn[0]; sc[1] = scn[1];
      cur_kb = next_kb;
    }
  }

  if (*abort_flag) {
    // let copies and MMAs already in flight finish before memory is released
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, P_TMEM_COLS);
  }
  if (threadIdx.x == 0 && bars->abort_flag) {
    atomicExch(p.status, (int)PEQA_ERR_DEVICE_TIMEOUT);
    p.status[1] = (int)blockIdx.x;
  }
}

template <int BITS, bool FOLD, bool ZF, bool DS>
int launch_pair_t(const CUtensorMap& tx, const CUtensorMap& tq, const CUtensorMap& ty, const PairParams& p,
                  int pairs, cudaStream_t st) {
  auto kern = qfwd_pair_kernel<BITS, FOLD, ZF, DS>;
  static std::atomic<uint64_t> done{0};
  PEQA_TRY(allow_smem(kern, P_SMEM_BYTES, done));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs, 1, 1);
  cfg.blockDim = dim3(kPairThreads, 1, 1);
  cfg.dynamicSmemBytes = P_SMEM_BYTES;
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
  PEQA_CUDA(cudaLaunchKernelEx(&cfg, kern, tx, tq, ty, p));
  return PEQA_OK;
}

}  // namespace

// The pair kernel needs a 16-byte row pitch of the packed matrix for its code
// boxes (always true for 4-bit, K % 128 == 0 for 3-bit); other shapes take the
// single-CTA kernel.
bool fwd_pair_supported(const peqa_qweight_t* w) {
  return ((size_t)w->in_features * w->bits / 8) % 16 == 0;
}

int launch_fwd_pair(const peqa_qweight_t* w, const float* zeros_f, int g, const void* X, int T,
                    void* Y, const void* dY, float* ds_part, cudaStream_t st, Side side) {
  PairParams p;
  p.side = side;
  p.zeros = w->zeros;
  p.zeros_f = zeros_f;
  p.scales = w->scales;
  p.out = static_cast<__nv_bfloat16*>(Y);
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
  p.n_tiles = (p.N + 255) / 256;
  p.t_tiles = (T + 511) / 512;
  p.k_blocks = (p.K + PK - 1) / PK;
  PEQA_TRY(status_word(st, &p.status));
  EncodeTiledFn enc = nullptr;
  PEQA_TRY(tensor_map_encoder(&enc));
  CUtensorMap tx, tq, ty;
  {
    // output Y [T, N]: boxes of 32 channels x 32 tokens, 64-byte swizzle (the epilogue's staging tile)
    cuuint64_t dims[2] = {(cuuint64_t)p.N, (cuuint64_t)T};
    cuuint64_t strides[1] = {(cuuint64_t)p.N * 2};
    cuuint32_t box[2] = {32, 32};
    cuuint32_t estr[2] = {1, 1};
    if (enc(&ty, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Y, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
            CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cuda_fail(cudaErrorInvalidValue);
  }
  {
    cuuint64_t dims[2] = {(cuuint64_t)p.K, (cuuint64_t)T};
    cuuint64_t strides[1] = {(cuuint64_t)p.K * 2};
    cuuint32_t box[2] = {64, 128};
    cuuint32_t estr[2] = {1, 1};
    if (enc(&tx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(X), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cuda_fail(cudaErrorInvalidValue);
  }
  {
    const int wpr = p.K * w->bits / 32;
    cuuint64_t dims[2] = {(cuuint64_t)wpr, (cuuint64_t)p.N};
    cuuint64_t strides[1] = {(cuuint64_t)wpr * 4};
    cuuint32_t box[2] = {8, 128};
    cuuint32_t estr[2] = {1, 1};
    if (enc(&tq, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<uint32_t*>(w->qweight), dims, strides,
            box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cuda_fail(cudaErrorInvalidValue);
  }
  int sms = 0, dev = 0;
  PEQA_CUDA(cudaGetDevice(&dev));
  PEQA_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int tiles = p.n_tiles * p.t_tiles;
  const int max_pairs = sms / 2;
  const int pairs = tiles < max_pairs ? tiles : max_pairs;
  p.items = make_pair_items(p.n_tiles, p.t_tiles, T, pairs);
  const bool fold = p.G > 1;
  if (zeros_f)   // a real-valued zero-point is folded into the operand whatever the group size
    return w->bits == 4 ? launch_pair_t<4, true, true, false>(tx, tq, ty, p, pairs, st)
                        : launch_pair_t<3, true, true, false>(tx, tq, ty, p, pairs, st);
  if (fold)
    return w->bits == 4 ? launch_pair_t<4, true, false, false>(tx, tq, ty, p, pairs, st)
                        : launch_pair_t<3, true, false, false>(tx, tq, ty, p, pairs, st);
  if (ds_part)
    return w->bits == 4 ? launch_pair_t<4, false, false, true>(tx, tq, ty, p, pairs, st)
                        : launch_pair_t<3, false, false, true>(tx, tq, ty, p, pairs, st);
  return w->bits == 4 ? launch_pair_t<4, false, false, false>(tx, tq, ty, p, pairs, st)
                      : launch_pair_t<3, false, false, false>(tx, tq, ty, p, pairs, st);
}

}  // namespace peqa
