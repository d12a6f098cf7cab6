// Small-batch forward (token generation) from a prepared copy of the frozen
// weights:  Y[m,i] = sum_g s[i,g] * sum_{j in g} X[m,j] * (Q[i,j] - z[i,g])   (Eq. 2 with
// M <= 16 tokens; Sec. 3.1 / 3.3: the memory-bound matrix-vector regime).
//
// The frozen matrix never changes after quantization (Sec. 3.3), so a server
// can keep it in whatever order suits the kernel.  The prepared layout stores the
// same bits as the canonical packed matrix, rearranged so that
//   * everything one warp needs for one step (8 rows x 512 columns) is one
//     contiguous block that a single bulk copy moves into shared memory, in the
//     order the lanes read it (16 bytes per lane and read, no bank conflicts);
//   * the contraction slots of a warp-level MMA are columns of one quantization
//     group, so the scale and zero-point can be applied per group to the accumulator.
//
// Layout.  rg = row / 8, r = row % 8, step t = column / 512 (T = ceil(K / 512)
// steps; columns beyond K hold zero codes), C = bits.  Block (rg, t) is C*512
// bytes at byte offset (((rg/2)*T + t)*2 + rg%2)*C*512, so the two row groups of a
// pair alternate step by step and a pair's consecutive steps are contiguous
// (an odd count of row groups is padded with a group of zero codes): chunk c
// (0..C-1), lane l (0..31), 16 bytes each, chunk-major.  Lane l = 4*r + c4 owns, of row 8*rg + r, columns
// 8*c4 .. 8*c4+7 of each of the step's sixteen 32-column runs.  Its 4*C words are
// four strings of C words; string s holds runs 4s .. 4s+3, its string column
// cs = 8*(run % 4) + (column % 8); string column 2k sits at code position
// stream_lo(k) and 2k+1 at stream_hi(k) (dequant.cuh), code position p being bits
// [bits*p, bits*p + bits) of the string read as a little-endian bit string.
//
// Work split.  One CTA per SM owns a contiguous range of 8-row groups and all
// of K for them, or, when the activations of more tokens would not fit beside
// the rings, a cluster of CTAs owns the range, each with a slice of K, and their
// sums meet in distributed shared memory (plan_prep): no workspace, no atomics.  Row
// groups 2P and 2P+1 form a "pair", the 16 rows of a warp-level mma.m16n8k16
// whose 8-wide side are the tokens (a range that starts or ends inside a pair
// runs that group as a half pair).  The CTA's (pair, step) list, pair-major, is cut into sixteen
// contiguous ranges of equal cost, one per warp.  A warp streams its range
// through a private ring in shared memory: lane 0 issues one bulk copy per slot
// (one or two steps of a pair: 3 to 8 KiB of contiguous memory; streaming reads
// on this part want few, large copies and well over 100 KiB in flight per SM)
// and all lanes wait on the slot's mbarrier.  The zero-point's term comes off the sums with the
// group (or the row):
//   y += s * (acc - z * sum_j x_j).
//
// Operands.  The integer pipe is what a step of 16 rows x 512 columns is made of, so codes go to the
// tensor core as the fp16 subnormals q * 2^(o - 24) that a code in the low bits of a half-word is
// after one AND (f16_pair in dequant.cuh): 21 integer operations for 32 three-bit codes and 20 for
// four-bit ones, where bf16 operands with an exponent put in took 26 and 28 and left a bias to take off every
// sum.  The activations are brought to the range of fp16 by a power of two per token and lose the 2^o: exact for
// elements down to 2^-25 of the token's largest, smaller ones lose bits (see the staging).  Seven linears of a LLaMA-65B layer in groups of 64, one token, 163.9 ->
// 150.4 us; of a LLaMA-7B layer in groups of 128, seven tokens of several tasks, 94.3 -> 85.1; one scale per
// channel, where the main loop is the smaller part, 16 tokens 230.9 -> 227.3, one token unchanged.
// When a warp's range crosses into the next pair it parks its sums in shared
// memory, in the pair's place or, if its range begins inside the pair, in its own; at the end the parked sums of each pair are added in warp order, so
// results do not depend on timing.  What that final pass needs per token, row and
// pair (sums of x, zero-point and scale, contributing warps) lies ready in tables
// by then: looked up per output it took twice as long as the main loop (12,000
// cycles against 11,400 for 8 tokens at 8192 x 8192; 2,300 with the tables).
//
// Activations are staged in shared memory, all of K when they fit, otherwise in
// chunks of steps with the per-output sums carried in shared memory.
//
// One or two tokens (I8).  Of the eight token columns of an fp16 MMA one or two would be used.  Integer MMAs cover
// twice the contraction, so the activations go in as whole numbers: a step's 512 are scaled by a power
// of two of their own to at most 2^30 and cut into four signed base-256 digits, which fill the eight
// columns for two tokens; the codes are unsigned bytes, eight integer operations for 32 four-bit codes
// and 14 (groups of 64: 18) for three-bit ones (i8_string).  A code at bit o of its byte counts 2^o, which comes off its
// activation before that is rounded, so 30 - o bits are kept, 25 at the least (o <= 5): an element's rounding error
// is at most 2^-25 of the step's largest, exact ones are those down to 2^-17 of it.  Sums of products are
// exact until a group (or a step) is scaled.  The grain is that of the step's largest element, for groups that do
// not hold it too; an emulation gave smaller errors than biased bf16 operands with outliers of 2^12 to
// 2^26 times the others.  A step of a warp takes
// about 1200 cycles instead of 2100 (groups of 64: 2200 / 3000).  One token, us, fp16 / here: 22016 x 8192 in
// groups of 64 28.8 / 25.0, 8192 x 8192 14.6 / 12.6, 11008 x 4096 9.5 / 7.7, 4096 x 4096 6.2 / 5.6, 256 x 256 5.0 / 4.1.
//
// Canonical rows (CANON).  Where no second copy of the weights is kept the same kernel streams the packed matrix
// itself: a step is 16 rows x 512 columns all the same, copied row by row with 16-byte asynchronous
// copies by all lanes, and since the order of a contraction is free a lane takes 32 columns in a
// row where the prepared order gives it eight of each of four runs.  The copies wait for the preceding
// kernel, which may have written the matrix; before that its codes are only asked for in L2.  LLaMA-7B layer in groups
// of 128, three sequences: 103.6 us through decode_stream_kernel, 72.7 here.
//
// Size.  A launch finds the instruction caches cold, and much of a launch of a few microseconds is the
// code's first pass, so there is one copy of everything: loops whose length is not known are not
// unrolled, half pairs run the body of full ones, the steps are cut evenly.  70 to 80 KB of instructions became 40 to
// 49, and one token at 22016 x 8192 in groups of 64 25.0 -> 22.1 us, 8192 x 8192 12.8 -> 11.3, per channel 10.1 ->
// 8.9, 4096 x 4096 5.6 -> 5.1, 256 x 256 4.0 -> 3.6; 16 tokens at 8192 x 8192 19.6 -> 17.7.
//
// Launch overlap.  The kernel is launched with programmatic stream
// serialization: it lets the next kernel in the stream start as soon as SMs
// free up, requests its own first weights at once, and only then waits for the
// preceding kernel before it touches X or Y.  The prepared weights are
// therefore read before earlier work in the stream is known to be complete:
// they must be final when the call is made.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "dequant.cuh"
#include "sm100_ptx.cuh"

namespace peqa {

namespace {

using namespace ptx;

#ifndef PEQA_PREP_WARPS
#define PEQA_PREP_WARPS 16
#endif
constexpr int kPWarps = PEQA_PREP_WARPS;
constexpr int kPThreads = kPWarps * 32;
constexpr int kPSmemLimit = 227 * 1024;
constexpr int kPSmemL1 = 195 * 1024;                              // what leaves 60 KB of L1 (see plan_prep)
constexpr int kPMaxSlots = 4;
constexpr int kStepCols = 512;
constexpr int kI8Units = 64;                                      // most (token, step)s of the integer kernel
constexpr int kPBarBytes = kPWarps * kPMaxSlots * 8;              // the warps' mbarriers
// + abort flag, wait limit, the bounds of the warps' steps and, per token, the sum of x and the factor of its sums
constexpr int kPHeadBytes = (kPBarBytes + 32 + (kPWarps + 1) * 4 + 4 + 16 * 8 + 127) / 128 * 128;

// A pair's sums in shared memory: token by token, the pair's sixteen rows side by side.  Tokens and halves of rows are
// exchanged so that the lanes of a warp that puts down the result of an MMA (rows r8, tokens 2 * c4) meet different banks.
__host__ __device__ inline int pair_sums(int M) { return ((M + 1) & ~1) * 16; }
__device__ __forceinline__ int sum_at(int token, int row) {
  return (token ^ ((token >> 2) & 1)) * 16 + (row ^ ((token << 2) & 8));
}
// n / d = __umulhi(n, quotient_magic(d)) for n * d < 2^32; 0 stands for d = 1.
__host__ __device__ inline uint32_t quotient_magic(int d) { return d > 1 ? 0xFFFFFFFFu / (uint32_t)d + 1u : 0u; }
__device__ __forceinline__ int quotient(int n, uint32_t magic) { return magic ? (int)__umulhi((uint32_t)n, magic) : n; }

struct PrepParams {
  const uint8_t* P;         // prepared or canonical weights
  const uint8_t* zeros;     // [N, G]
  const float* scales;      // [N, G] or table [n_tasks, N, G]
  const __nv_bfloat16* X;   // [M, K]
  __nv_bfloat16* Y;         // [M, N]
  const int32_t* task_ids;  // nullptr: one task
  int n_tasks;
  int N, K, G, M;
  int rgs;                  // row groups in the matrix (N / 8)
  int rg_per_cta;
  int T;                    // steps of 512 columns per row group
  int spc;                  // steps per staged chunk of activations
  int nchunks;
  int slots;                // ring slots per warp
  int sps;                  // steps per slot (1 or 2)
  int x_pitch;              // bytes between staged token rows
  int pairs_per_cta;
  int row_bytes;            // of the canonical matrix
  int cshift;               // log2 of the CTAs that share a range of rows, each with a slice of K
  uint32_t m_magic[2];      // quotient_magic of M and of (M + 1) / 2
  int* status;
};

// d += a * b, or d = a * b when FRESH
template <bool FRESH>
__device__ __forceinline__ void pmma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                           uint32_t b1) {
  if constexpr (FRESH) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
  } else {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  }
}

// Contiguous bulk copy global -> shared memory; its bytes are credited to `bar`.  Both
// addresses 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_load(uint32_t dst_smem, const void* src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(dst_smem), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
      : "memory");
}

// Asks for [src, src + bytes) in L2, shrunk to whole 16-byte units.
__device__ __forceinline__ void prefetch_l2(const void* src, size_t bytes) {
  const uint64_t a = (reinterpret_cast<uint64_t>(src) + 15) & ~(uint64_t)15;
  const uint64_t e = (reinterpret_cast<uint64_t>(src) + bytes) & ~(uint64_t)15;
  if (e > a)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((uint32_t)(e - a)) : "memory");
}

// 16 bytes of a ring slot.  Volatile at both compiler levels: the read must be issued before
// the bulk copy that refills the slot, and neither the compiler nor the assembler can see
// that the copy writes this memory, so an ordinary load could be moved behind it.
__device__ __forceinline__ uint4 ring_load(uint32_t addr) {
  uint4 v;
  asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

__device__ __forceinline__ uint32_t ring_load1(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ void st_shared_f32(uint32_t addr, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

__device__ __forceinline__ float ld_cluster_f32(uint32_t cluster_addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr));
  return v;
}

// Values of a step's quantization groups: the first `left` of TG adjacent entries (those beyond the
// row's last group read as zero).  V: entries come as aligned vectors of V, none of them partly beyond the row.
// (All forms in one kernel, behind a test of the alignment, were 2 KB more for a launch to fetch.  One token in
// groups of 64, us: 4096 x 4096 6.0 -> 5.3, 22016 x 8192 22.0 -> 21.3, 4096 x 11008, whose 172 groups a
// row were single loads, 12.0 -> 9.8; seven of several tasks in groups of 128, 4096 x 11008, 19.4 -> 16.2.)
template <int TG, int V>
__device__ __forceinline__ void load_groups(const float* src, int left, bool row_ok, float (&v)[TG]) {
#pragma unroll
  for (int q = 0; q < TG; q += V) {
    const bool on = row_ok && q < left;
    if constexpr (V == 4) {
      const float4 t = on ? ld_global(reinterpret_cast<const float4*>(src + q)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      v[q] = t.x; v[q + 1] = t.y; v[q + 2] = t.z; v[q + 3] = t.w;
    } else if constexpr (V == 2) {
      const float2 t = on ? ld_global(reinterpret_cast<const float2*>(src + q)) : make_float2(0.0f, 0.0f);
      v[q] = t.x; v[q + 1] = t.y;
    } else {
      v[q] = on ? ld_global(src + q) : 0.0f;
    }
  }
}
// The same for zero-points, four to a word.
template <int TG, int V>
__device__ __forceinline__ void load_zero_bytes(const uint8_t* src, int left, bool row_ok, uint32_t (&v)[(TG + 3) / 4]) {
#pragma unroll
  for (int q = 0; q < (TG + 3) / 4; ++q) v[q] = 0u;
#pragma unroll
  for (int q = 0; q < TG; q += V) {
    if (!row_ok || q >= left) continue;
    if constexpr (V == 4) v[q / 4] = ld_global(reinterpret_cast<const uint32_t*>(src + q));
    else if constexpr (V == 2) v[q / 4] |= (uint32_t)ld_global(reinterpret_cast<const uint16_t*>(src + q)) << (8 * (q & 3));
    else v[q / 4] |= (uint32_t)ld_global(src + q) << (8 * (q & 3));
  }
}

// d += a * b, or d = a * b when FRESH: unsigned codes, signed digits of the activations.
template <bool FRESH>
__device__ __forceinline__ void imma_16832(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                           uint32_t b0, uint32_t b1) {
  if constexpr (FRESH) {
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
        : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(0));
  } else {
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  }
}

// The activations that meet registers 2*JP*2 .. 2*JP*2 + 3 of a string (two MMAs), as signed base-256 digits:
// out[d] is the 16 bytes of digit d.  v: the string's 32 activations times the token's factor 2^k.
template <int BITS, bool CANON, bool HALF, int JP>
__device__ __forceinline__ void x_digits(const float (&v)[32], uint4 (&out)[4]) {
  uint32_t word[4][4];                             // [register][digit]
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t x[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int r = 4 * JP + q;
      const int col = dq::position_column(BITS, CANON, dq::i8_pos(BITS, HALF, r, b));
      // digits in [-128, 127]: 128 is added to the three lower bytes, with carries, and taken off each
      const int xi = __float2int_rn(v[col] * (1.0f / (float)(1 << dq::i8_o(BITS, HALF, r, b))));
      x[b] = ((uint32_t)xi + 0x00808080u) ^ 0x00808080u;
    }
    const uint32_t t0 = dq::prmt(x[0], x[1], 0x5140u), t1 = dq::prmt(x[2], x[3], 0x5140u);
    const uint32_t t2 = dq::prmt(x[0], x[1], 0x7362u), t3 = dq::prmt(x[2], x[3], 0x7362u);
    word[q][0] = dq::prmt(t0, t1, 0x5410u);
    word[q][1] = dq::prmt(t0, t1, 0x7632u);
    word[q][2] = dq::prmt(t2, t3, 0x5410u);
    word[q][3] = dq::prmt(t2, t3, 0x7632u);
  }
#pragma unroll
  for (int d = 0; d < 4; ++d) out[d] = make_uint4(word[0][d], word[1][d], word[2][d], word[3][d]);
}

// One lane's weights of one step: row r of the pair's two groups.
template <int BITS>
struct StepRegs {
  uint4 a[BITS];
  uint4 b[BITS];
};

// Pairs 4*MM .. 4*MM + 3 of a string, whose eight activations are one 16-byte word per token: two MMAs.
// FRESH: the first of a quantization group.
template <int BITS, int NT, int MM, bool FRESH>
__device__ __forceinline__ void run_mma2(const uint32_t (&wa)[BITS], const uint32_t (&wb)[BITS],
                                         const uint8_t* x0, const uint8_t* x1,
                                         float (&acc)[NT][4], float (&acc2)[NT][4]) {
  const uint4 xa = *reinterpret_cast<const uint4*>(x0 + MM * 64);
  uint4 xb = make_uint4(0u, 0u, 0u, 0u);
  if (NT == 2) xb = *reinterpret_cast<const uint4*>(x1 + MM * 64);
  uint32_t f0[4], f1[4];
  f0[0] = dq::f16_pair<BITS, 4 * MM>(wa);
  f0[2] = dq::f16_pair<BITS, 4 * MM + 1>(wa);
  f1[0] = dq::f16_pair<BITS, 4 * MM + 2>(wa);
  f1[2] = dq::f16_pair<BITS, 4 * MM + 3>(wa);
  f0[1] = dq::f16_pair<BITS, 4 * MM>(wb);
  f0[3] = dq::f16_pair<BITS, 4 * MM + 1>(wb);
  f1[1] = dq::f16_pair<BITS, 4 * MM + 2>(wb);
  f1[3] = dq::f16_pair<BITS, 4 * MM + 3>(wb);
  // the two MMAs go to different accumulators, so that consecutive MMAs of a warp do
  // not wait for one another (a single chain of 32 dependent MMAs per step cost 5 % of the
  // kernel); the halves are added when the sums are taken off
  pmma_16816<FRESH>(acc[0], f0, xa.x, xa.y);
  pmma_16816<false>(acc2[0], f1, xa.z, xa.w);
  if (NT == 2) {
    pmma_16816<FRESH>(acc[1], f0, xb.x, xb.y);
    pmma_16816<false>(acc2[1], f1, xb.z, xb.w);
  }
}

// The eight activations that meet pairs 4*MM .. 4*MM + 3 of a string, in that order and without the factors
// 2^o of the codes' places.  v: the string's 32 activations, multiplied by the token's factor, in the order
// of its columns (prepared: dq::string_column; canonical: the code at bit b is column b / BITS).
template <int BITS, bool CANON, int MM>
__device__ __forceinline__ uint4 x_pairs(const float (&v)[32]) {
  uint32_t out[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int j = 4 * MM + e;
    const int lo = CANON ? dq::f16_lo_bit(BITS, j) / BITS : dq::string_column(BITS, dq::f16_lo_bit(BITS, j));
    const int hi = CANON ? dq::f16_hi_bit(BITS, j) / BITS : dq::string_column(BITS, dq::f16_hi_bit(BITS, j));
    const __half2 h = __floats2half2_rn(v[lo] * (1.0f / (float)(1 << dq::f16_lo_o(BITS, j))),
                                        v[hi] * (1.0f / (float)(1 << dq::f16_hi_o(BITS, j))));
    out[e] = *reinterpret_cast<const uint32_t*>(&h);
  }
  return make_uint4(out[0], out[1], out[2], out[3]);
}

// A step of canonical rows in the ring.  Three-bit rows of 192 bytes at a pitch of 208: the 32 words that
// the lanes of a warp read at once (rows r8, columns c4) fall into different banks.  Four-bit rows of 256
// bytes, chunk c of row r at c ^ 4 * (r & 1), so that the 16-byte reads of two rows do not meet.
template <int BITS>
struct CanonRow {
  static constexpr int chunks = 4 * BITS;                    // 16-byte chunks of 512 codes
  static constexpr int pitch = BITS == 3 ? 208 : 256;
};

// V: the groups of a row are aligned vectors of so many, see load_groups.
// GSH: quantization groups of 32 << GSH columns (1: 64, 2: 128, 3: 256), or 0: one group
// per row or groups that are multiples of 512 columns (the sums of a whole staged chunk of
// steps are taken off at once, which needs the chunk to lie inside one group).
// TASKS: grouped scales with a table per task (NT = 1 only).
// CANON: the weights are the canonical packed matrix.
// I8 (one or two tokens, NT = 1, all of K staged at once): integer MMAs.  A token's activations are whole
// numbers of up to 31 bits times a power of two, cut into four signed digits, and the MMA's eight columns
// are two tokens x four digits, which fp16 operands would leave idle.  An MMA covers twice the columns,
// the codes are cheaper to take out (i8_string), and the sums of a group are exact.
template <int BITS, int NT, int GSH, bool TASKS, bool CANON, bool I8, int V>
__global__ void __launch_bounds__(kPThreads, 1)
decode_prep_kernel(const PrepParams p) {
  constexpr int C = BITS;                            // 16-byte chunks per lane, step and group
  constexpr int BLK = C * 512;                       // bytes of one block (rg, t)
  constexpr int TOKP = 8 * NT;
  constexpr bool GROUPED = GSH != 0;
  constexpr int RUNS_PER_GROUP = GROUPED ? (1 << GSH) : 16;
  constexpr int GPS = 16 / RUNS_PER_GROUP;           // groups per step (GROUPED)
  constexpr bool kIndexed = GSH == 1 && NT == 2 && BITS == 4, kWideIndex = kIndexed || (GSH == 1 && TASKS);    // see park
  extern __shared__ uint8_t prep_smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(prep_smem_raw) + 127) &
                                             ~static_cast<uintptr_t>(127));
  uint64_t* bars = reinterpret_cast<uint64_t*>(base);                        // [warps][kPMaxSlots]
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base + kPBarBytes);   // [0] flag, [1] limit
  int* wbound = const_cast<int*>(abort_flag) + 8;                            // [warps + 1] bounds of the chunk
  float* tsum = reinterpret_cast<float*>(wbound + kPWarps + 2);              // [16] sum of a token's x (not GROUPED)
  float* tinv = tsum + 16;                                                   // [16] factor of a token's sums, see stage
  const int pair_floats = pair_sums(p.M);
  // the warp that has a pair's first step leaves its sums in the pair's place, a warp whose range begins inside a pair (its
  // first) leaves them in its own; the pairs' places follow the warps'
  float* part = reinterpret_cast<float*>(base + kPHeadBytes);                // [warps][pair_floats], 128-byte aligned
  float* ywhole = part + kPWarps * pair_floats;                              // [pairs][pair_floats]
  float* yacc = ywhole + p.pairs_per_cta * pair_floats;                      // [pairs][pair_floats] (several chunks)
  // per row: zero-point and scale; per pair: see share_bounds
  float2* rowzs = reinterpret_cast<float2*>(p.nchunks > 1 ? yacc + p.pairs_per_cta * pair_floats : yacc);    // [pairs][16]
  int* pwarps = reinterpret_cast<int*>(rowzs + p.pairs_per_cta * 16);        // [pairs]
  float* xshare = reinterpret_cast<float*>(pwarps + ((p.pairs_per_cta + 3) & ~3));    // [warps] shares of a token's sum of x
  uint32_t* xmax = reinterpret_cast<uint32_t*>(xshare + kPWarps);        // [warps] largest |x| of a warp's share (bf16 bits)
  // I8, in their place: [steps of the tokens] sum of x and factor of the sums
  float* xsum = xshare;
  float* xinv = xshare + kI8Units;
  float* sums = xshare + (I8 ? 2 * kI8Units : 2 * kPWarps);              // GROUPED: [groups of the chunk][TOKP] sum of x
  const size_t sum_floats = GROUPED ? (size_t)p.spc * GPS * TOKP : 0;
  uint8_t* xs = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(sums + sum_floats) + 127) & ~static_cast<uintptr_t>(127));
  // I8: a row of x_pitch bytes per token and digit
  uint8_t* ring = xs + (((size_t)p.M * (I8 ? 4 : 1) * p.x_pitch + 127) & ~static_cast<size_t>(127));

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r8 = lane >> 2, c4 = lane & 3;
  // a cluster of 1 << cshift CTAs owns the rows, each of its CTAs steps [t_lo, t_lo + n_t) of K
  const int rank = (int)(blockIdx.x & ((1u << p.cshift) - 1u));
  const int t_lo = (p.T * rank) >> p.cshift;
  const int n_t = ((p.T * (rank + 1)) >> p.cshift) - t_lo;
  const int rg0 = (int)(blockIdx.x >> p.cshift) * p.rg_per_cta;
  const int rg_end = min(p.rgs, rg0 + p.rg_per_cta);
  // pairs are (2P, 2P+1) for the whole matrix; a range that starts (ends) at an odd row group
  // has a half pair in front (at the end)
  const int P0 = rg0 >> 1;
  const int lead = rg0 & 1;
  const int rest = rg_end - rg0 - lead;
  const int trail = rest & 1;
  const int F = rest >> 1;                           // full pairs
  const int npairs = lead + F + trail;
  using Row = CanonRow<BITS>;
  const int slot_bytes = CANON ? 16 * Row::pitch : 2 * BLK * p.sps;

  // the next kernel of the stream may be scheduled as SMs free up
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (threadIdx.x == 0) {
    abort_flag[0] = 0;
    abort_flag[1] = p.status[4];
  }
  if (lane == 0) {
#pragma unroll 1
    for (int s = 0; s < p.slots; ++s) mbar_init(smem_u32(&bars[warp * kPMaxSlots + s]), CANON ? 32 : 1);
    fence_mbar_init();
  }
  __syncwarp();

  // ---- this warp's steps of a chunk: [bound(w), bound(w+1)) of the pair-major list, equal parts (a half pair's
  // step costs what a full one's does: one copy of the loop body serves both, see below); with fewer
  // steps than warps a step each, so that the warps of a pair are always neighbours
  auto spc_of = [&](int ch) { return min(p.spc, n_t - ch * p.spc); };
  auto bound = [&](int w, int tot) { return tot >= kPWarps ? (int)((unsigned)(w * tot) / kPWarps) : min(w, tot); };
  auto pair_full = [&](int lp) { return lp >= lead && lp < lead + F; };
  // first row group of local pair lp (the only one of a half pair)
  auto pair_rg = [&](int lp) { return lp == 0 ? rg0 : 2 * (P0 + lp); };
  // ---- ring: issue cursor (canonical: the lanes copy together; prepared: only lane 0 uses it)
  const uint32_t ring_w = smem_u32(ring) + (uint32_t)warp * (uint32_t)(p.slots * slot_bytes);
  const uint32_t bar_w = smem_u32(&bars[warp * kPMaxSlots]);
  int i_ch = 0, i_lin = 0, i_hi = 0, i_spc = 1;
  int i_lp = 0, i_tl = 0, i_slot = 0;               // pair and step of i_lin; slot of the next copy
  auto issue_seek = [&]() {       // moves to the first chunk (from i_ch on) where this warp has steps
#pragma unroll 1
    while (i_ch < p.nchunks) {
      i_spc = spc_of(i_ch);
      i_lin = bound(warp, npairs * i_spc);
      i_hi = bound(warp + 1, npairs * i_spc);
      i_lp = i_lin / i_spc;
      i_tl = i_lin - i_lp * i_spc;
      if (i_lin < i_hi) return;
      ++i_ch;
    }
  };
  auto issue_next = [&]() {
    if (i_ch >= p.nchunks) return;
    const int lp = i_lp, tl = i_tl;
    const int t = t_lo + i_ch * p.spc + tl;
    const int n = (p.sps == 2 && i_lin + 1 < i_hi && tl + 1 < i_spc) ? 2 : 1;
    const int rg = pair_rg(lp);
    const int slot = i_slot;
    const uint32_t bar = bar_w + slot * 8;
    const uint32_t dst = ring_w + slot * slot_bytes;
    if constexpr (CANON) {
      // the rows' pieces of the step, 16 bytes per lane and copy; what lies beyond a row's end is not copied
      // (its places meet activations that are zero)
      const uint32_t off = (uint32_t)t * (Row::chunks * 16);
      const uint8_t* src = p.P + (size_t)rg * 8 * p.row_bytes + off;
      const int rows = pair_full(lp) ? 16 : 8;
#pragma unroll
      for (int q = 0; q < Row::chunks / 2; ++q) {
        const int idx = q * 32 + lane, r = idx / Row::chunks, c = idx - r * Row::chunks;
        if (r < rows && off + 16u * c < (uint32_t)p.row_bytes)
          cp_async_16(dst + r * Row::pitch + 16 * (BITS == 4 ? c ^ ((r & 1) << 2) : c),
                      src + (size_t)r * p.row_bytes + 16 * c);
      }
      cp_async_mbar_arrive_noinc(bar);
    } else {
    // block (rg, t) lies at (((rg >> 1) * T + t) * 2 + (rg & 1)) * BLK
    const uint8_t* src = p.P + ((((size_t)(rg >> 1) * p.T + t) * 2 + (rg & 1)) * BLK);
    if (pair_full(lp)) {
      mbar_arrive_expect_tx(bar, n * 2 * BLK);
      bulk_load(dst, src, n * 2 * BLK, bar);                       // steps t .. t+n-1 are contiguous
    } else {
      mbar_arrive_expect_tx(bar, n * BLK);
      bulk_load(dst, src, BLK, bar);
      if (n == 2) bulk_load(dst + 2 * BLK, src + 2 * BLK, BLK, bar);
    }
    }
    i_slot = i_slot + 1 == p.slots ? 0 : i_slot + 1;
    i_lin += n;
    i_tl += n;
    if (i_tl >= i_spc) {
      i_tl = 0;
      ++i_lp;
    }
    if (i_lin >= i_hi) {
      ++i_ch;
      if (!I8) issue_seek();                         // (I8: one chunk)
    }
  };
  // The warps' bounds in a chunk of spc_c steps and, per pair, the first and the last warp with steps of it.  Run by one warp.
  auto share_bounds = [&](int spc_c) {
    const int tot = npairs * spc_c;
    if (lane <= kPWarps) wbound[lane] = bound(lane, tot);
    auto owner = [&](int step) {                     // the last warp whose bound is not beyond the step
      return tot >= kPWarps ? (int)((unsigned)((step + 1) * kPWarps - 1) / (unsigned)tot) : step;
    };
#pragma unroll 1
    for (int lp = lane; lp < npairs; lp += 32) {
      const int l0 = lp * spc_c, l1 = l0 + spc_c;
      pwarps[lp] = owner(l0) | owner(l1 - 1) << 8;
    }
  };
  // One slot per warp is requested while the preceding kernel drains; the others follow the
  // activation requests of the first chunk, which would otherwise queue behind a full ring of
  // weights on their way into this SM (the CTAs that start last wait longest for them).
  // The canonical matrix may be the result of the preceding kernel, so its codes are only asked for in L2,
  // which a late write of them updates: two steps a warp.  All of the CTA's rows at once kept the activations waiting (one scale
  // per channel, us: 22016 x 8192, two tokens, 22.2 / 18.8, 8192 x 8192, one, 10.3 / 9.6); one step a warp is 2 to 3 %
  // slower than all in groups of 128 and 256.
  // What does not depend on the preceding kernel is worked out before the wait for it: where this warp's steps of
  // the first chunk lie (the chunks after it look theirs up), and the tables of the final pass.
  issue_seek();
  const int lo_first = i_ch == 0 ? i_lin : 0, hi_first = i_ch == 0 ? i_hi : 0;
  const int lp_first = i_ch == 0 ? i_lp : 0, tl_first = i_ch == 0 ? i_tl : 0;
  const int last_first = hi_first > lo_first ? (hi_first - 1) / i_spc : -1;
  if (warp == kPWarps - 1) share_bounds(spc_of(0));
  if (CANON) {
    // a row's piece of this warp's first two steps per lane
    const int rg = pair_rg(lp_first);
    const uint32_t off = (uint32_t)(t_lo + tl_first) * (Row::chunks * 16);
    if (hi_first > lo_first && lane < (pair_full(lp_first) ? 16 : 8))
      prefetch_l2(p.P + ((size_t)rg * 8 + lane) * p.row_bytes + off, min((uint32_t)p.row_bytes - off, (uint32_t)Row::chunks * 32));
  } else if (lane == 0) {
    issue_next();
  }
  // I8: sixteen lanes take a step of a token, a lane half of what one of its strings becomes (the half is
  // the warp's); the first of them
  const int u_first = (int)(threadIdx.x >> 4) & 15;
  const int tok_first = I8 && u_first >= n_t ? 1 : 0;

  // everything below reads X or writes Y: the preceding kernel must have completed
  asm volatile("griddepcontrol.wait;" ::: "memory");

  // Grouped scales and zero-points are read a few at a time throughout the kernel: the rows' share of
  // both is requested into L2 as a whole, so that those reads do not each wait for DRAM.
  if (GROUPED && warp == 2) {
    const size_t at = (size_t)rg0 * 8 * p.G, n = (size_t)(rg_end - rg0) * 8 * p.G;   // 8 rows: n % 8 == 0
    const size_t lo = (n * rank >> p.cshift) & ~(size_t)15, hi = (n * (rank + 1) >> p.cshift) & ~(size_t)15;
    const int tabs = p.task_ids ? min(p.n_tasks, 31) : 1;
    if (hi > lo) {
      if (lane < tabs) prefetch_l2(p.scales + (size_t)lane * p.N * p.G + at + lo, (hi - lo) * 4);
      if (lane == 31) prefetch_l2(p.zeros + at + lo, hi - lo);
    }
  }

  int c_slot = 0;
  uint32_t c_phase = 0;                              // parity of the ring's current round

#pragma unroll 1
  for (int ch = 0; ch < p.nchunks; ++ch) {
    const int spc_c = spc_of(ch);
    const int col0 = (t_lo + ch * p.spc) * kStepCols;              // first column of the chunk
    const int ccols = min(p.K - col0, spc_c * kStepCols);          // real columns in it
    if (ch > 0) __syncthreads();                                   // the previous chunk is no longer read
    // ---- stage X[:, chunk] (columns beyond K read as zero): copied as it is, then turned in place into
    // the fp16 operands that meet the codes (x_pairs), with the sums of x per token or per group.  A
    // token's activations are first multiplied by a power of two that brings the largest of them to
    // [2^15, 2^16), then by 2^-o of the code's place (o <= 7, four bits: 4).  Operands from 2^-14 on are normal numbers, which
    // hold a bf16; what is below 2^(o - 29) of the token's largest is rounded to a grain of 2^-24, an error of at most
    // 2^(o - 40) of the largest (bf16's eight bits fit down to 2^(o - 32)).  That is less than a fp32 sum with the largest in it
    // loses; the sums of groups without it get the same grain.  tinv undoes the factor and the 2^-24 of the codes.
    // zero-point and scale of a row, for the final sums (a table per task: scales are looked up there)
    auto row_zs = [&](int r, uint32_t& z, float& sc) {
      z = 0u;
      sc = 0.0f;
      const int lp = r >> 4, lr = r & 15;
      if (r >= npairs * 16 || (!pair_full(lp) && lr >= 8)) return;
      const size_t at = (size_t)(pair_rg(lp) * 8 + lr) * p.G + (p.G == 1 ? 0 : col0 / (p.K / p.G));
      z = ld_global(p.zeros + at);
      if (!p.task_ids) sc = ld_global(p.scales + at);
    };
    uint32_t z_own = 0u;
    float s_own = 0.0f;
    // A token belongs to 16 / Mp warps (Mp: M rounded up to a power of two); a warp copies and turns
    // every (16 / Mp)-th step of its token, two at a time: lane 16 * j + 4 * s + c4 owns what string s
    // of the j-th of them meets in lanes c4 of the MMAs, so it needs no other thread's copies.
    int mp = 1;                                                    // (fp16) M rounded up to a power of two
#pragma unroll 1
    while (mp < p.M) mp <<= 1;
    if constexpr (I8) {
      // A step has a factor of its own, so no thread waits for another's activations.  The next turn's are
      // loaded ahead.
      const int str = (lane >> 2) & 3, units = p.M * spc_c;
      const bool upper = warp >= kPWarps / 2;                      // which half of the string's registers
      const int own_col = str * 128 + (CANON ? c4 * 32 : c4 * 8);
      const __nv_bfloat16* xcol = p.X + col0 + own_col;
      uint4 next[4];
      int next_tok = tok_first;                                    // of unit u: (token, step), token-major, two tokens at most
      auto load = [&](int u) {
        const int col = (u - next_tok * spc_c) * kStepCols;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          next[r] = make_uint4(0u, 0u, 0u, 0u);
          if (u < units && col + own_col + (CANON ? r * 8 : r * 32) < ccols)
            next[r] = ld_global(reinterpret_cast<const uint4*>(xcol + (size_t)next_tok * p.K + col + (CANON ? r * 8 : r * 32)));
        }
      };
      load(u_first);
      if (CANON || lane == 0)
#pragma unroll 1
        for (int s = CANON ? 0 : 1; s < p.slots; ++s) issue_next();
#pragma unroll 1
      for (int u0 = 0; u0 < units; u0 += 16) {
        uint4 raw[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) raw[r] = next[r];
        const int u = u0 + u_first, tok = next_tok, st = u - tok * spc_c;
        const bool live = u < units;
        if (u0 + 16 < units) {
          next_tok = u + 16 >= spc_c ? 1 : 0;
          load(u + 16);
        }
        uint32_t mx = 0u;                                          // two largest |x|, as bf16 bits
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          mx = __vmaxu2(__vmaxu2(mx, raw[r].x & 0x7FFF7FFFu), raw[r].y & 0x7FFF7FFFu);
          mx = __vmaxu2(__vmaxu2(mx, raw[r].z & 0x7FFF7FFFu), raw[r].w & 0x7FFF7FFFu);
        }
        mx = max(mx & 0xFFFFu, mx >> 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        // |x| 2^k < 2^30 (2^-k a fp32 number: k <= 149), 2^k in two factors where it is not one
        const int k = min(156 - (int)(mx >> 7), 149);
        const float up = __uint_as_float((uint32_t)(min(k, 126) + 127) << 23);
        float v[32];
        float hsum[2] = {0.0f, 0.0f};                              // of the string's first and second half
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t wv[4] = {raw[q].x, raw[q].y, raw[q].z, raw[q].w};
          float t0 = 0.0f, t1 = 0.0f;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            v[q * 8 + 2 * e] = __uint_as_float(wv[e] << 16) * up;
            v[q * 8 + 2 * e + 1] = __uint_as_float(wv[e] & 0xFFFF0000u) * up;
            t0 += v[q * 8 + 2 * e];
            t1 += v[q * 8 + 2 * e + 1];
          }
          hsum[q >> 1] += t0 + t1;
        }
        if (k > 126) {
          const float up2 = __uint_as_float((uint32_t)(k - 126 + 127) << 23);
#pragma unroll
          for (int e = 0; e < 32; ++e) v[e] *= up2;
          hsum[0] *= up2;
          hsum[1] *= up2;
        }
        if (live) {
          uint8_t* at = xs + (size_t)tok * 4 * p.x_pitch + st * kStepCols + str * 128 + c4 * 16;
          uint4 dig[4];
          if (upper) {
            x_digits<BITS, CANON, GSH == 1, 1>(v, dig);
            at += 64;
          } else {
            x_digits<BITS, CANON, GSH == 1, 0>(v, dig);
          }
#pragma unroll
          for (int d = 0; d < 4; ++d) *reinterpret_cast<uint4*>(at + d * p.x_pitch) = dig[d];
        }
        if (upper) continue;                                       // (the warp) the sums are the other half's
        // 2^-k; an infinity or a NaN among the activations makes it a NaN, and with it the token
        const float inv = mx >= 0x7F80u ? __uint_as_float(0x7FC00000u)
                                        : __uint_as_float(k <= 126 ? (uint32_t)(127 - k) << 23 : 1u << (149 - k));
        if (live && (lane & 15) == 0) xinv[u] = inv;
        if (!GROUPED) {
          float t = hsum[0] + hsum[1];
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
          if (live && (lane & 15) == 0) xsum[u] = t * inv;
        } else {
          if (RUNS_PER_GROUP > 2) hsum[0] += hsum[1];
#pragma unroll
          for (int h = 0; h < (RUNS_PER_GROUP == 2 ? 2 : 1); ++h) {
            float t = hsum[h];
            t += __shfl_xor_sync(0xffffffffu, t, 1);
            t += __shfl_xor_sync(0xffffffffu, t, 2);
            if (RUNS_PER_GROUP == 8) t += __shfl_xor_sync(0xffffffffu, t, 4);
            const int gi = RUNS_PER_GROUP == 2 ? 2 * str + h : RUNS_PER_GROUP == 4 ? str : str >> 1;
            // in the units of the upper two digits' sums
            if (live && c4 == 0 && (RUNS_PER_GROUP != 8 || (str & 1) == 0))
              sums[(size_t)(st * GPS + gi) * TOKP + tok] = t * (1.0f / 65536.0f);
          }
        }
      }
    } else {
      const int wpt = kPWarps / mp;                                  // warps per token
      const int tok = warp / wpt, sub = warp - tok * wpt;
      const int str = (lane >> 2) & 3;                               // the lane's string of a step
      uint8_t* own = xs + (size_t)(tok < p.M ? tok : 0) * p.x_pitch + str * 256 + c4 * 16;
      const int st0 = sub + (lane >> 4) * wpt;
      if (tok < p.M)
#pragma unroll 1
        for (int st = st0; st < spc_c; st += 2 * wpt)
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            // the string's columns by eights: one in each of its four runs, or 32 in a row
            const int col = st * kStepCols + str * 128 + (CANON ? c4 * 32 + r * 8 : r * 32 + c4 * 8);
            uint8_t* dst = own + st * 1024 + r * 64;
            if (col < ccols) cp_async_16(smem_u32(dst), p.X + (size_t)tok * p.K + col0 + col);
            else *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
          }
      asm volatile("cp.async.commit_group;" ::: "memory");
      if (ch == 0 && (CANON || lane == 0))
#pragma unroll 1
        for (int s = CANON ? 0 : 1; s < p.slots; ++s) issue_next();
      if (ch > 0 && warp == kPWarps - 1) share_bounds(spc_c);                  // while the activations are on their way
      // (of the ring's copies the first chunk's are in no group yet; canonical ones issued since, while a chunk
      // was worked through, joined this chunk's group, and its activations wait for them too)
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      {
        uint32_t mx = 0u;                                            // two largest |x|, as bf16 bits
        if (tok < p.M)
#pragma unroll 1
          for (int st = st0; st < spc_c; st += 2 * wpt)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const uint4 v = *reinterpret_cast<const uint4*>(own + st * 1024 + r * 64);
              mx = __vmaxu2(__vmaxu2(mx, v.x & 0x7FFF7FFFu), v.y & 0x7FFF7FFFu);
              mx = __vmaxu2(__vmaxu2(mx, v.z & 0x7FFF7FFFu), v.w & 0x7FFF7FFFu);
            }
        mx = __reduce_max_sync(0xffffffffu, max(mx & 0xFFFFu, mx >> 16));
        if (lane == 0) xmax[warp] = mx;
      }
      __syncthreads();
      if (tok < p.M) {
        uint32_t mx = 0u;
#pragma unroll 1
        for (int w = 0; w < wpt; ++w) mx = max(mx, xmax[tok * wpt + w]);
        // factor 2^k, its exponent field: 15 - (E - 127) + 127 with E the largest one's, a finite number for all E
        const int kf = min(269 - (int)(mx >> 7), 253);
        const float up = __uint_as_float((uint32_t)kf << 23);        // 2^k, k = kf - 127 in [-113, 126]
        float sx = 0.0f;                                             // this lane's share of the token's sum (times 2^k)
#pragma unroll 1
        for (int sb = sub; sb < spc_c; sb += 2 * wpt) {
          const int st = sb + (lane >> 4) * wpt;
          const bool live = st < spc_c;
          float hsum[2] = {0.0f, 0.0f};                              // of the string's first and second half
          if (live) {
            uint8_t* at = own + st * 1024;
            float v[32];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint4 raw = *reinterpret_cast<const uint4*>(at + q * 64);
              const uint32_t wv[4] = {raw.x, raw.y, raw.z, raw.w};
              float t0 = 0.0f, t1 = 0.0f;
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                v[q * 8 + 2 * e] = __uint_as_float(wv[e] << 16) * up;
                v[q * 8 + 2 * e + 1] = __uint_as_float(wv[e] & 0xFFFF0000u) * up;
                t0 += v[q * 8 + 2 * e];
                t1 += v[q * 8 + 2 * e + 1];
              }
              hsum[q >> 1] += t0 + t1;
            }
            *reinterpret_cast<uint4*>(at) = x_pairs<BITS, CANON, 0>(v);
            *reinterpret_cast<uint4*>(at + 64) = x_pairs<BITS, CANON, 1>(v);
            *reinterpret_cast<uint4*>(at + 128) = x_pairs<BITS, CANON, 2>(v);
            *reinterpret_cast<uint4*>(at + 192) = x_pairs<BITS, CANON, 3>(v);
          }
          if (!GROUPED) {
            sx += hsum[0] + hsum[1];
          } else {
            // a group of 64 columns is half a string of the four lanes c4, 128 a string, 256 two strings;
            // in the units of the accumulators: 2^-24 for the codes
            if (RUNS_PER_GROUP > 2) hsum[0] += hsum[1];
#pragma unroll
            for (int h = 0; h < (RUNS_PER_GROUP == 2 ? 2 : 1); ++h) {
              float t = hsum[h];
              t += __shfl_xor_sync(0xffffffffu, t, 1);
              t += __shfl_xor_sync(0xffffffffu, t, 2);
              if (RUNS_PER_GROUP == 8) t += __shfl_xor_sync(0xffffffffu, t, 4);
              const int gi = RUNS_PER_GROUP == 2 ? 2 * str + h : RUNS_PER_GROUP == 4 ? str : str >> 1;
              if (live && c4 == 0 && (RUNS_PER_GROUP != 8 || (str & 1) == 0))
                sums[(size_t)(st * GPS + gi) * TOKP + tok] = t * 5.9604644775390625e-8f;
            }
          }
        }
        if (!GROUPED) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) sx += __shfl_xor_sync(0xffffffffu, sx, o);
          // 2^-k: its exponent field is 254 - kf, and 2^-126 (a normal number) at the least
          if (lane == 0) xshare[warp] = sx * __uint_as_float((uint32_t)(254 - kf) << 23);
        }
        // what is left of 2^(24 - k) after 2^12, which is applied first
        if (sub == 0 && lane == 0) tinv[tok] = __uint_as_float((uint32_t)(266 - kf) << 23);
      }
    }
    __syncthreads();

    // a row per thread is fetched now and put down after the main loop, so that nothing waits for it
    if (!GROUPED) row_zs((int)threadIdx.x, z_own, s_own);
    // ---- this warp's steps of the chunk
    int lo = lo_first, hi = hi_first, first_pair = lp_first, last_pair = last_first, tl = tl_first;
    if (!I8 && ch > 0) {
      lo = wbound[warp];
      hi = wbound[warp + 1];
      first_pair = lo / spc_c;
      last_pair = hi > lo ? (hi - 1) / spc_c : -1;
      tl = lo - first_pair * spc_c;
    }
    int cur_pair = -1;
    const int own_first = tl == 0 ? -1 : first_pair;               // begins inside it
    // I8: yv[0][0] and yv[0][1] are this lane's share of its two rows (rows r8 and r8 + 8), token c4 / 2, of the
    // lower (c4 even) or upper two digits
    float acc[NT][4], acc2[NT][4], yv[NT][4];
    const float zfac = (c4 & 1) ? -1.0f : 0.0f;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[nt][e] = acc2[nt][e] = yv[nt][e] = 0.0f;
    // By 32-bit addresses, the parts of a result apart by bits 5 and 6 of its own (a pair's sums begin at multiples of 128
    // bytes): with pointers the kernels ran out of registers.  us, pointers / this: 16 tokens at 4552 x 1536 6.45 / 6.1, nine
    // at 22016 x 8192 in groups of 128 37.1 / 34.2, two at 13752 x 3328 in groups of 128 8.0 / 7.65.  What a loop of 128 registers spills depends on
    // the arithmetic around it, so two kinds of kernel, whose scales of a step take the most registers, have it in another form
    // (kIndexed here, kWideIndex in the final pass; us, without / with them: 4 bits in groups of 64, 11 tokens at 22016 x 8192 51.4 / 47.4, 16 at
    // 4096 x 11008 22.1 / 20.9; 3 bits in groups of 64, nine tokens of several tasks at 17048 x 7040 92 / 84).
    auto park = [&]() {
      const uint32_t mine = smem_u32(part) + (uint32_t)((cur_pair == own_first ? warp : kPWarps + cur_pair) * pair_floats) * 4;
      if constexpr (I8) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float v = (c4 & 1) ? yv[0][e] * 65536.0f : yv[0][e];
          v += __shfl_xor_sync(0xffffffffu, v, 1);
          if ((c4 & 1) == 0) st_shared_f32(mine + ((c4 >> 1) * 16 + r8 + 8 * e) * 4, v);      // sum_at; there is room for two tokens
          yv[0][e] = 0.0f;
        }
      } else {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const int tk = nt * 8 + c4 * 2;
          float v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = (GROUPED ? yv[nt][e] : acc[nt][e] + acc2[nt][e]) * 4096.0f;
          if (tk < p.M) {
            const float2 f = *reinterpret_cast<const float2*>(tinv + tk);
            const uint32_t i = (uint32_t)(nt * 128 + sum_at(c4 * 2, r8)), at = mine + i * 4;
            st_shared_f32(at, v[0] * f.x);
            st_shared_f32(kIndexed ? mine + (i ^ 8) * 4 : at ^ 32, v[2] * f.x);
            st_shared_f32(kIndexed ? mine + (i ^ 16) * 4 : at ^ 64, v[1] * f.y);
            st_shared_f32(kIndexed ? mine + (i ^ 24) * 4 : at ^ 96, v[3] * f.y);
          }
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[nt][e] = acc2[nt][e] = yv[nt][e] = 0.0f;
        }
      }
    };
    // I8: this lane's column of the MMAs is digit r8 % 4 of token r8 / 4
    const uint8_t* xl = xs + (size_t)(I8 ? (p.M > 1 ? r8 : r8 & 3) : r8 < p.M ? r8 : 0) * p.x_pitch + c4 * 16;
    const uint8_t* xh = xs + (size_t)(r8 + 8 < p.M ? r8 + 8 : 0) * p.x_pitch + c4 * 16;

    // tasks of this lane's two tokens (grouped scales with a table per task)
    int task_of[2] = {0, 0};
    if (TASKS) {
#pragma unroll
      for (int e = 0; e < 2; ++e)
        if ((I8 ? c4 >> 1 : c4 * 2 + e) < p.M)
          task_of[e] = min(max(ld_global(p.task_ids + (I8 ? c4 >> 1 : c4 * 2 + e)), 0), p.n_tasks - 1);
    }
    int lin = lo;
    int lp = first_pair;
#pragma unroll 1
    while (lin < hi) {
      const int nsteps = (p.sps == 2 && lin + 1 < hi && tl + 1 < spc_c) ? 2 : 1;
      const int slot = c_slot;
      // A lane whose bound has run out goes on with the others, over whatever the slot holds: nothing behind
      // the wait then misses it.  (A vote of the warp cost up to 4 %: eight tokens of several tasks at 3520 x 512 5.65 / 5.9 us.)
      if (!mbar_wait(bar_w + slot * 8, c_phase, abort_flag)) i_ch = p.nchunks;     // nothing more is asked for
      if (++c_slot == p.slots) {
        c_slot = 0;
        c_phase ^= 1u;
      }
#pragma unroll 1
      for (int j = 0; j < nsteps; ++j) {
        if (lp != cur_pair) {
          if (cur_pair >= 0) park();
          cur_pair = lp;
        }
        const bool has_b = pair_full(lp);
        StepRegs<BITS> w;
        {
          const uint32_t sp = ring_w + (uint32_t)(slot * slot_bytes);
          if constexpr (CANON && BITS == 4) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const uint32_t at = sp + r8 * Row::pitch + (((4 * c + c4) ^ ((r8 & 1) << 2)) << 4);
              w.a[c] = ring_load(at);
              w.b[c] = has_b ? ring_load(at + 8 * Row::pitch) : make_uint4(0u, 0u, 0u, 0u);
            }
          } else if constexpr (CANON) {
            uint32_t* wa = reinterpret_cast<uint32_t*>(w.a);
            uint32_t* wb = reinterpret_cast<uint32_t*>(w.b);
#pragma unroll
            for (int c = 0; c < 12; ++c) {
              const uint32_t at = sp + r8 * Row::pitch + (c / 3) * 48 + c4 * 12 + (c % 3) * 4;
              wa[c] = ring_load1(at);
              wb[c] = has_b ? ring_load1(at + 8 * Row::pitch) : 0u;
            }
          } else {
            const uint32_t at = sp + (uint32_t)(j * 2 * BLK + lane * 16);
#pragma unroll
            for (int c = 0; c < C; ++c) w.a[c] = ring_load(at + c * 512);
            if (has_b) {
#pragma unroll
              for (int c = 0; c < C; ++c) w.b[c] = ring_load(at + (C + c) * 512);
            } else {
#pragma unroll
              for (int c = 0; c < C; ++c) w.b[c] = make_uint4(0u, 0u, 0u, 0u);
            }
          }
        }

        // scales (with a table per task: of this lane's two tokens) and zero-points of this lane's
        // two rows for all groups of the step, requested before the first MMA: loaded one by one
        // where a group ends, their latency was on the path of every group
        const int rowa = pair_rg(lp) * 8 + r8, rowb = rowa + 8;
        const int gstep0 = (t_lo + ch * p.spc + tl) * GPS;         // first group of the step
        constexpr int TG = GROUPED ? GPS : 1, NS = TASKS && !I8 ? 2 : 1;
        float gsa[NS][TG], gsb[NS][TG];
        uint32_t gza[(TG + 3) / 4], gzb[(TG + 3) / 4];             // four zero-points to a word
        if (GROUPED) {
          load_zero_bytes<TG, V>(p.zeros + (size_t)rowa * p.G + gstep0, p.G - gstep0, true, gza);
          load_zero_bytes<TG, V>(p.zeros + (size_t)rowb * p.G + gstep0, p.G - gstep0, has_b, gzb);
#pragma unroll
          for (int e = 0; e < NS; ++e) {
            const float* tab = p.scales + (TASKS ? (size_t)task_of[e] * p.N * p.G : 0) + gstep0;
            load_groups<TG, V>(tab + (size_t)rowa * p.G, p.G - gstep0, true, gsa[e]);
            load_groups<TG, V>(tab + (size_t)rowb * p.G, p.G - gstep0, has_b, gsb[e]);
          }
        }
        if constexpr (I8) {
          // per string (a lane's 32 columns) four MMAs; a group is half a string (two MMAs), a string or two
          const uint32_t* fa = reinterpret_cast<const uint32_t*>(w.a);
          const uint32_t* fb = reinterpret_cast<const uint32_t*>(w.b);
          const uint8_t* x0 = xl + (size_t)tl * kStepCols;
          int d0[4], d1[4];
          float ys[2] = {0.0f, 0.0f};              // of the step, in units of 2^-k
          // rows r8 (d[0], d[1]: the lower and the higher of two digits) and r8 + 8; exact in 32 bits for 256 columns
          auto value = [&](const int (&d)[4], int e) { return (float)(d[2 * e] + d[2 * e + 1] * 256); };
          auto flush = [&](int gi, const int (&d)[4]) {
            const int q = gi % TG;
            const float sx = sums[(size_t)(tl * GPS + gi) * TOKP + (c4 >> 1)] * zfac;
            const float za = (float)((gza[q >> 2] >> (8 * (q & 3))) & 0xFFu);
            const float zb = (float)((gzb[q >> 2] >> (8 * (q & 3))) & 0xFFu);
            ys[0] = fmaf(gsa[0][q], fmaf(za, sx, value(d, 0)), ys[0]);
            ys[1] = fmaf(gsb[0][q], fmaf(zb, sx, value(d, 1)), ys[1]);
          };
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            uint32_t wa[BITS], wb[BITS], ra[8], rb[8];
#pragma unroll
            for (int e = 0; e < BITS; ++e) {
              wa[e] = fa[s * BITS + e];
              wb[e] = fb[s * BITS + e];
            }
            dq::i8_string<BITS, GSH == 1>(wa, ra);
            dq::i8_string<BITS, GSH == 1>(wb, rb);
            const uint4 xa = *reinterpret_cast<const uint4*>(x0 + s * 128);
            const uint4 xb = *reinterpret_cast<const uint4*>(x0 + s * 128 + 64);
            constexpr bool kHalf = GSH == 1;
            const bool fresh = GSH == 1 || GSH == 2 || s == 0 || (GSH == 3 && (s & 1) == 0);
            // two chains of MMAs, so that they do not wait for one another; half a string (kHalf): a chain each
            if (fresh) {
              imma_16832<true>(d0, ra[0], rb[0], ra[1], rb[1], xa.x, xa.y);
              imma_16832<true>(d1, ra[4], rb[4], ra[5], rb[5], xb.x, xb.y);
            } else {
              imma_16832<false>(d0, ra[0], rb[0], ra[1], rb[1], xa.x, xa.y);
              imma_16832<false>(d1, ra[4], rb[4], ra[5], rb[5], xb.x, xb.y);
            }
            imma_16832<false>(d0, ra[2], rb[2], ra[3], rb[3], xa.z, xa.w);
            imma_16832<false>(d1, ra[6], rb[6], ra[7], rb[7], xb.z, xb.w);
            if (kHalf) {
              flush(2 * s, d0);
              flush(2 * s + 1, d1);
            } else if (GROUPED && (RUNS_PER_GROUP == 4 || (s & 1))) {
#pragma unroll
              for (int e = 0; e < 4; ++e) d0[e] += d1[e];
              flush(RUNS_PER_GROUP == 4 ? s : s >> 1, d0);
            }
          }
          if (!GROUPED) {
            // a step's sums of one digit are below 2^24: exact as fp32, each chain's
#pragma unroll
            for (int e = 0; e < 2; ++e)
              ys[e] = fmaf(256.0f, (float)(d0[2 * e + 1] + d1[2 * e + 1]), (float)(d0[2 * e] + d1[2 * e]));
          }
          const float inv = xinv[(p.M > 1 && c4 >= 2 ? spc_c : 0) + tl];
          yv[0][0] = fmaf(ys[0], inv, yv[0][0]);
          yv[0][1] = fmaf(ys[1], inv, yv[0][1]);
        } else {
          // group gi of the step begins: one of its two accumulators starts at -z * sum x ...
          auto begin = [&](int gi) {
            const int q = gi % TG;
            const float za = -(float)((gza[q >> 2] >> (8 * (q & 3))) & 0xFFu);
            const float zb = -(float)((gzb[q >> 2] >> (8 * (q & 3))) & 0xFFu);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
              const float2 sx = *reinterpret_cast<const float2*>(sums + (size_t)(tl * GPS + gi) * TOKP + nt * 8 + c4 * 2);
              acc2[nt][0] = za * sx.x;
              acc2[nt][1] = za * sx.y;
              acc2[nt][2] = zb * sx.x;
              acc2[nt][3] = zb * sx.y;
            }
          };
          // ... and ends: scale
          auto flush = [&](int gi) {
            const int q = gi % TG;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                yv[nt][e] = fmaf(gsa[e % NS][q], acc[nt][e] + acc2[nt][e], yv[nt][e]);
                yv[nt][2 + e] = fmaf(gsb[e % NS][q], acc[nt][2 + e] + acc2[nt][2 + e], yv[nt][2 + e]);
              }
          };

          const uint32_t* fa = reinterpret_cast<const uint32_t*>(w.a);
          const uint32_t* fb = reinterpret_cast<const uint32_t*>(w.b);
          const uint8_t* x0 = xl + (size_t)tl * (kStepCols * 2);
          const uint8_t* x1 = xh + (size_t)tl * (kStepCols * 2);
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            uint32_t wa[BITS], wb[BITS];
#pragma unroll
            for (int e = 0; e < BITS; ++e) {
              wa[e] = fa[s * BITS + e];
              wb[e] = fb[s * BITS + e];
            }
            const uint8_t* xs0 = x0 + s * 256;
            const uint8_t* xs1 = x1 + s * 256;
            constexpr bool kHalf = GROUPED && RUNS_PER_GROUP == 2;     // a group is half a string
            if (GROUPED && RUNS_PER_GROUP <= 4) begin(kHalf ? 2 * s : s);
            if (GROUPED && RUNS_PER_GROUP == 8 && (s & 1) == 0) begin(s >> 1);
            constexpr bool kFresh = GROUPED && RUNS_PER_GROUP <= 4;
            if (GROUPED && RUNS_PER_GROUP == 8 && (s & 1) == 0) {
#pragma unroll
              for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[nt][e] = 0.0f;
            }
            // (a half pair's second rows are codes of zero: a copy of the body without them saved a quarter of
            // such a step, but the kernel's 70 to 80 KB of instructions are fetched anew in every launch)
            run_mma2<BITS, NT, 0, kFresh>(wa, wb, xs0, xs1, acc, acc2);
            run_mma2<BITS, NT, 1, false>(wa, wb, xs0, xs1, acc, acc2);
            if (kHalf) {
              flush(2 * s);
              begin(2 * s + 1);
            }
            run_mma2<BITS, NT, 2, kHalf>(wa, wb, xs0, xs1, acc, acc2);
            run_mma2<BITS, NT, 3, false>(wa, wb, xs0, xs1, acc, acc2);
            if (kHalf) flush(2 * s + 1);
            if (GROUPED && RUNS_PER_GROUP == 4) flush(s);
            if (GROUPED && RUNS_PER_GROUP == 8 && (s & 1)) flush(s >> 1);
          }
        }
        if (j + 1 == nsteps) {
          // Every lane has read its part of the slot: it can be refilled.  Behind the step's MMAs, where
          // the fence finds the reads done; right behind the reads it waits for them (LLaMA-65B layer in
          // groups of 64, one token: 166 us there, 164 here).
          if constexpr (CANON) {
            __syncwarp();               // these copies go through the proxy of the reads
            issue_next();
          } else {
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) issue_next();
          }
        }
        ++lin;
        if (++tl == spc_c) {
          tl = 0;
          ++lp;
        }
      }
    }
    if (cur_pair >= 0) park();
    if (!GROUPED) {
      if (warp == kPWarps - 1) {                       // the tokens' sums of x from their warps' shares
        if constexpr (I8) {
#pragma unroll 1
          for (int m = 0; m < p.M; ++m) {
            float t = 0.0f;
#pragma unroll 1
            for (int st = lane; st < spc_c; st += 32) t += xsum[m * spc_c + st];
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) tsum[m] = t;
          }
        } else {
          float t = lane < kPWarps ? xshare[lane] : 0.0f;
#pragma unroll 1
          for (int o = kPWarps / mp / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
          if (lane < kPWarps && (lane & (kPWarps / mp - 1)) == 0) tsum[lane / (kPWarps / mp)] = t;
        }
      }
      if (threadIdx.x < npairs * 16) rowzs[threadIdx.x] = make_float2((float)z_own, s_own);
#pragma unroll 1
      for (int r = threadIdx.x + kPThreads; r < npairs * 16; r += kPThreads) {
        row_zs(r, z_own, s_own);
        rowzs[r] = make_float2((float)z_own, s_own);
      }
    }
    __syncthreads();

    const bool last = ch + 1 == p.nchunks;
    // ---- add the parked sums of every pair in warp order: a thread finishes two tokens of a row
    const int mpairs = (p.M + 1) >> 1;
#pragma unroll 1
    for (int idx = threadIdx.x; idx < npairs * 16 * mpairs; idx += kPThreads) {
      const int lr = idx & 15, lp = quotient(idx >> 4, p.m_magic[1]), m = ((idx >> 4) - lp * mpairs) * 2;
      if (!pair_full(lp) && lr >= 8) continue;                     // a half pair has eight rows
      const int row = pair_rg(lp) * 8 + lr;
      const int pw = pwarps[lp], wa = pw & 0xFF, wb = pw >> 8;
      const int at0 = sum_at(m, lr), at1 = sum_at(m + 1, lr);
      float* mine = ywhole + lp * pair_floats;
      float sum[2] = {mine[at0], mine[at1]};
      // four at a time, so that the reads do not wait for one another
#pragma unroll 1
      for (int w = wa + 1; w <= wb; w += 4) {
        float v[4][2];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float* from = part + (kWideIndex ? (size_t)(w + q) * pair_floats : (size_t)((w + q) * pair_floats));
          v[q][0] = w + q <= wb ? from[at0] : 0.0f;
          v[q][1] = w + q <= wb ? from[at1] : 0.0f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          sum[0] += v[q][0];
          sum[1] += v[q][1];
        }
      }
      if (!GROUPED) {
        // the chunk lies inside one group: take its zero-point term off, then scale
        const float2 zs = rowzs[lp * 16 + lr];
        const float t0 = tsum[m], t1 = tsum[m + 1];
        float s0 = zs.y, s1 = zs.y;
        if (p.task_ids) {
          const int gg = p.G == 1 ? 0 : col0 / (p.K / p.G);
          const float* tab = p.scales + (size_t)row * p.G + gg;
          const size_t per = (size_t)p.N * p.G;
          s0 = ld_global(tab + (size_t)min(max(ld_global(p.task_ids + m), 0), p.n_tasks - 1) * per);
          if (m + 1 < p.M) s1 = ld_global(tab + (size_t)min(max(ld_global(p.task_ids + m + 1), 0), p.n_tasks - 1) * per);
        }
        sum[0] = fmaf(-zs.x, t0, sum[0]) * s0;
        sum[1] = fmaf(-zs.x, t1, sum[1]) * s1;
      }
      if (p.nchunks > 1) {
        float* ya = yacc + lp * pair_floats;
        if (ch > 0) {
          sum[0] += ya[at0];
          sum[1] += ya[at1];
        }
        if (!last) {
          ya[at0] = sum[0];
          ya[at1] = sum[1];
          continue;
        }
      } else if (p.cshift) {
        mine[at0] = sum[0];                                        // read above by this thread alone
        mine[at1] = sum[1];
        continue;
      }
      p.Y[(size_t)m * p.N + row] = __float2bfloat16_rn(sum[0]);
      if (m + 1 < p.M) p.Y[(size_t)(m + 1) * p.N + row] = __float2bfloat16_rn(sum[1]);
    }
  }

  // ---- the cluster's CTAs hold the sums over their slices of K: added in rank order, a share of the outputs per
  // CTA.  A warp reads the sixteen rows of two tokens, two runs of 64 bytes, from each: with a row's tokens side by side a warp's
  // reads fell into 32 pieces, and the pass took 2900 cycles for 256 rows of 16 tokens.
  if (p.cshift) {
    __syncwarp();
    cluster_sync_shared();
    const int csize = 1 << p.cshift;
    const uint32_t ysum = smem_u32(ywhole);
#pragma unroll 1
    for (int idx = (int)threadIdx.x + rank * kPThreads; idx < npairs * 16 * p.M; idx += csize * kPThreads) {
      const int lr = idx & 15, lp = quotient(idx >> 4, p.m_magic[0]), m = (idx >> 4) - lp * p.M;
      if (!pair_full(lp) && lr >= 8) continue;
      const uint32_t at = ysum + (uint32_t)((lp * pair_floats + sum_at(m, lr)) * 4);
      float sum = 0.0f;
#pragma unroll 1
      for (int rh = 0; rh < csize; rh += 4) {
        float v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = rh + r < csize ? ld_cluster_f32(mapa_shared(at, (uint32_t)(rh + r))) : 0.0f;
#pragma unroll
        for (int r = 0; r < 4; ++r) sum += v[r];
      }
      p.Y[(size_t)m * p.N + pair_rg(lp) * 8 + lr] = __float2bfloat16_rn(sum);
    }
    __syncwarp();
    cluster_sync_reads();     // the sums are read by the whole cluster until here
  }

  if (abort_flag[0]) {
    // let copies already in flight land before shared memory is released
#pragma unroll 1
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncthreads();
    if (threadIdx.x == 0) {
      atomicExch(p.status, (int)PEQA_ERR_DEVICE_TIMEOUT);
      p.status[1] = (int)blockIdx.x;
    }
  }
}

// ------------------------------------------------------------- prepare / unprepare
// One thread per (row group, step, lane, string): moves the string's 32 codes between the
// two layouts.  TO_PREPARED: canonical -> prepared, else the inverse.
template <int BITS, bool TO_PREPARED>
__global__ void prep_layout_kernel(const uint32_t* __restrict__ src, uint32_t* __restrict__ dst,
                                   int N, int K, int T) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int rgs = N / 8, rgs2 = (rgs + 1) & ~1;      // the buffer holds whole pairs of row groups
  const size_t total = (size_t)rgs2 * T * 128;
  if (idx >= total) return;
  const int s = (int)(idx & 3), lane = (int)((idx >> 2) & 31);
  const size_t rt = idx >> 7;
  const int t = (int)(rt % T), rg = (int)(rt / T);
  const size_t blk = ((size_t)(rg >> 1) * T + t) * 2 + (rg & 1);
  const int r8 = lane >> 2, c4 = lane & 3;
  const int row = rg * 8 + r8;
  // word e of string s of this lane: word index wi = s*BITS + e of the lane's 4*BITS words
  auto prep_word = [&](int e) -> size_t {
    const int wi = s * BITS + e;
    const int c = wi >> 2, wo = wi & 3;
    return ((blk * BITS + c) * 32 + lane) * 4 + wo;
  };
  if (rg >= rgs) {                                   // the missing half of the last pair
    if (TO_PREPARED) {
#pragma unroll
      for (int e = 0; e < BITS; ++e) dst[prep_word(e)] = 0u;
    }
    return;
  }
  const int wpr = K * BITS / 32;
  const uint32_t* canon_r = (TO_PREPARED ? src : dst) + (size_t)row * wpr;
  uint32_t* canon_w = dst + (size_t)row * wpr;
  // code of column j of a canonical row
  auto canon_get = [&](int j) -> uint32_t {
    const int bit = j * BITS;
    uint32_t v = canon_r[bit >> 5] >> (bit & 31);
    if ((bit & 31) + BITS > 32) v |= canon_r[(bit >> 5) + 1] << (32 - (bit & 31));
    return v & ((1u << BITS) - 1u);
  };
  uint32_t str[BITS];
#pragma unroll
  for (int e = 0; e < BITS; ++e) str[e] = TO_PREPARED ? 0u : src[prep_word(e)];
  auto str_get = [&](int pos) -> uint32_t {
    const int bit = pos * BITS;
    uint32_t v = str[bit >> 5] >> (bit & 31);
    if ((bit & 31) + BITS > 32) v |= str[(bit >> 5) + 1] << (32 - (bit & 31));
    return v & ((1u << BITS) - 1u);
  };
  auto str_put = [&](int pos, uint32_t code) {
    const int bit = pos * BITS;
    str[bit >> 5] |= code << (bit & 31);
    if ((bit & 31) + BITS > 32) str[(bit >> 5) + 1] |= code >> (32 - (bit & 31));
  };
  if (TO_PREPARED) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int cs = 2 * k + h;
        const int col = t * kStepCols + 32 * (4 * s + (cs >> 3)) + 8 * c4 + (cs & 7);
        const uint32_t code = col < K ? canon_get(col) : 0u;
        str_put(h ? dq::stream_hi(BITS, k) : dq::stream_lo(BITS, k), code);
      }
    }
#pragma unroll
    for (int e = 0; e < BITS; ++e) dst[prep_word(e)] = str[e];
  } else {
    // the eight columns of a run this lane owns are BITS whole bytes of the canonical row
    uint8_t* rowb = reinterpret_cast<uint8_t*>(canon_w);
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
      const int col = t * kStepCols + 32 * (4 * s + rr) + 8 * c4;
      if (col >= K) continue;
      uint32_t bits8 = 0u;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int cs = 8 * rr + e, k = cs >> 1;
        const uint32_t code = str_get((cs & 1) ? dq::stream_hi(BITS, k) : dq::stream_lo(BITS, k));
        bits8 |= code << (BITS * e);
      }
      uint8_t* o = rowb + (size_t)col * BITS / 8;
#pragma unroll
      for (int b = 0; b < BITS; ++b) o[b] = (uint8_t)(bits8 >> (8 * b));
    }
  }
}

struct PrepPlan {
  int rg_per_cta, grid, T, spc, nchunks, slots, sps, x_pitch, pairs, cshift;
  bool i8;
  size_t smem;
  long long ns;      // estimated time
};

int x_pitch_for(int steps) {
  const int raw = steps * kStepCols * 2;
  return raw + 64;                                                // pitch % 128 == 64
}

// Chooses how many CTAs share a range of rows (each with a slice of K), how many steps of
// activations are staged at a time and the shape of the warps' rings.  gcols: columns of one
// quantization group.
//
// One CTA per range needs no exchange of sums, but it stages all of its K: from five to eight tokens
// on, the activations do not fit beside the rings, and working through K in chunks costs a
// staging, a parking and a reduce per chunk.  A cluster of 2, 4 or 8 CTAs stages a slice each and
// adds its sums up through distributed shared memory.  Before / after, 3-bit: 16 tokens at 8192 x 8192 36 / 19 us, at
// 22016 x 8192 65 / 50, in groups of 64 at 8192 x 8192 97 / 28.
//
// The estimate, in ns: 2330 a launch; a step of a pair, per turn of the busiest warp, 1440 (2120 with groups inside the step, 9 % more
// where these have little L1, 25 with a table per task, whose tokens read scales of their own each; 13 % less with two token
// tiles; integer kernel 1180 and 1360; canonical rows 330 more); staging a token's step 31, 63 in the integer kernel, 91 from canonical
// rows, whose order takes the activations in half sectors; 2.4 per row group, token and chunk for the final pass, 3.6 where a
// cluster shares it, and 370 for the cluster's exchange, 170 more for each doubling; 5500 per further chunk; 10000 more for a
// second wave of clusters.  The constants are those that choose best, not each what its part was measured to take (nine of ten
// estimates are 0.7 to 1.2 of the time): over 942 random calls (1 to 16 tokens, prepared, of several tasks and canonical), each timed
// with clusters of 1, 2, 4 and 8, one wave and two, as one launch and as two where these fit, the choice costs 0.45 % more
// than the best on average, 12 % at worst.  (Turns are counted chunk by chunk, since each chunk is dealt to the warps anew: with
// the steps of all chunks dealt out once, nine chunks of five steps counted as ten turns instead of eighteen, and 13 tokens of 4-bit
// weights took one launch where two are faster, us: 8192 x 22016 in groups of 128 99 / 56, 8192 x 16384 in groups of 64 82 / 51.)
//
// tasks: a table per task.  (With 9 % for it too, eight tokens at 17128 x 11904 in groups of 64, 3 bits, took 163 us on two CTAs a
// range, whose rings leave 28 KB of L1, where four a range take 87.)
//
// i8 (one or two tokens): the plan of the integer kernel, whose activations take four bytes each and are all
// staged at once, at most four steps to a half-warp.
int plan_prep(int N, int K, int M, int bits, int gcols, bool canon, bool i8, bool tasks, PrepPlan* plan) {
  const int sms = sm_count_or(148);
  const int rgs = N / 8;
  const int NT = M <= 8 ? 1 : 2, TOKP = 8 * NT;
  const int step_bytes = canon ? 16 * (bits == 3 ? CanonRow<3>::pitch : CanonRow<4>::pitch) : 2 * bits * 512;
  const bool grouped = gcols < kStepCols;
  const int gps = grouped ? kStepCols / gcols : 0;
  // a chunk must lie inside one quantization group unless the groups are applied per step
  const int steps_per_group = grouped ? 1 : gcols / kStepCols;     // one group per row: >= T
  const bool one_group = gcols >= K;
  // clusters of 1, 2, 4, 8 CTAs that run at once (the larger ones leave SMs of a GPC idle)
  const int active[4] = {sms, sms / 2, sms * 33 / 148, sms * 15 / 148};
  auto pitch_for = [&](int spc) { return i8 ? spc * kStepCols + 64 : x_pitch_for(spc); };    // i8: of a digit
  plan->ns = -1;
  for (int ci = 0; ci < 4; ++ci)
    for (int waves = 1; waves <= (ci ? 2 : 1); ++waves) {
      PrepPlan c = {};
      c.cshift = ci;
      c.T = (K + kStepCols - 1) / kStepCols;
      if (ci > 0 && (c.T < (1 << ci) || active[ci] < 1 || !(grouped || one_group))) continue;
      const int Tl = (c.T + (1 << ci) - 1) >> ci;                     // most steps of a CTA
      c.rg_per_cta = (rgs + active[ci] * waves - 1) / (active[ci] * waves);
      c.grid = ((rgs + c.rg_per_cta - 1) / c.rg_per_cta) << ci;
      // a range that starts and ends at an odd row group holds the most pairs
      c.pairs = c.rg_per_cta / 2 + 1;
      auto need = [&](int spc, int slots, int sps) -> size_t {
        const size_t sums = (size_t)pair_sums(M) * 4;                 // one pair's
        size_t b = 128 + kPHeadBytes + (kPWarps + c.pairs) * sums;
        if (spc < Tl) b += c.pairs * sums;
        b += (size_t)((c.pairs + 3) & ~3) * 4 + (size_t)c.pairs * 16 * 8;
        b += ((grouped ? (size_t)spc * gps * TOKP : 0) + (i8 ? 2 * kI8Units : 2 * kPWarps)) * 4 + 128;
        b += (((size_t)M * (i8 ? 4 : 1) * pitch_for(spc)) + 127) / 128 * 128;
        b += (size_t)kPWarps * slots * sps * step_bytes;
        return b;
      };
      // ring shapes in order of preference: bytes in flight first, larger copies on a tie
      const int shapes[4][2] = {{2, 2}, {4, 1}, {3, 1}, {2, 1}};   // {slots, steps per slot}
      // all of the CTA's K staged at once, with the best ring that fits, groups inside the step: that fits and leaves L1 60 KB
      // instead of 28, which is what it has from 195 KB of shared memory on.  A row's scales are read a vector a step and found there again (us, all /
      // this: eight tokens of several tasks, 8192 x 8192 in groups of 64 24.4 / 21.0, seven, 4096 x 11008 in groups of
      // 128 17.5 / 14.5; one token, 8192 x 22016 in groups of 64 23.3 / 22.2) ...
      if ((grouped || one_group) && (!i8 || M * Tl <= kI8Units)) {
        for (int i = grouped ? 0 : 4; i < 8 && c.spc == 0; ++i) {
          const int slots = shapes[i & 3][0], sps = shapes[i & 3][1];
          if (canon && sps > 1) continue;
          if (need(Tl, slots, sps) <= (size_t)(i < 4 ? kPSmemL1 : kPSmemLimit)) {
            c.spc = Tl;
            c.slots = slots;
            c.sps = sps;
          }
        }
      }
      // ... else (one CTA per range) the largest chunk of steps beside a ring of two single steps
      if (c.spc == 0 && ci == 0 && !i8) {
        for (int spc = c.T; spc >= 1 && c.spc == 0; --spc) {
          if (!grouped && !one_group && (steps_per_group % spc) != 0) continue;
          if (need(spc, 2, 1) <= (size_t)kPSmemLimit) {
            c.spc = spc;
            c.slots = 2;
            c.sps = 1;
          }
        }
      }
      if (c.spc == 0) continue;
      c.nchunks = (Tl + c.spc - 1) / c.spc;
      c.x_pitch = pitch_for(c.spc);
      c.i8 = i8;
      c.smem = need(c.spc, c.slots, c.sps);
      auto turns = [&](int spc) { return (((long long)c.rg_per_cta * spc + 1) / 2 + kPWarps - 1) / kPWarps; };
      const long long all_turns = Tl / c.spc * turns(c.spc) + turns(Tl % c.spc);
      long long per_step = (i8 ? (grouped ? 1360 : 1180) : (grouped ? 2120 : 1440) * (NT == 2 ? 87 : 100) / 100) + (canon ? 330 : 0);
      if (grouped && c.smem > (size_t)kPSmemL1) per_step = per_step * (tasks && !i8 ? 125 : 109) / 100;
      const long long per_unit = canon ? 91 : i8 ? 63 : 31;
      c.ns = waves * (2330 + all_turns * per_step + (long long)M * Tl * per_unit +
                      (long long)c.rg_per_cta * M * c.nchunks * (ci ? 36 : 24) / 10 + (ci ? 370 + 170 * ci : 0) + (c.nchunks - 1) * 5500) +
             (waves - 1) * 10000;
      if (plan->ns < 0 || c.ns < plan->ns) *plan = c;
    }
  return plan->ns < 0 ? PEQA_ERR_TOO_LARGE : PEQA_OK;
}

template <int BITS, int NT, int GSH, bool TASKS, bool CANON, bool I8, int V>
int launch_prep_t(const PrepParams& p, int grid, size_t smem, cudaStream_t st) {
  auto kern = decode_prep_kernel<BITS, NT, GSH, TASKS, CANON, I8, V>;
  static std::atomic<uint64_t> done{0};
  PEQA_TRY(allow_smem(kern, kPSmemLimit, done));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(kPThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1 << p.cshift;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.cshift ? 2 : 1;
  PEQA_CUDA(cudaLaunchKernelEx(&cfg, kern, p));
  return PEQA_OK;
}

template <int BITS, int NT, bool TASKS, bool CANON, bool I8>
int launch_prep_g(const PrepParams& p, int gsh, int grid, size_t smem, cudaStream_t st) {
  // A step holds 8, 4 or 2 groups of a row; vectors of them where every row's groups start on one and are whole ones
  // (a row of 11008 columns has 172 groups of 64 and 86 of 128).
  auto in_vectors = [&](int v) {
    return p.G % v == 0 && reinterpret_cast<uintptr_t>(p.scales) % (4 * v) == 0 && reinterpret_cast<uintptr_t>(p.zeros) % v == 0;
  };
  switch (gsh) {
    case 1:
      if constexpr (!CANON)
        return in_vectors(4) ? launch_prep_t<BITS, NT, 1, TASKS, CANON, I8, 4>(p, grid, smem, st)
                             : launch_prep_t<BITS, NT, 1, TASKS, CANON, I8, 1>(p, grid, smem, st);
      return PEQA_ERR_BAD_SHAPE;
    case 2:
      return in_vectors(4)   ? launch_prep_t<BITS, NT, 2, TASKS, CANON, I8, 4>(p, grid, smem, st)
             : in_vectors(2) ? launch_prep_t<BITS, NT, 2, TASKS, CANON, I8, 2>(p, grid, smem, st)
                             : launch_prep_t<BITS, NT, 2, TASKS, CANON, I8, 1>(p, grid, smem, st);
    case 3: return launch_prep_t<BITS, NT, 3, TASKS, CANON, I8, 1>(p, grid, smem, st);   // two groups a step
    default: return launch_prep_t<BITS, NT, 0, false, CANON, I8, 1>(p, grid, smem, st);   // tasks: looked up per row
  }
}

template <int BITS, bool CANON>
int launch_prep_b(const PrepParams& p, bool i8, int gsh, int grid, size_t smem, cudaStream_t st) {
  if constexpr (!CANON) {                              // (canonical rows: at most eight tokens, see decode_rows_supported)
    if (p.M > 8) return launch_prep_g<BITS, 2, false, false, false>(p, gsh, grid, smem, st);
    if (p.task_ids)
      return i8 ? launch_prep_g<BITS, 1, true, false, true>(p, gsh, grid, smem, st)
                : launch_prep_g<BITS, 1, true, false, false>(p, gsh, grid, smem, st);
  }
  return i8 ? launch_prep_g<BITS, 1, false, CANON, true>(p, gsh, grid, smem, st)
            : launch_prep_g<BITS, 1, false, CANON, false>(p, gsh, grid, smem, st);
}

int check_prep_layer(const peqa_qweight_t* w) {
  if (!w) return PEQA_ERR_NULL;
  PEQA_TRY(check_bits_shape(w->out_features, w->in_features, w->bits, w->group_size));
  if (w->in_features % 128 != 0 || w->out_features % 8 != 0) return PEQA_ERR_BAD_SHAPE;
  return PEQA_OK;
}

// Group sizes the prepared kernel serves: one group per row, groups that are multiples of
// 512 columns, and groups of 64, 128 or 256 columns.
bool prep_group_supported(int K, int g) {
  return g == K || g % kStepCols == 0 || g == 64 || g == 128 || g == 256;
}

// One launch over prepared or canonical weights, or (prepared ones) two of at most eight tokens each.
int run_decode(const peqa_qweight_t* w, const void* weights, bool canon, int g, const void* X, int M, void* Y,
               const float* scale_table, int n_tasks, const int32_t* task_ids, cudaStream_t st) {
  PrepPlan plan;
  bool two = false;
  // A row that is one group of 64, 128 or 256 columns is taken for one with groups inside the step, but for canonical rows with a
  // table per task: their instances look the table up where a row's sums are added, which is for one scale per row.
  const int gcols = canon && task_ids && g < kStepCols ? kStepCols : g;
  if (M > 8) {
    PrepPlan half;
    PEQA_TRY(plan_prep(w->out_features, w->in_features, (M + 1) / 2, w->bits, g, false, false, task_ids != nullptr, &half));
    two = task_ids || plan_prep(w->out_features, w->in_features, M, w->bits, g, false, false, false, &plan) != PEQA_OK ||
          2 * half.ns < plan.ns;
  } else if (M > 2 || plan_prep(w->out_features, w->in_features, M, w->bits, gcols, canon, true, task_ids != nullptr, &plan) != PEQA_OK) {
    PEQA_TRY(plan_prep(w->out_features, w->in_features, M, w->bits, gcols, canon, false, task_ids != nullptr, &plan));
  }
  if (two) {
    // Two launches of at most eight tokens each, the second of which finds the weights in L2: with a
    // table per task (the scales of four tokens per lane do not fit in registers), where all tokens
    // at once would be worked through in more chunks or waves, and where their parked sums leave no
    // room in shared memory (beside many columns, from about 105000 rows of 3-bit weights on for 16 tokens, 150000 for 12, 186000
    // for 9; of 4-bit weights, whose rings are larger, 70000, 103000 and 131000; with 512 columns about 1.9 times as many).
    const int h = (M + 1) / 2;
    const size_t K = (size_t)w->in_features, N = (size_t)w->out_features;
    PEQA_TRY(run_decode(w, weights, false, g, X, h, Y, scale_table, n_tasks, task_ids, st));
    return run_decode(w, weights, false, g, static_cast<const char*>(X) + (size_t)h * K * 2, M - h,
                      static_cast<char*>(Y) + (size_t)h * N * 2, scale_table, n_tasks,
                      task_ids ? task_ids + h : nullptr, st);
  }
  PrepParams p;
  p.P = static_cast<const uint8_t*>(weights);
  p.zeros = w->zeros;
  p.scales = task_ids ? scale_table : w->scales;
  p.X = static_cast<const __nv_bfloat16*>(X);
  p.Y = static_cast<__nv_bfloat16*>(Y);
  p.task_ids = task_ids;
  p.n_tasks = n_tasks;
  p.N = w->out_features;
  p.K = w->in_features;
  p.G = p.K / g;
  p.M = M;
  p.rgs = p.N / 8;
  p.rg_per_cta = plan.rg_per_cta;
  p.T = plan.T;
  p.spc = plan.spc;
  p.nchunks = plan.nchunks;
  p.slots = plan.slots;
  p.sps = plan.sps;
  p.x_pitch = plan.x_pitch;
  p.pairs_per_cta = plan.pairs;
  p.cshift = plan.cshift;
  p.row_bytes = p.K / 8 * w->bits;
  p.m_magic[0] = quotient_magic(M);
  p.m_magic[1] = quotient_magic((M + 1) / 2);
  PEQA_TRY(status_word(st, &p.status));
  const int gsh = gcols == 64 ? 1 : gcols == 128 ? 2 : gcols == 256 ? 3 : 0;
  if (canon)
    return w->bits == 3 ? launch_prep_b<3, true>(p, plan.i8, gsh, plan.grid, plan.smem, st)
                        : launch_prep_b<4, true>(p, plan.i8, gsh, plan.grid, plan.smem, st);
  return w->bits == 3 ? launch_prep_b<3, false>(p, plan.i8, gsh, plan.grid, plan.smem, st)
                      : launch_prep_b<4, false>(p, plan.i8, gsh, plan.grid, plan.smem, st);
}

}  // namespace

bool decode_rows_supported(const peqa_qweight_t* w, int g, int M) {
  PrepPlan plan;
  return M <= 8 && w->in_features % 128 == 0 && w->out_features % 8 == 0 && (g == w->in_features || g == 128 || g == 256) &&
         plan_prep(w->out_features, w->in_features, M, w->bits, g, true, false, false, &plan) == PEQA_OK;
}

int launch_decode_rows(const peqa_qweight_t* w, int g, const void* X, int M, void* Y, const float* scale_table,
                       int n_tasks, const int32_t* task_ids, cudaStream_t st) {
  // the instances of canonical rows have one token tile, and know a table per task with one scale per channel only
  if (M > 8 || (task_ids && g != w->in_features)) return PEQA_ERR_BAD_SHAPE;
  return run_decode(w, w->qweight, true, g, X, M, Y, scale_table, n_tasks, task_ids, st);
}

}  // namespace peqa

using namespace peqa;

extern "C" size_t peqa_decode_prepared_bytes(const peqa_qweight_t* w) {
  if (check_prep_layer(w) != PEQA_OK) return 0;
  const size_t T = ((size_t)w->in_features + kStepCols - 1) / kStepCols;
  const size_t rgs2 = ((size_t)w->out_features / 8 + 1) & ~(size_t)1;   // whole pairs of row groups
  return rgs2 * T * w->bits * 512;
}

static int run_layout(const peqa_qweight_t* w, const uint32_t* src, uint32_t* dst, bool to_prepared,
                      void* stream) {
  PEQA_TRY(check_prep_layer(w));
  if (!src || !dst) return PEQA_ERR_NULL;
  if (!aligned16(src) || !aligned16(dst)) return PEQA_ERR_ALIGNMENT;
  const int T = (w->in_features + kStepCols - 1) / kStepCols;
  const size_t n = (size_t)((w->out_features / 8 + 1) & ~1) * T * 128;
  const int threads = 256;
  const unsigned blocks = (unsigned)((n + threads - 1) / threads);
  cudaStream_t st = as_stream(stream);
  const int N = w->out_features, K = w->in_features;
  if (w->bits == 3) {
    if (to_prepared) prep_layout_kernel<3, true><<<blocks, threads, 0, st>>>(src, dst, N, K, T);
    else prep_layout_kernel<3, false><<<blocks, threads, 0, st>>>(src, dst, N, K, T);
  } else {
    if (to_prepared) prep_layout_kernel<4, true><<<blocks, threads, 0, st>>>(src, dst, N, K, T);
    else prep_layout_kernel<4, false><<<blocks, threads, 0, st>>>(src, dst, N, K, T);
  }
  PEQA_CUDA(cudaGetLastError());
  return PEQA_OK;
}

extern "C" int peqa_decode_prepare(const peqa_qweight_t* w, uint32_t* prepared, void* stream) {
  if (!w || !w->qweight) return PEQA_ERR_NULL;
  return run_layout(w, w->qweight, prepared, true, stream);
}

extern "C" int peqa_decode_unprepare(const peqa_qweight_t* w, const uint32_t* prepared,
                                     uint32_t* qweight_out, void* stream) {
  return run_layout(w, prepared, qweight_out, false, stream);
}

extern "C" int peqa_qlinear_decode_prepared(const peqa_qweight_t* w, const uint32_t* prepared,
                                            const void* X, int M, void* Y,
                                            const float* scale_table, int n_tasks,
                                            const int32_t* task_ids, void* stream) {
  PEQA_TRY(check_prep_layer(w));
  if (!prepared || !X || !Y || !w->zeros) return PEQA_ERR_NULL;
  const int g = effective_group(w->in_features, w->group_size);
  if (!prep_group_supported(w->in_features, g)) return PEQA_ERR_BAD_SHAPE;
  if (M < 1 || M > 16) return PEQA_ERR_BAD_SHAPE;
  if (task_ids) {
    if (!scale_table) return PEQA_ERR_NULL;
    if (n_tasks < 1) return PEQA_ERR_BAD_SHAPE;
  } else if (!w->scales) {
    return PEQA_ERR_NULL;
  }
  if (!aligned16(prepared) || !aligned16(X) || !aligned16(Y)) return PEQA_ERR_ALIGNMENT;
  PEQA_TRY(check_arch());
  return run_decode(w, prepared, false, g, X, M, Y, scale_table, n_tasks, task_ids, as_stream(stream));
}
