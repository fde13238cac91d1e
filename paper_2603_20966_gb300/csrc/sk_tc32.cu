// sk_tc32.cu -- FP32 form of the left sketch Y[k x n] = S[k x m] A[m x n] on
// the tensor cores (tcgen05 + TMEM), every FP32 operand as the exact sum of
// three BF16 values.
//
// The local multiply of the paper's Alg. 1 with the random operand
// regenerated tile by tile, as k_sketch_fp32_simt does it on the CUDA cores.
// Those are what bounded that kernel: it reached half of their 80 TFLOP/s,
// and its 128 x 256 tiles cover a 333-column A to 65 %.  A 24-bit significand
// splits without error into three of 8 bits, x = x1 + x2 + x3 (round to
// nearest each time), and of the nine products of two such sums six carry
// everything above 2^-24 of the whole:
//   main   s1 a1
//   cross  s1 a2 + s2 a1 + s2 a2 + s1 a3 + s3 a1
// each exact in the tensor core, summed in FP32.  The tensor core truncates
// where an FMA rounds, which shrinks a sum by about 2^-26 per K step, so the
// two groups have accumulators of their own (the cross terms are 2^-8 of the
// main ones, and so is what they lose): the main one is a chain of at most
// 6 or 8 stages that is added, with IEEE adds, to the ones before it, the
// cross one is added with every chain that ends 128 stages or so.  A
// Rademacher S is exact in one BF16 value: s1 a1, then s1 a2 + s1 a3.
// The parts of an element below 2^-110 reach into BF16's subnormals and lose
// bits.  A column whose elements are all small in an item is therefore
// multiplied by 2^48 on the way in and by 2^-48 on the way out (exact); which
// columns these are is known when the item has been read, so such items run a
// second time at the end.
//
// A CTA owns a 128 x NT tile of Y (NT <= 256: two accumulators of NT TMEM
// columns) and a list of (tile, split of m) items:
//   warp 0       TMEM allocation, MMA issuer: per stage of 32 rows of m
//                2 K steps x 6 (3) tcgen05.mma kind::f16, M = 128, N = NT;
//   warps 1-4    epilogue: a finished chain leaves TMEM (the item's last one
//                with the cross sums) through staging tiles and the TMA for
//                the item's FP32 partial (store, later chains add);
//   warps 5-20   workers, two groups of 8 that take turns on stages: load the
//                stage's rows of A (any alignment), generate the S tile while
//                they arrive, split both into their operand layouts.
// The workers bound it: 4096 generated entries and 32 NT split elements per
// stage keep the issue slots 56 % busy, the MMAs the tensor pipe 23 %.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "sk_internal.h"
#include "sk_rng.cuh"
#include "sk_tc.cuh"

namespace sk {
namespace {

using namespace tc;

constexpr int BM = 128;      // rows of S per tile
constexpr int SL = 32;       // rows of m per stage
constexpr int SLOTS = 3;     // stages in the ring
constexpr int NCH = 4;       // most 64-column chunks of a tile
// Most stages per chain of the main accumulator: 192 rows of m, 256 from
// kLongRows on (Rademacher products are BF16 values and truncate less: 1024).
// Longer chains are faster and truncate more; these stay at half the error of
// the CUDA cores' form.  With chains of 4, 6, 8, 10 stages and there (Gaussian
// S, n = 512, k = 2048):
//   4096 rows    1.4, 1.7, 1.7, 3.0e-7, there 3.3e-7    126, 107, 107, 93 us
//   8192 rows    1.5, 1.6, 2.1, 2.8e-7, there 4.6e-7    208, 190, 175, 163 us
//   16384 rows   1.5, 2.0, 2.4, 2.9e-7, there 6.4e-7    396, 353, 318, 303 us
//   65536 rows   1.9, 2.2, 2.6, 3.1e-7, there 12.6e-7   1.45, 1.29, 1.20, 1.14 ms
constexpr int CHAIN = 6, CHAIN_LONG = 8, CHAIN_R = 32;
// Stages after which the cross accumulator is read out with the chain that
// ends there and starts again.  What it loses grows with its length: never
// read out before an item's end, one split of 2^18, 2^20 and 2^22 rows had
// errors of 3.6e-6, 1.4e-5 and 5.7e-5 (Gaussian S; the CUDA cores 6.5e-6,
// 1.3e-5 and 2.6e-5), with this 6.2e-7, 1.2e-6 and 2.3e-6.  32 and 64 stages
// have the same errors and cost up to 1 %, 128 cost 0.2 %.
constexpr int CROSS = 128;
constexpr int64_t kLongRows = 16384;  // rows of m from which chains are CHAIN_LONG
constexpr int N_EPI = 4;
constexpr int GROUPS = 2, GROUP_WARPS = 8;
constexpr int W_EPI0 = 1, W_WORK0 = W_EPI0 + N_EPI;
constexpr int THREADS = 32 * (W_WORK0 + GROUPS * GROUP_WARPS);

// Slot of a stage: the parts of S (K-major core matrices without swizzle, two
// slabs of 16 columns each), then those of A (MN-major with the 128-byte
// swizzle: chunks of 64 columns x 32 rows).
constexpr uint32_t S_SLAB = BM * 16 * 2;        // 4096
constexpr uint32_t S_PART = 2 * S_SLAB;         // 8192
constexpr uint32_t A_CHUNK = SL * 64 * 2;       // 4096
constexpr uint32_t OFF_A = 3 * S_PART;
constexpr uint32_t SLOT_MAX = OFF_A + 3 * NCH * A_CHUNK;
// Staging tile of a drain: 32 rows x 16 columns with the 64-byte swizzle
// (4-column unit u of row r at u ^ (r / 2 mod 4)).  Behind the ring an
// epilogue warp has one, or four where tiles of fewer columns leave room.
constexpr uint32_t EPI_TILE = 32 * 16 * 4;
constexpr uint32_t OFF_BAR = SLOTS * SLOT_MAX + N_EPI * EPI_TILE;
constexpr uint32_t NUM_BARS = 2 * SLOTS + 3;
constexpr uint32_t OFF_MISC = OFF_BAR + NUM_BARS * 8;  // abort flag, TMEM slot
constexpr uint32_t OFF_SEEN = OFF_MISC + 16;           // column flags (Seen)
constexpr int SEEN = 4;         // items whose flags are kept at a time
constexpr int REDO_BITS = 512;  // items (modulo this) that run a second time
struct Seen {
  // columns 64 c + 2 l + x of an item's tile as bit l of word 2 c + x
  uint32_t normal[SEEN][2 * NCH];  // a warp that met small elements saw one of kSmall or more
  uint32_t small[SEEN][2 * NCH];   // a warp saw smaller ones (not zeros) and none of those
  uint32_t all[SEEN];              // a warp saw one of kSmall or more in every column
  uint32_t redo[REDO_BITS / 32];   // items with columns that may be small all through,
  uint32_t any_redo;               // and whether there are any
  uint32_t scaled[2 * NCH];        // columns that the second run multiplies by kUp
};
constexpr uint32_t SMEM = OFF_SEEN + sizeof(Seen) + 1024;  // + slack for 1 KB alignment
static_assert(SMEM <= 227 * 1024, "shared memory budget");
static_assert(SLOT_MAX % 1024 == 0 && OFF_A % 1024 == 0, "swizzle atoms on 1 KB boundaries");
static_assert(SLOTS * (SLOT_MAX - 3 * A_CHUNK) + N_EPI * 4 * EPI_TILE <= OFF_BAR, "staging tiles");
static_assert(GROUPS <= SLOTS, "worker groups vs ring depth");

// |a| above this rounds to an infinite BF16; such a value is truncated.
constexpr float kRoundsToInf = 0x1.fep127f;
// Magnitudes from 2^-110 on split without error.  A column of an item with
// none of at least kSmall runs again, times kUp: its elements are then below
// 2^-52 and the smallest subnormal at 2^-101.  (In a column with one, what the
// others lose is below 2^-33 of it.)
constexpr float kSmall = 0x1p-100f;
constexpr float kUp = 0x1p48f, kDown = 0x1p-48f;

struct F32Params {
  const float* A;
  int64_t lda;
  float* part;  // partials [splits][P][ldp]
  int64_t P, Q, L, ldp;
  int64_t chunk;  // contracted length per split (a multiple of SL)
  int tiles_p, tiles_q, nitems;
  int nt;     // columns per tile, a multiple of 64
  int chain;  // stages per accumulation chain
  int cross;  // chains per accumulation of the cross terms
  int vec2;   // rows of A on 8-byte boundaries
  PhiloxRoundKeys rk;
  int* status;
  uint64_t timeout_ns;
  // failure-injection hook of the tests, -1 otherwise: this stage (counted over
  // a block's items) is never handed to the MMA issuer
  int64_t stall_stage;
};

struct Item {
  int64_t p0, q0, lbeg, lend;
  int z, nsteps, nchains;
};

__device__ __forceinline__ Item get_item(const F32Params& p, int idx) {
  Item it;
  const int t = idx / p.tiles_p;
  it.p0 = static_cast<int64_t>(idx - t * p.tiles_p) * BM;
  it.q0 = static_cast<int64_t>(t % p.tiles_q) * p.nt;
  it.z = t / p.tiles_q;
  it.lbeg = static_cast<int64_t>(it.z) * p.chunk;
  it.lend = min(p.L, it.lbeg + p.chunk);
  it.nsteps = static_cast<int>((it.lend - it.lbeg + SL - 1) / SL);
  it.nchains = (it.nsteps + p.chain - 1) / p.chain;
  return it;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo_elem, float hi_elem) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo_elem, hi_elem);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float2 unpack_bf16(uint32_t w) {
  return f2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
// x minus the BF16 values packed in w (exact: both have at most 24 bits and
// the difference fits)
__device__ __forceinline__ float2 minus_bf16(float2 x, uint32_t w) {
  return __ffma2_rn(unpack_bf16(w), f2(-1.0f, -1.0f), x);
}

// The two elements of x as sums of three BF16 values, packed by part.
// HUGE_OK: elements that would round to infinity are truncated.
template <bool HUGE_OK>
__device__ __forceinline__ void split3(float2 x, uint32_t (&w)[3]) {
  w[0] = pack_bf16(x.x, x.y);
  if (HUGE_OK) {
    if (fabsf(x.x) >= kRoundsToInf && !isinf(x.x))
      w[0] = (w[0] & 0xffff0000u) | (__float_as_uint(x.x) >> 16);
    if (fabsf(x.y) >= kRoundsToInf && !isinf(x.y))
      w[0] = (w[0] & 0x0000ffffu) | (__float_as_uint(x.y) & 0xffff0000u);
  }
  const float2 r = minus_bf16(x, w[0]);
  w[1] = pack_bf16(r.x, r.y);
  const float2 q = minus_bf16(r, w[1]);
  w[2] = pack_bf16(q.x, q.y);
}

// The columns of an item (`rows` rows of its tile of A) that hold small
// elements and no others, as bits of seen->scaled; whether there are any.  By
// all threads of the block, with the ring idle.
__device__ __noinline__ bool find_small_columns(const float* A, int64_t lda, int64_t rows,
                                                int ncols, Seen* seen, uint32_t* colmax) {
  const int tid = static_cast<int>(threadIdx.x), lane = tid & 31, warp = tid >> 5;
  for (int c = tid; c < 64 * NCH; c += THREADS) colmax[c] = 0u;
  if (tid < 2 * NCH) seen->scaled[tid] = 0u;
  __syncthreads();
  for (int c = lane; c < ncols; c += 32) {
    uint32_t mx = 0u;  // magnitudes order as their bits do (NaN above all)
#pragma unroll 4
    for (int64_t l = warp; l < rows; l += THREADS / 32)
      mx = max(mx, __float_as_uint(A[l * lda + c]) & 0x7fffffffu);
    atomicMax(colmax + c, mx);
  }
  __syncthreads();
  bool any = false;
  if (tid < ncols && colmax[tid] != 0u && colmax[tid] < __float_as_uint(kSmall)) {
    any = true;
    atomicOr(seen->scaled + 2 * (tid >> 6) + (tid & 1), 1u << ((tid & 63) >> 1));
  }
  return __syncthreads_or(any) != 0;
}

// What a warp has to find out about the columns of an item: nothing (any more),
// whether any holds small elements, or first whether all of them are normal.
constexpr int kLookNone = 0, kLookSmall = 1, kLookFirst = 2;

// Two rows of an item show these magnitudes (the larger of the two) in this
// lane's columns; the flags of column i = 2 c + x are bits i (a normal element)
// and 8 + i (any but zeros) of `cols`.  Dense data of ordinary size is done
// with after the first rows; without small elements the others cost a
// comparison.
__device__ __forceinline__ int look_at_columns(const float2 (&mx)[NCH], int nconv, int look,
                                               uint32_t* cols, uint32_t* all) {
  if (look == kLookFirst) {
    float least = kSmall;
#pragma unroll
    for (int c = 0; c < NCH; ++c)
      if (c < nconv) least = fminf(least, fminf(mx[c].x, mx[c].y));
    if (__all_sync(0xffffffffu, least >= kSmall)) {
      *all = 1u;
      return kLookNone;
    }
  }
  uint32_t low = 0xffffffffu;  // zeros wrap around to the largest number
#pragma unroll
  for (int c = 0; c < NCH; ++c)
    low = min(low, min(__float_as_uint(mx[c].x) - 1u, __float_as_uint(mx[c].y) - 1u));
  if (__any_sync(0xffffffffu, low < __float_as_uint(kSmall) - 1u)) {
#pragma unroll
    for (int i = 0; i < 2 * NCH; ++i) {
      const float m = i & 1 ? mx[i >> 1].y : mx[i >> 1].x;
      if (m >= kSmall) *cols |= 1u << i;
      if (m > 0.0f) *cols |= 0x100u << i;
    }
  }
  return kLookSmall;
}

// A warp's flags of an item, for the epilogue.
__device__ __noinline__ void publish_columns(uint32_t cols, uint32_t* normal, uint32_t* small) {
  for (int i = 0; i < 2 * NCH; ++i) {
    const uint32_t n = __ballot_sync(0xffffffffu, (cols >> i) & 1u);
    const uint32_t z = __ballot_sync(0xffffffffu, (cols >> (8 + i)) & 1u) & ~n;
    if ((threadIdx.x & 31) == 0) {
      if (n) atomicOr(normal + i, n);
      if (z) atomicOr(small + i, z);
    }
  }
}

// The roles of a block's warps over its items first_item, + item_step, ... below
// end_item, after `runs` calls and in them g stages, gc chains and j items.
// AGAIN: items with columns to scale.
template <int DIST, bool AGAIN>
__device__ __forceinline__ void run_items(const CUtensorMap* pmap, const F32Params& p,
                                          uint8_t* smem, uint32_t tmem, int first_item,
                                          int item_step, int end_item, uint32_t runs, int g,
                                          int gc, int j) {
  constexpr int NS = DIST == kRademacher ? 1 : 3;  // parts of S
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + OFF_BAR;
  // full: a worker group has written the slot; empty: its MMAs have completed
  auto full = [&](int i) { return bar0 + 8u * i; };
  auto empty = [&](int i) { return bar0 + 8u * (SLOTS + i); };
  const uint32_t acc_full = bar0 + 8u * (2 * SLOTS);
  const uint32_t acc_empty = acc_full + 8u;
  const uint32_t drain_bar = acc_full + 16u;
  // flags of the last four items: the workers are at most three stages, hence
  // three items, ahead of the epilogue
  Seen* seen = reinterpret_cast<Seen*>(smem + OFF_SEEN);
  const Abort ab{reinterpret_cast<volatile int*>(smem + OFF_MISC), p.status, p.timeout_ns};
  const int warp = uniform(static_cast<int>(threadIdx.x >> 5));
  const int lane = threadIdx.x & 31;
  const uint32_t a_part = static_cast<uint32_t>(p.nt / 64) * A_CHUNK;  // one part of A in a slot
  const uint32_t slot_bytes = OFF_A + 3u * a_part;

  if (warp == 0) {  // the whole warp; one lane issues
    const uint32_t el = elect_one();
    const uint32_t idesc =
        idesc_bf16_f32(BM, static_cast<uint32_t>(p.nt)) | (1u << 16);  // B is MN-major
    const uint64_t a_base = smem_desc(sbase, 128u, 256u);
    const uint64_t b_base = smem_desc_sw128(sbase + OFF_A, A_CHUNK, 1024u);
    bool stop = false;
    for (int idx = first_item; idx < end_item && !stop; idx += item_step, ++j) {
      const int nsteps = get_item(p, idx).nsteps;
      int in_chain = 0, in_cross = 0;  // stages of the chain, chains of the cross terms so far
      for (int s = 0; s < nsteps; ++s, ++g) {
        const int so = g % SLOTS;
        if (in_chain == 0 && gc > 0) {
          // every epilogue warp has read the last chain (and its item's flags)
          if (!mbar_wait_warp(acc_empty, (gc - 1) & 1, ab, 0x25, gc)) {
            stop = true;
            break;
          }
          if (s == 0) {
            const int e = (j - 1) % SEEN;
            if (lane < 2 * NCH) seen->normal[e][lane] = seen->small[e][lane] = 0u;
            if (lane == 0) seen->all[e] = 0u;
          }
          __syncwarp();
        }
        if (!mbar_wait_warp(full(so), (g / SLOTS) & 1, ab, 0x22, g)) {
          stop = true;
          break;
        }
        tc_fence_after();
        // offsets are multiples of 16 B below 256 KB: added to the low word
        const uint64_t a0 = a_base + ((static_cast<uint32_t>(so) * slot_bytes) >> 4);
        const uint64_t b0 = b_base + ((static_cast<uint32_t>(so) * slot_bytes) >> 4);
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          auto mma = [&](int sp, int ap, uint32_t col, uint32_t acc) {
            mma_bf16(tmem + col, a0 + ((sp * S_PART + ks * S_SLAB) >> 4),
                     b0 + ((static_cast<uint32_t>(ap) * a_part + ks * 2048u) >> 4), idesc, acc, el);
          };
          mma(0, 0, 0u, in_chain > 0 || ks > 0 ? 1u : 0u);
          mma(0, 1, 256u, in_chain > 0 || in_cross > 0 || ks > 0 ? 1u : 0u);
          mma(0, 2, 256u, 1u);
          if (NS == 3) {
            mma(1, 0, 256u, 1u);
            mma(1, 1, 256u, 1u);
            mma(2, 0, 256u, 1u);
          }
        }
        mma_commit(empty(so), el);
        if (++in_chain == p.chain || s == nsteps - 1) {
          mma_commit(acc_full, el);
          in_chain = 0;
          if (++in_cross == p.cross) in_cross = 0;
          ++gc;
        }
      }
    }
    mma_commit(drain_bar, el);
    drain_wait(drain_bar, runs & 1, 200000000ull);
  } else if (warp < W_WORK0) {
    // ---- epilogue: lanes are accumulator rows, main in columns 0 .. nt - 1,
    // cross in 256 .. ----
    const int quarter = warp & 3;
    const int ntile = p.nt == 64 * NCH ? 1 : 4;
    uint8_t* tiles = smem + SLOTS * slot_bytes + (warp - W_EPI0) * ntile * EPI_TILE;
    const uint32_t usw = (static_cast<uint32_t>(lane) >> 1) & 3u;
    bool stop = false;
    for (int idx = first_item; idx < end_item && !stop; idx += item_step, ++j) {
      const Item it = get_item(p, idx);
      const int64_t r0 = it.p0 + quarter * 32;
      int in_cross = 0;
      for (int c0 = 0; c0 < it.nchains; ++c0, ++gc) {
        const bool ok = mbar_wait(acc_full, gc & 1, ab, 0x34, gc);
        if (!__all_sync(0xffffffffu, ok)) {
          stop = true;
          break;
        }
        tc_fence_after();
        const bool first = c0 == 0, last = c0 == it.nchains - 1;
        const bool with_cross = last || ++in_cross == p.cross;
        if (with_cross) in_cross = 0;
        // the earlier chains' adds have been performed: those of one element
        // stay in chain order
        if (lane == 0) bulk_wait<0>();
        __syncwarp();
        if (last && !AGAIN && warp == W_EPI0 && lane < 2 * NCH) {
          const volatile Seen* f = seen;
          const int e = j % SEEN;
          if (f->all[e] == 0u && (f->small[e][lane] & ~f->normal[e][lane]) != 0u) {
            atomicOr(seen->redo + (j % REDO_BITS) / 32, 1u << (j % 32));
            seen->any_redo = 1u;
          }
        }
        const int nchunk =
            r0 >= p.P ? 0
                      : static_cast<int>((min(static_cast<int64_t>(p.nt), p.Q - it.q0) + 31) / 32);
        int nb = 0;
        for (int ci = 0; ci < nchunk; ++ci) {
          uint32_t v[32], w[32];
          const uint32_t src =
              tmem + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(ci * 32);
          tmem_ld32(src, v);
          if (with_cross) {
            tmem_ld32(src + 256u, w);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              // the cross terms of an infinite or NaN element mean nothing:
              // the main sum is infinite or NaN already
              const float c = __uint_as_float(w[i]);
              if (fabsf(c) <= 0x1.fffffep127f)
                v[i] = __float_as_uint(__fadd_rn(__uint_as_float(v[i]), c));
            }
          } else {
            tmem_ld_wait();
          }
          if constexpr (AGAIN) {  // columns that were multiplied by kUp
            const uint32_t* m = seen->scaled + (ci >> 1) * 2;
            const uint32_t even = m[0] >> (16 * (ci & 1)), odd = m[1] >> (16 * (ci & 1));
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (((i & 1 ? odd : even) >> (i >> 1)) & 1u)
                v[i] = __float_as_uint(__fmul_rn(__uint_as_float(v[i]), kDown));
          }
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            const int64_t col = it.q0 + ci * 32 + 16 * half;
            if (col >= p.Q) break;
            if (nb >= ntile) {  // the TMA has read what the tile held before
              if (lane == 0) {
                if (ntile == 1)
                  bulk_wait_read<0>();
                else
                  bulk_wait_read<3>();
              }
              __syncwarp();
            }
            uint8_t* tile = tiles + (nb % ntile) * EPI_TILE;
            ++nb;
#pragma unroll
            for (int q = 0; q < 4; ++q)
              *reinterpret_cast<float4*>(tile + lane * 64 + ((static_cast<uint32_t>(q) ^ usw) << 4)) =
                  make_float4(__uint_as_float(v[16 * half + 4 * q]),
                              __uint_as_float(v[16 * half + 4 * q + 1]),
                              __uint_as_float(v[16 * half + 4 * q + 2]),
                              __uint_as_float(v[16 * half + 4 * q + 3]));
            fence_proxy_async_smem();  // the tile is read by the TMA
            __syncwarp();
            if (lane == 0) {
              if (first)
                tma_store_3d(pmap, smem_u32(tile), static_cast<int32_t>(col),
                             static_cast<int32_t>(r0), it.z);
              else
                tma_reduce_add_3d(pmap, smem_u32(tile), static_cast<int32_t>(col),
                                  static_cast<int32_t>(r0), it.z);
              bulk_commit();
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
      }
    }
    if (lane == 0) bulk_wait<0>();  // the last copies have completed
  } else {
    // ---- workers ----
    const int grp = (warp - W_WORK0) / GROUP_WARPS;
    const int w = (warp - W_WORK0) % GROUP_WARPS;
    // Gaussian and uniform tasks: quad qd of row rbase + 64 i in both slabs
    // (the lanes of a store phase write every bank once)
    const uint32_t qd = static_cast<uint32_t>(lane) >> 3;
    const uint32_t rbase = static_cast<uint32_t>(w * 8 + (lane & 7));
    const uint32_t s_off =
        (rbase & 7u) * 16u + (rbase >> 3) * 256u + (qd >> 1) * 128u + (qd & 1u) * 8u;
    bool stop = false;
    for (int idx = first_item; idx < end_item && !stop; idx += item_step, ++j) {
      const Item it = get_item(p, idx);
      const int g_item = g;
      int look = AGAIN ? kLookNone : kLookFirst;
      uint32_t cols = 0u;
      // columns of the tile: nfull whole chunks, then perhaps part of one,
      // where lanes past the last column read that one again (what they
      // contribute to is never read out)
      const int ncols = static_cast<int>(min(static_cast<int64_t>(p.nt), p.Q - it.q0));
      const int nfull = ncols / 64, nconv = (ncols + 63) / 64;
      const int edge0 = min(64 * nfull + 2 * lane, ncols - 1);
      const int edge1 = min(64 * nfull + 2 * lane + 1, ncols - 1);
      for (int s = (grp + GROUPS - g_item % GROUPS) % GROUPS; s < it.nsteps; s += GROUPS) {
        g = g_item + s;
        const int so = g % SLOTS;
        uint8_t* slot = smem + static_cast<uint32_t>(so) * slot_bytes;
        const int64_t cbase = it.lbeg + static_cast<int64_t>(s) * SL;
        bool ok = true;
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          // this warp's rows 16 half + 2 w, + 1 of the stage, columns 2 lane,
          // + 1 of each chunk, in flight while the S rows are generated
          // (ordinary loads: the kernel before this one may have written A while
          // this one was already resident)
          float2 x[2][NCH];
#pragma unroll
          for (int j2 = 0; j2 < 2; ++j2) {
            const int64_t l = cbase + 16 * half + 2 * w + j2;
            const float* row = p.A + l * p.lda + it.q0;
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
              x[j2][c] = f2(0.0f, 0.0f);
              if (l >= it.lend) continue;
              if (c < nfull) {
                const float* src = row + 2 * lane + 64 * c;
                if (p.vec2)
                  x[j2][c] = *reinterpret_cast<const float2*>(src);
                else
                  x[j2][c] = f2(src[0], src[1]);
              } else if (c < nconv) {
                x[j2][c] = f2(row[edge0], row[edge1]);
              }
            }
          }
          if (half == 0) {  // the MMAs that read the slot last time have completed
            ok = g < SLOTS || mbar_wait(empty(so), ((g / SLOTS) & 1) ^ 1, ab, 0x43, g);
            if (!__all_sync(0xffffffffu, ok)) break;
          }
          // S rows 64 half .. 64 half + 63 (those past P are never read out)
          if constexpr (DIST == kRademacher) {
            const int r = 64 * half + (w & 1) * 32 + lane;  // and 8 columns per warp pair
            if (it.p0 + r < p.P) {
              const int kc = w >> 1;
              const uint32_t c = static_cast<uint32_t>(cbase);
              const uint4 x4 = rademacher_bits(p.rk, static_cast<uint32_t>(it.p0 + r), c >> 7);
              const uint32_t ws = (c >> 5) & 3u;
              const uint32_t b = (ws == 0 ? x4.x : ws == 1 ? x4.y : ws == 2 ? x4.z : x4.w) >> (8 * kc);
              uint4 v;
              v.x = 0x3F803F80u | ((b & 1u) << 15) | ((b & 2u) << 30);
              v.y = 0x3F803F80u | ((b & 4u) << 13) | ((b & 8u) << 28);
              v.z = 0x3F803F80u | ((b & 16u) << 11) | ((b & 32u) << 26);
              v.w = 0x3F803F80u | ((b & 64u) << 9) | ((b & 128u) << 24);
              *reinterpret_cast<uint4*>(slot + (kc >> 1) * S_SLAB + (r & 7) * 16 + (r >> 3) * 256 +
                                        (kc & 1) * 128) = v;
            }
          } else {
            const int64_t grow = it.p0 + rbase + 64 * half;
            if (grow < p.P) {
              const PhiloxRow pr = philox_row(p.rk, static_cast<uint32_t>(grow));
              const uint32_t j0 = static_cast<uint32_t>(cbase >> 2) + qd;
#pragma unroll
              for (int slab = 0; slab < 2; ++slab) {
                const float4 v = entries4<DIST>(pr, philox_col(p.rk, j0 + 4u * slab), p.rk);
                uint32_t lo[3], hi[3];
                split3<false>(f2(v.x, v.y), lo);
                split3<false>(f2(v.z, v.w), hi);
#pragma unroll
                for (int pt = 0; pt < 3; ++pt)
                  *reinterpret_cast<uint2*>(slot + pt * S_PART + slab * S_SLAB + half * 2048 +
                                            s_off) = make_uint2(lo[pt], hi[pt]);
              }
            }
          }
          if constexpr (AGAIN) {
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
              const float2 up = f2((seen->scaled[2 * c] >> lane) & 1u ? kUp : 1.0f,
                                   (seen->scaled[2 * c + 1] >> lane) & 1u ? kUp : 1.0f);
#pragma unroll
              for (int j2 = 0; j2 < 2; ++j2) x[j2][c] = __fmul2_rn(x[j2][c], up);
            }
          }
          float2 mx[NCH];
          float hmax = 0.0f;
#pragma unroll
          for (int c = 0; c < NCH; ++c) {
            mx[c] = f2(fmaxf(fabsf(x[0][c].x), fabsf(x[1][c].x)),
                       fmaxf(fabsf(x[0][c].y), fabsf(x[1][c].y)));
            hmax = fmaxf(hmax, fmaxf(mx[c].x, mx[c].y));
          }
          if (look != kLookNone)
            look = look_at_columns(mx, nconv, look, &cols, seen->all + j % SEEN);
          auto store = [&](auto huge) {
#pragma unroll
            for (int j2 = 0; j2 < 2; ++j2) {
              const int r = 16 * half + 2 * w + j2;
              uint8_t* dst =
                  slot + OFF_A + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + ((lane & 3) << 2);
#pragma unroll
              for (int c = 0; c < NCH; ++c) {
                if (c >= nconv) break;
                uint32_t q[3];
                split3<decltype(huge)::value>(x[j2][c], q);
#pragma unroll
                for (int pt = 0; pt < 3; ++pt)
                  *reinterpret_cast<uint32_t*>(dst + pt * a_part + c * A_CHUNK) = q[pt];
              }
            }
          };
          if (hmax >= kRoundsToInf)
            store(std::true_type{});
          else
            store(std::false_type{});
        }
        if (!__all_sync(0xffffffffu, ok)) {
          stop = true;
          break;
        }
        // (the group's last stage of the item)
        if (s + GROUPS >= it.nsteps && __any_sync(0xffffffffu, cols != 0u))
          publish_columns(cols, seen->normal[j % SEEN], seen->small[j % SEEN]);
        fence_proxy_async_smem();  // the slot is read by the tensor core
        __syncwarp();
        if (lane == 0 && g != p.stall_stage) mbar_arrive(full(so));
      }
      g = g_item + it.nsteps;
    }
  }
}

// The second run: items with columns of small elements, one by one, after the
// first one and a __syncthreads().  A sketch whose items all have such columns
// takes almost three times as long (30011 x 333, k = 666 192 -> 525 us; the
// CUDA cores take 644).  That its code is there at all costs the first run
// registers, inlined or not (192 us against 174 without it, 4096 x 256, k = 64
// 14.4 against 12.7), about what the code it stands for, FP32 FMAs in the
// epilogue warps, cost before (194 and 14.0 us; 13.3 ms for small elements).
template <int DIST>
__device__ __noinline__ void run_again(const CUtensorMap* pmap, const F32Params& p, uint8_t* smem,
                                       uint32_t tmem) {
  Seen* seen = reinterpret_cast<Seen*>(smem + OFF_SEEN);
  const volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + OFF_MISC);
  const int item_step = static_cast<int>(gridDim.x);
  int g = 0, gc = 0, j = 0;  // the first run's
  for (int idx = static_cast<int>(blockIdx.x); idx < p.nitems; idx += item_step, ++j) {
    const Item it = get_item(p, idx);
    g += it.nsteps;
    gc += it.nchains;
  }
  uint32_t runs = 1;
  int jj = 0;  // number of the item among the block's
  for (int idx = static_cast<int>(blockIdx.x); idx < p.nitems && *abort_flag == 0;
       idx += item_step, ++jj) {
    if (((seen->redo[(jj % REDO_BITS) / 32] >> (jj % 32)) & 1u) == 0u) continue;
    const Item it = get_item(p, idx);
    if (!find_small_columns(p.A + it.lbeg * p.lda + it.q0, p.lda, it.lend - it.lbeg,
                            static_cast<int>(min(static_cast<int64_t>(p.nt), p.Q - it.q0)), seen,
                            reinterpret_cast<uint32_t*>(smem)))
      continue;
    run_items<DIST, true>(pmap, p, smem, tmem, idx, item_step, idx + 1, runs++, g, gc, j);
    g += it.nsteps;
    gc += it.nchains;
    ++j;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }
}

template <int DIST>
__global__ void __launch_bounds__(THREADS, 1)
    k_sketch_fp32_left(const __grid_constant__ CUtensorMap pmap,
                       const __grid_constant__ F32Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + OFF_MISC);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + OFF_MISC + 4);
  Seen* seen = reinterpret_cast<Seen*>(smem + OFF_SEEN);
  const int warp = uniform(static_cast<int>(threadIdx.x >> 5));

  if (threadIdx.x == 0) {
    const uint32_t bar0 = smem_u32(smem) + OFF_BAR;  // (see run_items)
    for (int i = 0; i < SLOTS; ++i) {
      mbar_init(bar0 + 8u * i, GROUP_WARPS);
      mbar_init(bar0 + 8u * (SLOTS + i), 1);
    }
    mbar_init(bar0 + 8u * (2 * SLOTS), 1);
    mbar_init(bar0 + 8u * (2 * SLOTS + 1), N_EPI);
    mbar_init(bar0 + 8u * (2 * SLOTS + 2), 1);
    *abort_flag = 0;
    mbar_fence_init();
  }
  for (uint32_t i = threadIdx.x; i < sizeof(Seen) / 4; i += THREADS)
    reinterpret_cast<uint32_t*>(seen)[i] = 0u;
  if (warp == 0) {
    tmem_alloc(smem_u32(tmem_slot), 512u);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();
  pdl_trigger();
  const uint32_t tmem = uniform(*tmem_slot);

  run_items<DIST, false>(&pmap, p, smem, tmem, static_cast<int>(blockIdx.x),
                         static_cast<int>(gridDim.x), p.nitems, 0u, 0, 0, 0);
  // every chain has been read out (or the block gives up)
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (__builtin_expect(seen->any_redo != 0u, 0)) run_again<DIST>(&pmap, p, smem, tmem);
  if (warp == 0) {
    __syncwarp();
    tmem_dealloc(tmem, 512u);
  }
}

// ---- host side ----
int sm_count() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 148;
  }
  return sms;
}

struct F32Plan {
  int nt, splits, chain, cross;
  int64_t tiles_p, tiles_q, chunk, ldp;
};

F32Plan plan_f32(const GemmShape& s, int dist = kGaussian) {
  F32Plan pl;
  const int64_t chunks = (s.Q + 63) / 64;
  pl.tiles_q = (chunks + NCH - 1) / NCH;
  pl.tiles_p = (s.P + BM - 1) / BM;
  pl.ldp = (s.Q + 3) / 4 * 4;
  // splits of m that fill whole waves of CTAs, each at least one stage per
  // worker group; where the most of them leave SMs idle, narrower tiles (each
  // generates its S again, but drains sooner: 4096 x 256, k = 64 18.5 -> 15.4
  // us); more than 64 splits (whose partials the reduction reads) only of
  // eight stages or more (65536 x 32, k = 64 57 -> 31 us)
  const int64_t sms = sm_count();
  const int64_t steps = (s.L + SL - 1) / SL;
  const int64_t smax = std::max<int64_t>(
      {int64_t{1}, std::min<int64_t>(steps / GROUPS, 64), std::min<int64_t>(steps / 8, sms)});
  while (pl.tiles_q < chunks && pl.tiles_p * (pl.tiles_q + 1) * smax <= sms) ++pl.tiles_q;
  pl.nt = static_cast<int>((chunks + pl.tiles_q - 1) / pl.tiles_q) * 64;
  pl.tiles_q = (chunks * 64 + pl.nt - 1) / pl.nt;
  const int64_t tiles = pl.tiles_p * pl.tiles_q;
  const int64_t best = best_splits(tiles, sms, smax);
  int64_t per = (steps + best - 1) / best;
  pl.chunk = per * SL;
  pl.splits = static_cast<int>((steps + per - 1) / per);
  const int64_t cap = dist == kRademacher ? CHAIN_R : s.L >= kLongRows ? CHAIN_LONG : CHAIN;
  const int64_t nchains = (per + cap - 1) / cap;
  pl.chain = static_cast<int>((per + nchains - 1) / nchains);
  pl.cross = std::max(1, CROSS / pl.chain);
  return pl;
}

// The partials [splits][P][ldp] in boxes of 16 columns x 32 rows with the
// 64-byte swizzle.
bool encode_partials(CUtensorMap* map, float* part, int64_t Q, int64_t P, int splits, int64_t ldp) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (enc == nullptr) return false;
  const cuuint64_t gdim[3] = {static_cast<cuuint64_t>(Q), static_cast<cuuint64_t>(P),
                              static_cast<cuuint64_t>(splits)};
  const cuuint64_t gstride[2] = {static_cast<cuuint64_t>(ldp) * 4,
                                 static_cast<cuuint64_t>(P) * static_cast<cuuint64_t>(ldp) * 4};
  const cuuint32_t box[3] = {16, 32, 1}, estride[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, part, gdim, gstride, box, estride,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
             CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int DIST>
cudaError_t launch_f32(const CUtensorMap& pmap, const F32Params& p, unsigned grid,
                       cudaStream_t st) {
  static bool done = false;
  if (!done) {
    const cudaError_t e = cudaFuncSetAttribute(k_sketch_fp32_left<DIST>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (e != cudaSuccess) return e;
    done = true;
  }
  return launch_overlapped(k_sketch_fp32_left<DIST>, dim3(grid), dim3(THREADS), SMEM, st, 1, pmap,
                           p);
}

}  // namespace

// The left sketch with at least two stages of m.  Time, and relative
// Frobenius error against 64 bits, with FP32 FMAs on the CUDA cores and here
// (Gaussian S; m x n, k):
//   4096 x 256, 64       39 -> 15.4 us    2.3e-7 -> 1.5e-7
//   30011 x 333, 666     644 -> 193 us    5.4e-7 -> 2.5e-7
//   65536 x 512, 1024    1590 -> 609 us   1.1e-6 -> 2.6e-7
//   65536 x 32, 64       253 -> 31 us     5.9e-7 -> 3.0e-7
//   16384 x 100, 300     85 -> 35 us      3.2e-7 -> 2.1e-7
//   200000 x 16, 16      754 -> 59 us     1.1e-6 -> 3.0e-7
//   1000 x 1, 1          44 -> 14 us      1.3e-7 -> 2.3e-8
//   64 x 32, 64          21 -> 13 us      1.5e-7 -> 6.7e-8
//   32 x 512, 512        15.2 -> 17.5 us  (one stage: stays on the CUDA cores)
// Chains of 11, 19 and 32 stages had errors of 3.4e-7, 5.8e-7 and 8.3e-7.
// Sums that all grow the same way lose most to truncation: a uniform S and an
// A without negative elements have 3.4e-7 at 30011 x 333, k = 666 (the CUDA
// cores 1.2e-7, a normal A 2.3e-7 here and 5.2e-7 there).
size_t tc32_workspace_bytes(const GemmShape& s) {
  if (!s.left || s.L < 2 * SL) return 0;
  // (a k of more than 65535 tiles is refused, as the CUDA-core form does)
  if (s.P > 65535LL * (s.Q > 128 ? 128 : 256)) return 0;
  const F32Plan pl = plan_f32(s);
  // 32-bit item numbers, and strides that a tensor map holds
  if (pl.tiles_p * pl.tiles_q * pl.splits >= (int64_t(1) << 31) || s.Q >= (int64_t(1) << 31) ||
      s.P * pl.ldp * 4 >= (int64_t(1) << 40))
    return 0;
  return static_cast<size_t>(pl.splits) * s.P * pl.ldp * sizeof(float);
}

cudaError_t tc32_sketch_left(const sk_sketch* h, const GemmShape& s, const float* A, int64_t lda,
                             float* Y, int64_t ldy, void* ws, size_t ws_bytes, cudaStream_t st) {
  const F32Plan pl = plan_f32(s, h->dist);
  if (ws == nullptr ||
      ws_bytes < static_cast<size_t>(pl.splits) * s.P * pl.ldp * sizeof(float))
    return cudaErrorInvalidValue;
  F32Params p;
  memset(&p, 0, sizeof(p));
  p.A = A;
  p.lda = lda;
  p.part = static_cast<float*>(ws);
  p.P = s.P;
  p.Q = s.Q;
  p.L = s.L;
  p.ldp = pl.ldp;
  p.chunk = pl.chunk;
  p.tiles_p = static_cast<int>(pl.tiles_p);
  p.tiles_q = static_cast<int>(pl.tiles_q);
  p.nitems = static_cast<int>(pl.tiles_p * pl.tiles_q * pl.splits);
  p.nt = pl.nt;
  p.chain = pl.chain;
  p.cross = pl.cross;
  p.vec2 = reinterpret_cast<uintptr_t>(A) % 8 == 0 && lda % 2 == 0;
  p.rk = round_keys(make_key(h->seed));
  p.status = h->d_status;
  p.timeout_ns = h->wait_limit_ns;
  p.stall_stage = h->stall_stage;
  CUtensorMap pmap;
  if (!encode_partials(&pmap, p.part, s.Q, s.P, pl.splits, pl.ldp)) return cudaErrorInvalidValue;
  const unsigned grid = static_cast<unsigned>(std::min(p.nitems, sm_count()));
  prof_mark(h->prof_start, st);
  const cudaError_t e = h->dist == kRademacher ? launch_f32<kRademacher>(pmap, p, grid, st)
                        : h->dist == kUniform  ? launch_f32<kUniform>(pmap, p, grid, st)
                                               : launch_f32<kGaussian>(pmap, p, grid, st);
  prof_mark(h->prof_stop, st);
  if (e != cudaSuccess) return e;
  count_launches(1);
  return splitk_reduce(p.part, pl.splits, s.P, s.Q, pl.ldp, h->scale, Y, ldy, st);
}

cudaError_t fp32_sketch(const sk_sketch* h, const GemmShape& s, const float* A, int64_t lda,
                        float* Y, int64_t ldy, void* ws, size_t ws_bytes, cudaStream_t st) {
  const size_t tc = tc32_workspace_bytes(s);
  if (tc != 0 && ws != nullptr && ws_bytes >= tc)
    return tc32_sketch_left(h, s, A, lda, Y, ldy, ws, ws_bytes, st);
  return simt_sketch(h, s, A, lda, Y, ldy, ws, ws_bytes, st);
}

}  // namespace sk
