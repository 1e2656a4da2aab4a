// fp32 contractions of large dense problems on the tensor cores, at the precision of fp32 multiply-adds.
//
//   forward:  Z[i][j] = sum_d A[i][d] * W[j][d]          (z_i = W a_i; Section 2, problem (P))
//   apply  :  W[j][d] -= eta * sum_i U[i][j] * V[i][d]   (W <- W - eta * sum_i u_i v_i^T; Section 3)
//
// Every fp32 operand x below 2^36 is 2^-24 times the exact sum of three bf16 values (24 significant bits in three times 8):
// hi = bf16(2^24 x), mid = bf16(2^24 x - hi), lo = 2^24 x - hi - mid.  (The scheme is that of G. Henry, P. T. P. Tang,
// A. Heinecke, "Leveraging the bfloat16 Artificial Intelligence Datatype For Higher-Precision Computations", ARITH 2019.)
// With no factor, operands below 2^-109 lose bits under bf16's smallest subnormal; the last bit of fp32's own subnormals
// asks for 2^16.  The tensor cores' power depends on how many bits of the parts' exponents change from one value to the
// next: 1000 x 20000, K = 1024 478.5 us a step with no factor, 482.5 with 2^16, 480.5 with 2^24, 479 with 2^32, which leaves
// operands below 2^28 only.
// A product is formed from six of the nine products of parts,
//   a b = hi hi + (hi mid + mid hi) + mid mid + (hi lo + lo hi),
// what is left out (mid lo, lo mid, lo lo) is below 2^-24 of it and of either sign.  The tensor core's fp32 accumulator
// rounds toward zero once per instruction of 16 reduction steps, about 2^-26 of the sum each time, so it only ever holds
// the sum of ONE chunk of 64 reduction steps, small products first and the four hi hi instructions last; the chunk
// sums are added in registers, rounded to nearest.  That makes sums of a chunk good to about 6e-8 and long sums better than
// a chain of fp32 multiply-adds, which rounds after every step: u of 600 x 10000, K = 2048 is 1.3e-7 from its 64-bit value
// (multiply-adds: 5.4e-7), of 129 x 2050, K = 195 1.1e-7 (2.0e-7).  Sums of few products are less exact than multiply-adds: for
// updates see FEW_ROWS; u = L d of 300 x 8192 with 1, 16, 64, 256 nonzero features 4.6e-8, 7.9e-8, 9.3e-8, 1.03e-7 (2.5e-8,
// 6.9e-8, 8.7e-8, 1.08e-7).
//
// The parts ("planes") are written by a bandwidth-bound pass: [3][rows][row length padded to 8] bf16 in the order of
// `Plane`.  The same planes of the samples serve the forward (contiguous along the reduction: K-major) and the update
// (contiguous along the output: MN-major).
//
// What bounds the GEMMs: the tensor pipe (six bf16 instructions per product), under the power cap.  A 256 x 256 tile of a
// CTA pair loads 96 KB per CTA and chunk for 3072 clocks of tensor work, 32 bytes a clock, half of what the tf32 kernels
// need for a tile of the same shape, because each part meets two or three others: by the clock counter a chunk takes 3072
// clocks once the pipeline runs.  1000 x 20000, K = 1024: forward 164.5 us (246 GFLOP of bf16), update 174.0, each alone and on
// cold caches.
#include <cuda.h>

#include <cstring>
#include <new>

#include "umma.cuh"
#include "umma_api.cuh"

namespace sfb {
namespace {

constexpr int BM = 128;                      // accumulator rows of a CTA (tensor memory lanes)
constexpr int BN = 256;                      // columns of a whole tile; a half tile has 128
constexpr int CHUNK = 64;                    // reduction steps an accumulator takes
constexpr float PARTS_SCALE = 0x1p24f;       // of the parts, on both sides of a product
constexpr float SUM_SCALE = 0x1p-48f;        // takes a chunk's sum back
constexpr int THREADS = 384;                 // TMA warp, MMA warp, two idle ones (whole warpgroups), 8 epilogue warps
constexpr int LAUNCH_REGS = 168;             // per thread: 384 of them fill the register file
constexpr int A_BYTES = BM * 128, SLOT_BYTES = 2 * A_BYTES;   // one plane of a chunk: 128 rows of A, up to 128 columns of B
constexpr int BUFS = 2;                      // accumulators in tensor memory
constexpr int FULL = 3;                      // chunks that may be on their way at a time, a barrier each
enum Plane { HI = 0, MID = 1, LO = 2 };

// Why the CUDA cores do a product (bits of its word): an operand that the parts cannot carry; an update of so few rows that the
// truncation of a chunk's sum shows, as it does not in longer ones (update of 300 x 8192 by 1, 2, 4, 5, 6, 8 rows: 4.6e-8
// at all of them from its 64-bit value, multiply-adds 2.5e-8, 3.2e-8, 4.0e-8, 4.4e-8, 4.7e-8, 5.3e-8).
enum Bad { BAD_VALUE = 1, BAD_FEW = 2 };
constexpr int FEW_ROWS = 6;

// Work of one launch: m_tiles x (columns / 256) whole tiles in every range of the reduction, of which the last ones
// are cut in two, and one half tile per row tile where the columns end within the first half of a tile.
struct Tiles {
  int m_tiles, n_whole;        // row tiles (256 rows of a CTA pair); whole tiles side by side
  int ranges;
  int whole, cut, ends;        // whole tiles done as such; cut in two; half tiles at the end of the columns
  int m_fastest;               // consecutive items share the B columns (1) or the A rows (0)
};
struct Item { int mt, col, width, range; };

struct TcParams {
  Tiles t;
  int k_chunks;                // chunks of the reduction (apply: an upper bound)
  int k_per_range;
  int M, N;                    // valid output rows and columns
  RowMap z;                    // forward: fp32 rows of the products
  long long range_stride;      // ... bytes from one range's to the next
  float* W;                    // apply: updated in place (rows of M values: output row = column of W)
  float eta;
  const int* n_rows;           // apply: factor rows in the planes (device)
  const int* bad;              // not zero: the CUDA cores do it, nothing is done here
  const int* status_ro;        // apply: a refused buffer
  int* status;
};

struct Ctl {
  uint64_t full[FULL], empty[7], acc_full[BUFS], acc_empty[BUFS];
  uint32_t tmem_base;
  volatile int abort;
};

template <bool APPLY>
struct Smem {
  static constexpr int SLOTS = APPLY ? 7 : 6;               // of the ring
  static constexpr int STAGE = APPLY ? 0 : 8 * 4096;        // forward: one swizzled 32 x 32 fp32 block per epilogue warp
  static constexpr int BYTES = SLOTS * SLOT_BYTES + STAGE + 1024 + (int)sizeof(Ctl);
};

// All whole tiles of the first range, then all of the second, ...: the pairs at work share the operands of a range.
__device__ __forceinline__ Item whole_tile(const Tiles& t, int w) {
  const int per = t.m_tiles * t.n_whole, range = w / per, i = w - range * per;
  int mt, nt;
  if (t.m_fastest) { nt = i / t.m_tiles; mt = i - nt * t.m_tiles; }
  else { mt = i / t.n_whole; nt = i - mt * t.n_whole; }
  return {mt, nt * BN, BN, range};
}
__device__ __forceinline__ Item half_tile(const Tiles& t, int w) {
  if (w < 2 * t.cut) {
    Item i = whole_tile(t, t.whole + (w >> 1));
    i.width = BN / 2;
    i.col += (w & 1) * (BN / 2);
    return i;
  }
  w -= 2 * t.cut;
  const int range = w / t.m_tiles;
  return {w - range * t.m_tiles, t.n_whole * BN, BN / 2, range};
}
// The i-th item of a pair: whole tiles round by round, then half tiles, of which the pairs that a last, incomplete round of
// whole tiles left out take two before the rest is dealt.
__device__ __forceinline__ bool item_of(const Tiles& t, int pair, int pairs, int i, Item& out) {
  const int rounds = t.whole / pairs, odd = t.whole - rounds * pairs;   // `odd` pairs have a round more
  const int mine = rounds + (pair < odd ? 1 : 0);
  if (i < mine) {
    out = whole_tile(t, i * pairs + pair);
    return true;
  }
  i -= mine;
  int w = pair + i * pairs;
  if (odd > 0) {
    const int first = 2 * (pairs - odd);
    if (pair < odd) w = first + pair + i * pairs;
    else w = i < 2 ? 2 * (pair - odd) + i : first + pair + (i - 2) * pairs;
  }
  if (w >= 2 * t.cut + t.ends) return false;
  out = half_tile(t, w);
  return true;
}

// CTA pairs (tcgen05.mma.cta_group::2, 256 rows) on tiles of 256 or 128 columns.  A ring slot holds one plane of a chunk:
// this CTA's 128 rows of A and its half of B's columns.  The slots of a chunk come in the order lo, mid, hi, in
// which they fall free again.
//   forward: rows = samples, columns = classes, both operands contiguous along the reduction (K-major).
//   apply:   rows = columns d of W, columns = rows j of W, both contiguous along the output (MN-major).  A thread of the
//            epilogue then holds one d and many j, and a warp's access to a row of W is one line at any alignment.
template <bool APPLY>
__global__ void __launch_bounds__(THREADS, 1)
umma_f32_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const __grid_constant__ TcParams p) {
  constexpr int SLOTS = Smem<APPLY>::SLOTS;
  constexpr int BLOCKS = BN / 64;                      // 32-column blocks of an epilogue warp (half tiles: half of them)
  constexpr uint32_t IDESC = ptx::instr_desc(1u, APPLY ? 1u : 0u, APPLY ? 1u : 0u, 2 * BM, BN);
  constexpr uint32_t IDESC_HALF = ptx::instr_desc(1u, APPLY ? 1u : 0u, APPLY ? 1u : 0u, 2 * BM, BN / 2);

  extern __shared__ uint8_t smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  float* stages = reinterpret_cast<float*>(ring + SLOTS * SLOT_BYTES);
  Ctl* ctl = reinterpret_cast<Ctl*>(ring + SLOTS * SLOT_BYTES + Smem<APPLY>::STAGE);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (uniform: see elect_one)
  chain_next();
  const uint32_t rank = ptx::cluster_ctarank();        // 0 issues the MMAs of the pair
  const int pair = blockIdx.x / 2, pairs = gridDim.x / 2;

  if (threadIdx.x == 0) {
    for (int f = 0; f < FULL; ++f) ptx::mbar_init(&ctl->full[f], 1);
    for (int s = 0; s < SLOTS; ++s) ptx::mbar_init(&ctl->empty[s], 1);
    for (int b = 0; b < BUFS; ++b) {
      ptx::mbar_init(&ctl->acc_full[b], 1);
      ptx::mbar_init(&ctl->acc_empty[b], 16);          // the epilogue warps of both CTAs
    }
    ctl->abort = 0;
    ptx::fence_barrier_init();
    ptx::prefetch_tmap(&tmA);
    ptx::prefetch_tmap(&tmB);
  }
  if (warp == 1) {
    ptx::tmem_alloc<2>(&ctl->tmem_base, 512);
    ptx::tmem_relinquish<2>();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();
  ptx::tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  chain_wait();
  // uniform over the grid: nothing writes these words while the kernel runs
  const bool idle = *p.bad != 0 || (APPLY && (*p.status_ro & SFB_DEV_BAD_HEADER) != 0);
  int k_chunks = p.k_chunks, k_per_range = p.k_per_range;
  if (APPLY) k_chunks = k_per_range = min(k_chunks, (*p.n_rows + CHUNK - 1) / CHUNK);
  const bool work = !idle && k_chunks > 0;
  Item w;

  if (warp < 4) {
  ptx::regs_dec<56>();   // 128 x 56 + 256 x 224 registers = the 384 x 168 of the launch
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    int s = 0, it = 0;
    uint32_t ph = 0;
    bool ok = true;
    const uint64_t pol = ptx::l2_policy(0);
    for (int i = 0; work && ok && item_of(p.t, pair, pairs, i, w); ++i) {
      const int row0 = (w.mt * 2 + (int)rank) * BM, col0 = w.col + (int)rank * (w.width / 2);
      const uint32_t chunk_bytes = 3 * 2 * (A_BYTES + w.width / 2 * 128);
      const int k_end = min((w.range + 1) * k_per_range, k_chunks);
      for (int k = w.range * k_per_range; k < k_end && ok; ++k, ++it) {
        uint64_t* full = &ctl->full[it % FULL];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int plane = q == 0 ? LO : q == 1 ? MID : HI;
          // (the first round of the ring is free: no wait, which takes 150 clocks even where there is nothing to wait for)
          ok = it * 3 + q < SLOTS || wait_or_abort(&ctl->empty[s], ph ^ 1u, ctl, p.status);
          if (!ok) break;
          if (lane == 0) {
            uint8_t* a_dst = ring + s * SLOT_BYTES;
            uint8_t* b_dst = a_dst + A_BYTES;
            const uint32_t bar = ptx::map_to_cta(ptx::smem_u32(full), 0);
            if (rank == 0 && q == 0) ptx::mbar_expect_tx(full, chunk_bytes);
            if (!APPLY) {
              ptx::tma_load_3d_hint_pair(a_dst, &tmA, bar, k * CHUNK, row0, plane, pol);
              ptx::tma_load_3d_hint_pair(b_dst, &tmB, bar, k * CHUNK, col0, plane, pol);
              if (w.width == BN) ptx::tma_load_3d_hint_pair(b_dst + 64 * 128, &tmB, bar, k * CHUNK, col0 + 64, plane, pol);
            } else {
              ptx::tma_load_3d_hint_pair(a_dst, &tmA, bar, row0, k * CHUNK, plane, pol);
              ptx::tma_load_3d_hint_pair(a_dst + 64 * 128, &tmA, bar, row0 + 64, k * CHUNK, plane, pol);
              ptx::tma_load_3d_hint_pair(b_dst, &tmB, bar, col0, k * CHUNK, plane, pol);
              if (w.width == BN) ptx::tma_load_3d_hint_pair(b_dst + 64 * 128, &tmB, bar, col0 + 64, k * CHUNK, plane, pol);
            }
          }
          __syncwarp();
          if (++s == SLOTS) { s = 0; ph ^= 1u; }
        }
      }
    }
    if ((!ok || ctl->abort) && rank == 0) {   // copies in flight land before the CTA goes away (bounded)
      for (int q = 1; q <= FULL && q <= it; ++q)
        ptx::mbar_wait(&ctl->full[(it - q) % FULL], (uint32_t)((it - q) / FULL) & 1u, 1u << 16);
      if (!ok) ptx::mbar_wait(&ctl->full[it % FULL], (uint32_t)(it / FULL) & 1u, 1u << 16);   // (of a chunk begun)
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (even CTA)
    int s = 0, it = 0;
    bool ok = rank == 0;
    for (int i = 0; work && ok && item_of(p.t, pair, pairs, i, w); ++i) {
      const uint32_t idesc = w.width == BN ? IDESC : IDESC_HALF;
      const int k_end = min((w.range + 1) * k_per_range, k_chunks);
      for (int k = w.range * k_per_range; k < k_end && ok; ++k, ++it) {
        const int buf = it % BUFS;
        ok = it < BUFS || wait_or_abort(&ctl->acc_empty[buf], ((uint32_t)(it / BUFS) & 1u) ^ 1u, ctl, p.status);
        if (!ok) break;
        const uint32_t acc = tmem_base + buf * BN;
        int slot[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          slot[q] = s;
          if (++s == SLOTS) s = 0;
        }
        ok = wait_or_abort(&ctl->full[it % FULL], (uint32_t)(it / FULL) & 1u, ctl, p.status);
        if (!ok) break;
        ptx::tc_fence_after();
        if (ptx::elect_one()) {   // small products first: the accumulator's rounding is relative to what it holds
          uint64_t a[3], b[3];
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const uint32_t addr = ptx::smem_u32(ring) + slot[q] * SLOT_BYTES;
            a[q] = ptx::smem_desc(addr, APPLY ? CHUNK * 128 : 16, 1024, 2);
            b[q] = a[q] + (A_BYTES >> 4);
          }
          constexpr uint32_t STEP = APPLY ? (16 * 128) >> 4 : 32 >> 4;   // 16 reduction steps further
          auto product = [&](int qa, int qb) {
#pragma unroll
            for (int m = 0; m < CHUNK / 16; ++m) ptx::mma_f16<2>(acc, a[qa] + m * STEP, b[qb] + m * STEP, idesc, 1u);
          };
          ptx::mma_f16<2>(acc, a[0], b[2], idesc, 0u);            // lo hi, hi lo
#pragma unroll
          for (int m = 1; m < CHUNK / 16; ++m) ptx::mma_f16<2>(acc, a[0] + m * STEP, b[2] + m * STEP, idesc, 1u);
          product(2, 0);
          ptx::mma_commit_pair(&ctl->empty[slot[0]]);
          product(1, 1);                                          // mid mid, mid hi, hi mid
          product(1, 2);
          product(2, 1);
          ptx::mma_commit_pair(&ctl->empty[slot[1]]);
          product(2, 2);                                          // hi hi
          ptx::mma_commit_pair(&ctl->empty[slot[2]]);
          ptx::mma_commit_pair(&ctl->acc_full[buf]);
        }
        __syncwarp();
      }
    }
  }
  } else {
    ptx::regs_inc<224>();
    // ------------------------------------------------------------------ epilogue (eight warps, both CTAs)
    // A warp reads the tensor memory lanes of its quarter and half of the tile's columns; its part of the tile stays in
    // registers (an output row per thread) while the chunks are added up.
    const int e = warp - 4, quarter = warp & 3, half = e >> 2;
    float* stage = stages + e * 1024;
    const float2 back = make_float2(SUM_SCALE, SUM_SCALE);
    int it = 0;
    bool ok = true;
    for (int i = 0; work && ok && item_of(p.t, pair, pairs, i, w); ++i) {
      const int row0 = (w.mt * 2 + (int)rank) * BM + quarter * 32;   // the warp's 32 output rows
      const int col0 = w.col + half * (w.width / 2);                 // ... and width / 2 columns
      const bool all = w.width == BN;
      const int k_begin = w.range * k_per_range, k_end = min(k_begin + k_per_range, k_chunks);
      float2 acc[BLOCKS][16];
#pragma unroll
      for (int b = 0; b < BLOCKS; ++b)
#pragma unroll
        for (int q = 0; q < 16; ++q) acc[b][q] = make_float2(0.f, 0.f);
      for (int k = k_begin; k < k_end; ++k, ++it) {
        const int buf = it % BUFS;
        ok = wait_or_abort(&ctl->acc_full[buf], (uint32_t)(it / BUFS) & 1u, ctl, p.status);
        if (!ok) break;
        ptx::tc_fence_after();
        const uint32_t taddr = tmem_base + buf * BN + ((uint32_t)(quarter * 32) << 16) + half * (w.width / 2);
#pragma unroll
        for (int b = 0; b < BLOCKS; b += 2) {
          if (b > 0 && !all) break;
          uint32_t v0[32], v1[32];
          ptx::tmem_ld32(taddr + b * 32, v0);
          ptx::tmem_ld32(taddr + b * 32 + 32, v1);
          ptx::tmem_ld_wait();
          if (b + 2 == (all ? BLOCKS : BLOCKS / 2)) {
            // the last of it is in registers (tcgen05.wait::ld), so the next MMAs may overwrite it: nothing else to publish
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) {
              if (rank == 0) ptx::mbar_arrive(&ctl->acc_empty[buf]);
              else ptx::mbar_arrive_cluster_relaxed(ptx::map_to_cta(ptx::smem_u32(&ctl->acc_empty[buf]), 0));
            }
          }
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            acc[b][q] = __ffma2_rn(make_float2(__uint_as_float(v0[2 * q]), __uint_as_float(v0[2 * q + 1])), back, acc[b][q]);
            acc[b + 1][q] = __ffma2_rn(make_float2(__uint_as_float(v1[2 * q]), __uint_as_float(v1[2 * q + 1])), back, acc[b + 1][q]);
          }
        }
        if (APPLY && k == max(k_begin, k_end - 3) && row0 < p.M)   // W's part of the tile on its way to L2: a row of W per lane
          for (int c = lane; c < w.width / 2 && col0 + c < p.N; c += 32)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p.W + (size_t)(col0 + c) * p.M + row0));
      }
      if (!ok) break;
      if constexpr (APPLY) {
        // A lane per column of W, a row of W per register, in pieces of 16 rows; the old values are loaded two pieces ahead
        // where the whole part of the tile exists.  (Any more of them in flight, or conditional ones, and the compiler
        // puts loaded values on the stack one by one: 27000 clocks a tile instead of the 6000 that the next tile's
        // first two chunks hide.)
        constexpr int PIECES = BN / 32;
        const int left = min(p.N - col0, w.width / 2);               // rows of W of this part of the tile
        const int whole = row0 + 32 <= p.M && left > 0 ? left / 16 : 0;   // pieces without a missing value
        const float* rd = p.W + (size_t)col0 * p.M + row0 + lane;
        float* wr = p.W + (size_t)col0 * p.M + row0 + lane;
        float old[2][16];
        auto fetch = [&](int s) {
#pragma unroll
          for (int q = 0; q < 16; ++q, rd += p.M)
            asm volatile("ld.global.cs.f32 %0, [%1];" : "=f"(old[s & 1][q]) : "l"(rd) : "memory");
        };
        if (whole > 0) {
          fetch(0);
          if (whole > 1) fetch(1);
#pragma unroll
          for (int s = 0; s < PIECES; ++s) {
            if (s >= whole) break;
#pragma unroll
            for (int q = 0; q < 16; ++q, wr += p.M) {
              const float2 sum = acc[s >> 1][(s & 1) * 8 + (q >> 1)];
              asm volatile("st.global.cs.f32 [%0], %1;" ::"l"(wr), "f"(fmaf(-p.eta, q & 1 ? sum.y : sum.x, old[s & 1][q])) : "memory");
            }
            if (s + 2 < PIECES && s + 2 < whole) fetch(s + 2);
          }
        }
        if (whole * 16 < left && row0 + lane < p.M) {   // ragged edges of W
#pragma unroll
          for (int s = 0; s < PIECES; ++s) {
            if (s < whole || s * 16 >= left) continue;
#pragma unroll
            for (int q = 0; q < 16; ++q, wr += p.M) {
              const float2 sum = acc[s >> 1][(s & 1) * 8 + (q >> 1)];
              if (s * 16 + q < left) *wr = fmaf(-p.eta, q & 1 ? sum.y : sum.x, *wr);
            }
          }
        }
        __syncwarp();
      } else {
#pragma unroll
        for (int b = 0; b < BLOCKS; ++b) {   // 32 x 32 blocks through shared memory, so that global memory sees whole lines
          if (b >= BLOCKS / 2 && !all) break;
          const int c0 = col0 + b * 32;
          const int lrow = lane >> 3, lq = lane & 7, c = c0 + lq * 4;
#pragma unroll
          for (int q = 0; q < 8; ++q)
            *reinterpret_cast<float4*>(stage + lane * 32 + ((q ^ (lane & 7)) << 2)) =
                make_float4(acc[b][2 * q].x, acc[b][2 * q].y, acc[b][2 * q + 1].x, acc[b][2 * q + 1].y);
          __syncwarp();
          if (c < p.z.ld) {
#pragma unroll
            for (int g = 0; g < 8; ++g) {
              const int lr = 4 * g + lrow, r = row0 + lr;
              if (r < p.M)
                *reinterpret_cast<float4*>(p.z.row(r) + w.range * p.range_stride + (size_t)c * 4) =
                    *reinterpret_cast<const float4*>(stage + lr * 32 + ((lq ^ (lr & 7)) << 2));
            }
          }
          __syncwarp();
        }
      }
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();   // nobody leaves while its pair may still signal it or read its tiles
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc<2>(tmem_base, 512);
  }
}

// ------------------------------------------------------------------------------------------------- planes
// One operand: `rows` rows of C fp32 values (minus those of `sub`) to planes dst + plane * plane_bytes, rows of ldc
// values (a multiple of 8; columns from C on zeros), and unchanged to `copy` (its pad columns zeros).
// idx / n_rows (device): row r of the planes is source row idx[r], r < *n_rows; rows from there to the end of their
// chunk are zeros.  rest: idx also names the rows left out (idx[r], *n_rows <= r < rows), whose values are only looked at.
struct PlaneJob {
  RowMap src, sub, copy;
  char* dst;
  long long plane_bytes;
  int rows, C, ldc;
  int vec;                 // source rows are whole 16-byte units
  const int* idx;
  const int* n_rows;
  int rest;
  int keep_if_all;         // *n_rows == rows: the planes are there already
  int blocks;
};

__device__ __forceinline__ void load8(const char* row, int c, int C, bool vec, float (&x)[8]) {
  const float* f = reinterpret_cast<const float*>(row) + c;
  if (vec && c + 8 <= C) {
    const float4 a = *reinterpret_cast<const float4*>(f), b = *reinterpret_cast<const float4*>(f + 4);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = c + q < C ? f[q] : 0.f;
  }
}

__device__ __forceinline__ void zero_planes(const PlaneJob& j, int r, int c) {
  char* d = j.dst + ((long long)r * j.ldc + c) * 2;
#pragma unroll
  for (int s = 0; s < 3; ++s) *reinterpret_cast<uint4*>(d + s * j.plane_bytes) = make_uint4(0u, 0u, 0u, 0u);
}
// Parts below this bound, operands below 2^36, have products below 2^120: no instruction and no chunk sum overflows (two
// infinite products of parts with different signs would make a NaN of a sum that is an infinity).
constexpr float PARTS_BOUND = 0x1p60f;
// Eight values of source row i at column c: to row r of the planes (put), or only looked at.  False: one of them is not
// finite, or not below 2^36.
__device__ __forceinline__ bool make_planes(const PlaneJob& j, int i, int r, int c, bool put) {
  float x[8];
  load8(j.src.row(i), c, j.C, j.vec, x);
  if (j.sub.base != nullptr) {
    float y[8];
    load8(j.sub.row(i), c, j.C, j.vec, y);
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = __fsub_rn(x[q], y[q]);
  }
  if (j.copy.base != nullptr) {
    float4* d = reinterpret_cast<float4*>(j.copy.row(i) + (size_t)c * 4);
    if (c < j.copy.ld) d[0] = make_float4(x[0], x[1], x[2], x[3]);
    if (c + 4 < j.copy.ld) d[1] = make_float4(x[4], x[5], x[6], x[7]);
  }
  uint32_t w[3][4];
  bool fine = true;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float a = x[2 * q] * PARTS_SCALE, b = x[2 * q + 1] * PARTS_SCALE;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
      const uint32_t u = *reinterpret_cast<const uint32_t*>(&h);
      const float ha = __uint_as_float(u << 16), hb = __uint_as_float(u & 0xffff0000u);
      if (s == HI) fine = fine && fabsf(ha) < PARTS_BOUND && fabsf(hb) < PARTS_BOUND;
      w[s][q] = u;
      a -= ha; b -= hb;                              // exact: the parts of a value do not overlap
    }
  }
  if (put) {
    char* d = j.dst + ((long long)r * j.ldc + c) * 2;
#pragma unroll
    for (int s = 0; s < 3; ++s) *reinterpret_cast<uint4*>(d + s * j.plane_bytes) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
  }
  return fine;
}

// Bound: HBM.  Eight values a thread at a time: 32 bytes in, 16 bytes to each plane; samples and W of 1000 x 20000,
// K = 1024 (487 MB) 74 us, 6.6 TB/s.
// refused: see is_refused.
__global__ void __launch_bounds__(256) planes_kernel(const __grid_constant__ PlaneJob j0, const __grid_constant__ PlaneJob j1,
                                                     int* bad, const int* refused) {
  chain();
  const bool second = (int)blockIdx.x >= j0.blocks;
  const PlaneJob j = second ? j1 : j0;
  const unsigned per_row = j.ldc >> 3, units = j.rows * per_row;   // (the workspace limit keeps them below 2^31)
  const int n_listed = j.n_rows != nullptr ? *j.n_rows : j.rows;   // (asked for together with the status word)
  if (is_refused(refused)) return;
  const int n = min(n_listed, j.rows);
  if (j.n_rows != nullptr && n > 0 && n < FEW_ROWS && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(bad, BAD_FEW);
  if (j.keep_if_all && n == j.rows) return;
  const int n_chunk = (n + CHUNK - 1) / CHUNK * CHUNK;
  bool fine = true;
  for (unsigned u = (blockIdx.x - (second ? j0.blocks : 0)) * 256u + threadIdx.x; u < units; u += j.blocks * 256u) {
    const int r = (int)(u / per_row), c = (int)(u - (unsigned)r * per_row) * 8;
    if (r >= n && r < n_chunk) zero_planes(j, r, c);
    if (r >= n && !j.rest) continue;
    fine = make_planes(j, j.idx != nullptr ? j.idx[r] : r, r, c, r < n) && fine;
  }
  if (!fine) atomicOr(bad, BAD_VALUE);
}

// idx[0 .. n): the rows i < K with flags[i] != 0, ascending; idx[n ..): the others.  *n_active (optional): rows with
// active[i] != 0.  One block; a thread takes K / 1024 consecutive rows.
__global__ void __launch_bounds__(1024) list_rows_kernel(const uint8_t* flags, const uint8_t* active, int K, int* idx,
                                                         int* n_out, int* n_active) {
  chain();
  __shared__ int warp_sum[32], act_sum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (K + 1023) / 1024, lo = min(K, (int)threadIdx.x * per), hi = min(K, lo + per);
  int n = 0, na = 0;
  for (int i = lo; i < hi; ++i) {
    n += flags[i] != 0 ? 1 : 0;
    if (active != nullptr) na += active[i] != 0 ? 1 : 0;
  }
  int inc = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
    na += __shfl_xor_sync(0xffffffffu, na, o);
  }
  if (lane == 31) warp_sum[warp] = inc;
  if (lane == 0) act_sum[warp] = na;
  __syncthreads();
  int before = 0, total = 0, total_active = 0;
  for (int w = 0; w < 32; ++w) {
    before += w < warp ? warp_sum[w] : 0;
    total += warp_sum[w];
    total_active += act_sum[w];
  }
  int at = before + inc - n, rest = total + lo - at;
  for (int i = lo; i < hi; ++i) idx[flags[i] != 0 ? at++ : rest++] = i;
  if (threadIdx.x == 0) {
    *n_out = total;
    if (n_active != nullptr) *n_active = total_active;
  }
}

// planes as (column, row, plane), boxes of 64 columns x box_rows rows of one plane
bool encode_planes(CUtensorMap* m, const void* base, int C, int rows, int ldc, long long plane_bytes, int box_rows) {
  auto fn = tensor_map_encoder();
  if (fn == nullptr) return false;
  cuuint64_t dims[3] = {(cuuint64_t)C, (cuuint64_t)rows, 3};
  cuuint64_t strides[2] = {(cuuint64_t)ldc * 2, (cuuint64_t)plane_bytes};
  cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// How many CTA pairs the device holds at once (0: the kernel cannot run).
template <bool APPLY>
int pairs_at_once(int num_sms) {
  constexpr int smem = Smem<APPLY>::BYTES;
  static PerDeviceOnce once;
  static int pairs = 0;
  const bool ready = set_up_device(once, [&] {
    auto kernel = umma_f32_kernel<APPLY>;
    cudaFuncAttributes fa;
    if (!allow_smem(kernel, smem) || cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) return false;
    if (fa.numRegs != LAUNCH_REGS) return false;   // the register split would wait for ever
    pairs = cta_pairs_at_once(kernel, THREADS, smem, num_sms);
    return true;
  });
  return ready ? pairs : 0;
}

template <bool APPLY>
int launch_gemm(cudaStream_t s, const CUtensorMap& a, const CUtensorMap& b, const TcParams& p, int num_sms) {
  const int pairs = pairs_at_once<APPLY>(num_sms);
  if (pairs < 1) return SFB_ERR_CUDA;
  auto kernel = umma_f32_kernel<APPLY>;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  const int work = p.t.whole + 2 * p.t.cut + p.t.ends;
  cfg.gridDim = dim3(2 * (work < pairs ? work : pairs), 1, 1);
  cfg.blockDim = dim3(THREADS, 1, 1);
  cfg.dynamicSmemBytes = Smem<APPLY>::BYTES;
  cfg.stream = s;
  cfg.attrs = at; cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, a, b, p) == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

// Tiles, and (forward) number of ranges, with the least estimated time: a chunk takes T_WHOLE or T_HALF on the busiest pair
// and at least the time of a tile's stores, EPI, has to pass per tile; partial products go out and come back at 5 TB/s.
constexpr double T_WHOLE = 2.4, T_HALF = 1.4, EPI = 4.0;   // us
struct Geometry {
  Tiles t;
  int per;     // chunks of a range
  double us;
};
Geometry pick(int M, int N, long long chunks, long long max_ranges, int pairs) {
  Geometry best;
  best.us = -1.0;
  const long long m_tiles = (M + 2 * BM - 1) / (2 * BM);
  const int halves = (N + BN / 2 - 1) / (BN / 2), n_whole = halves / 2;
  for (long long ks = 1; ks <= max_ranges && (ks == 1 || chunks >= 4 * ks); ++ks) {
    const long long per = (chunks + ks - 1) / ks, ranges = (chunks + per - 1) / per;
    const long long whole = m_tiles * n_whole * ranges, ends = m_tiles * (halves & 1) * ranges;
    // the last, incomplete round of whole tiles as it is, or cut in two: beside the half tiles at the end either way
    for (int c = 0; c < 2; ++c) {
      const long long cut = c == 0 ? 0 : whole % pairs;
      if (c == 1 && cut == 0) continue;
      const long long rounds = (whole - cut + pairs - 1) / pairs, left = rounds * pairs - (whole - cut);   // pairs with a round less
      const long long small = 2 * cut + ends, beside = small < 2 * left ? small : 2 * left;
      const double small_rounds = (double)((small - beside + pairs - 1) / pairs);
      const double tw = per * T_WHOLE > EPI ? per * T_WHOLE : EPI, th = per * T_HALF > 0.6 * EPI ? per * T_HALF : 0.6 * EPI;
      const double us = rounds * tw + small_rounds * th + EPI + (ranges > 1 ? (double)ranges * M * N * 8 / 5e6 : 0.0);
      if (best.us < 0 || us < best.us) {
        best.t = {(int)m_tiles, n_whole, (int)ranges, (int)(whole - cut), (int)cut, (int)ends, 0};
        best.per = (int)per;
        best.us = us;
      }
    }
  }
  return best;
}

}  // namespace

constexpr int F32TC_MAX_RANGES = 16;
// Planes a context may hold: six bytes for every value of samples, W and u, beside the caller's own four.  The limit is a choice
// and no measured line: the largest problems keep that memory.  (planes_kernel counts units of eight values in 32 bits and
// relies on it.)
constexpr long long F32TC_MAX_BYTES = 2LL << 30;

struct F32Tc {
  int J, D, K, B, num_sms;
  int ldd, ldj, ldp;           // row lengths of the planes (multiples of 8) and of the partial products
  char* mem;                   // one allocation for all of the following
  char *xp, *wp, *up;          // planes of the samples (update: of the listed v rows), of W, of the listed u rows
  float* part;
  long long part_rows;         // rows of partial products there is room for
  uint8_t* flags;              // which u rows hold a nonzero value
  int* idx;                    // list_rows_kernel
  int* words;                  // rows in the list; operands not finite: of the forward, of the update
};

// Estimated microseconds of a step on this route and on the CUDA cores, fitted to 200 shapes timed on both (15 million to 20
// billion multiply-adds; the line lies near 200 million for a few hundred samples, lower where few tiles leave the
// CUDA cores a long serial reduction).  87 of the 200 go to the tensor cores, none of them slower, the median 1.6 times
// faster; 600 x 10000, K = 2048 950 -> 318 us, 1000 x 20000, K = 1024 1737 -> 479.
static bool pays(int K, int J, int D, bool pair, double cores_forward_us, int pairs) {
  if (D < 2 * CHUNK) return false;
  const Geometry f = pick(K, J, (D + CHUNK - 1) / CHUNK, F32TC_MAX_RANGES, pairs), a = pick(D, J, (K + CHUNK - 1) / CHUNK, 1, pairs);
  const double planes = ((double)K * D * 14 + (double)J * D * 10 + (double)K * J * 10) / 5e6;
  const double chain = 0.68 * K / 16, rate = 2.0 * K * (double)J * D / 46e6;
  const double cores = 13.0 + 1.05 * cores_forward_us + (chain > rate ? chain : rate) + (pair ? 10.0 + (double)K * D * 12 / 4e6 : 0.0);
  return f.us + a.us + planes + 27.0 < cores;
}

int f32tc_create(const sfb_desc& d, cudaStream_t s, double cores_forward_us, F32Tc** out) {
  *out = nullptr;
  const long long K = (long long)d.P * d.B, ldd = pad_to(d.D, 8), ldj = pad_to(d.J, 8), ldp = pad_to(d.J, 4);
  if (tensor_map_encoder() == nullptr) return SFB_OK;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (!pays((int)K, d.J, d.D, d.model == SFB_DML, cores_forward_us, sms / 2)) return SFB_OK;
  // a kernel that cannot run here (see pairs_at_once) is found out now: the CUDA cores have their workspaces or not from here on
  if (pairs_at_once<false>(sms) < 1 || pairs_at_once<true>(sms) < 1) return SFB_OK;
  const Geometry f = pick((int)K, d.J, (d.D + CHUNK - 1) / CHUNK, F32TC_MAX_RANGES, sms / 2);
  const long long part = f.t.ranges > 1 ? f.t.ranges * K * ldp * 4 : 0;
  if (6 * (K * ldd + d.J * ldd + K * ldj) > F32TC_MAX_BYTES) return SFB_OK;
  F32Tc* t = new (std::nothrow) F32Tc();
  if (t == nullptr) return SFB_ERR_ALLOC;
  memset(t, 0, sizeof(*t));
  t->J = d.J; t->D = d.D; t->K = (int)K; t->B = d.B; t->num_sms = sms;
  t->ldd = (int)ldd; t->ldj = (int)ldj; t->ldp = (int)ldp;
  t->part_rows = f.t.ranges > 1 ? f.t.ranges * K : 0;
  // (seven allocations take twice as long: 1000 x 20000, K = 1024 1.74 ms for sfb_create, 0.74 with one)
  long long bytes = 0;
  auto take = [&](long long n) {
    const long long at = bytes;
    bytes += pad_to(n, 256);
    return at;
  };
  const long long xp = take(6 * K * ldd), wp = take(6 * d.J * ldd), up = take(6 * K * ldj), pt = take(part), fl = take(K), ix = take(K * 4),
                  wd = take(256);
  bool ok = cudaMalloc(&t->mem, (size_t)bytes) == cudaSuccess;
  if (ok) {
    t->xp = t->mem + xp; t->wp = t->mem + wp; t->up = t->mem + up;
    t->part = reinterpret_cast<float*>(t->mem + pt);
    t->flags = reinterpret_cast<uint8_t*>(t->mem + fl);
    t->idx = reinterpret_cast<int*>(t->mem + ix);
    t->words = reinterpret_cast<int*>(t->mem + wd);
    ok = cudaMemsetAsync(t->words, 0, 256, s) == cudaSuccess;
  }
  if (!ok) {   // the CUDA-core route needs none of this
    cudaGetLastError();
    f32tc_destroy(t);
    return SFB_OK;
  }
  *out = t;
  return SFB_OK;
}

void f32tc_destroy(F32Tc* t) {
  if (t == nullptr) return;
  cudaFree(t->mem);
  delete t;
}

uint8_t* f32tc_flags(F32Tc* t) { return t->flags; }
int* f32tc_bad_forward(F32Tc* t) { return t->words + 1; }
int* f32tc_bad_apply(F32Tc* t) { return t->words + 2; }

static RowMap plain_rows(const void* base, int ld, int rows) {
  RowMap m;
  m.base = const_cast<char*>(reinterpret_cast<const char*>(base));
  m.worker_stride = 0; m.ld = ld; m.B = rows; m.es = 4;
  return m;
}

static int launch_planes(cudaStream_t s, PlaneJob a, PlaneJob b, int num_sms, int* bad, const int* refused) {
  auto blocks = [=](const PlaneJob& j) {
    const long long n = ((long long)j.rows * (j.ldc / 8) + 255) / 256;
    return (int)(j.keep_if_all && n > num_sms * 16 ? num_sms * 16 : n);   // (blocks that most often have nothing to do: 13 -> 5 us)
  };
  a.blocks = blocks(a);
  b.blocks = blocks(b);
  launch_chained(planes_kernel, a.blocks + b.blocks, 256, 0, s, a, b, bad, refused);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

int f32tc_forward(F32Tc* t, cudaStream_t s, const float* W, const float* X, const float* Xb, int K, RowMap u, RowMap v,
                  int* dev_status, RowMap* z, int* nsplit, long long* split_stride) {
  const int D = t->D, J = t->J;
  const bool vec = (D & 3) == 0;
  PlaneJob jx = {}, jw = {};
  jx.src = plain_rows(X, D, K);
  if (Xb != nullptr) jx.sub = plain_rows(Xb, D, K);
  jx.copy = v;
  jx.dst = t->xp; jx.plane_bytes = (long long)t->K * t->ldd * 2;
  jx.rows = K; jx.C = D; jx.ldc = t->ldd; jx.vec = vec;
  jw.src = plain_rows(W, D, J);
  jw.dst = t->wp; jw.plane_bytes = (long long)J * t->ldd * 2;
  jw.rows = J; jw.C = D; jw.ldc = t->ldd; jw.vec = vec;
  int r, launches = 0;
  if ((r = launch_planes(s, jx, jw, t->num_sms, f32tc_bad_forward(t), nullptr)) < 0) return r;
  launches += r;

  const int chunks = (D + CHUNK - 1) / CHUNK;
  long long max_ranges = t->part_rows / K;
  if (max_ranges > F32TC_MAX_RANGES) max_ranges = F32TC_MAX_RANGES;
  const Geometry g = pick(K, J, chunks, max_ranges < 1 ? 1 : max_ranges, t->num_sms / 2);
  TcParams p;
  memset(&p, 0, sizeof(p));
  p.t = g.t;
  p.t.m_fastest = J > K;
  p.k_chunks = chunks;
  p.k_per_range = g.per;
  p.M = K; p.N = J;
  p.z = u;
  if (g.t.ranges > 1) {
    p.z.base = reinterpret_cast<char*>(t->part); p.z.worker_stride = (long long)t->B * t->ldp * 4;
    p.z.ld = t->ldp; p.z.B = t->B; p.z.es = 4;
    p.range_stride = (long long)K * t->ldp * 4;
  }
  p.bad = f32tc_bad_forward(t);
  p.status = dev_status;
  CUtensorMap ta, tb;
  if (!encode_planes(&ta, t->xp, D, K, t->ldd, jx.plane_bytes, BM) ||
      !encode_planes(&tb, t->wp, D, J, t->ldd, jw.plane_bytes, 64))
    return SFB_ERR_CUDA;
  if ((r = launch_gemm<false>(s, ta, tb, p, t->num_sms)) < 0) return r;
  launches += r;
  // operands that are not finite, or not below 2^36: the same products on the CUDA cores
  if ((r = launch_forward_f32_if(s, W, X, Xb, K, J, D, p.z, p.range_stride, g.t.ranges, p.bad)) < 0) return r;
  launches += r;
  *z = p.z; *nsplit = g.t.ranges; *split_stride = p.range_stride;
  return launches;
}

int f32tc_list(F32Tc* t, cudaStream_t s, RowMap u, int K, bool flags_ready, const uint8_t* active, int* n_active,
               const int* refused) {
  int r, launches = 0;
  if (!flags_ready) {
    if ((r = launch_row_nonzero(s, u, K, t->J, t->flags, refused)) < 0) return r;
    launches += r;
  }
  launch_chained(list_rows_kernel, 1, 1024, 0, s, t->flags, active, K, t->idx, t->words, n_active);
  return cudaGetLastError() == cudaSuccess ? launches + 1 : SFB_ERR_CUDA;
}

int f32tc_apply(F32Tc* t, cudaStream_t s, float* W, RowMap u, RowMap v, int K, float eta, int* dev_status, const int* idx,
                const int* n_rows, bool v_planes, bool left_out, const int* refused) {
  const int D = t->D, J = t->J;
  PlaneJob ju = {}, jv = {};
  ju.src = u; ju.dst = t->up; ju.plane_bytes = (long long)t->K * t->ldj * 2;
  ju.rows = K; ju.C = J; ju.ldc = t->ldj; ju.vec = 1;
  jv.src = v; jv.dst = t->xp; jv.plane_bytes = (long long)t->K * t->ldd * 2;
  jv.rows = K; jv.C = D; jv.ldc = t->ldd; jv.vec = 1;
  const bool own = idx == nullptr;
  ju.idx = jv.idx = own ? t->idx : idx;
  ju.n_rows = jv.n_rows = own ? t->words : n_rows;
  jv.rest = own && !v_planes ? 1 : 0;   // (the pass that made the planes has looked at every row)
  jv.keep_if_all = v_planes ? 1 : 0;
  int r, launches = 0;
  if ((r = launch_planes(s, ju, jv, t->num_sms, f32tc_bad_apply(t), refused)) < 0) return r;
  launches += r;
  const int chunks = (K + CHUNK - 1) / CHUNK;
  const Geometry g = pick(D, J, chunks, 1, t->num_sms / 2);
  TcParams p;
  memset(&p, 0, sizeof(p));
  p.t = g.t;
  p.t.m_fastest = J > D;
  p.k_chunks = p.k_per_range = chunks;
  p.M = D; p.N = J;
  p.W = W; p.eta = eta;
  p.n_rows = ju.n_rows;
  p.bad = f32tc_bad_apply(t);
  p.status_ro = p.status = dev_status;
  CUtensorMap ta, tb;
  if (!encode_planes(&ta, t->xp, D, K, t->ldd, jv.plane_bytes, CHUNK) || !encode_planes(&tb, t->up, J, K, t->ldj, ju.plane_bytes, CHUNK))
    return SFB_ERR_CUDA;
  if ((r = launch_gemm<true>(s, ta, tb, p, t->num_sms)) < 0) return r;
  launches += r;
  if ((r = launch_apply_f32(s, W, u, v, K, J, D, eta, dev_status, ju.idx, ju.n_rows, p.bad, left_out ? 0 : BAD_VALUE)) < 0) return r;
  return launches + r;
}

}  // namespace sfb
