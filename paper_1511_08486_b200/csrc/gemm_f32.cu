// fp32 CUDA-core contractions of the SF hot path.
//
//   forward:  Z[i][j] = sum_d A[i][d] * W[j][d]      (z_i = W a_i for every sample; Section 2, (P))
//   apply  :  W[j][d] -= eta * sum_i U[i][j] * V[i][d]  (W <- W - eta * sum_i u_i v_i^T; Section 3)
//
// All are register-blocked shared-memory SGEMMs: 256 threads, a 128 x 128 or 64 x 64 output tile, a reduction step of 16,
// operands staged k-major in shared memory so that every inner-loop read is a conflict-free 16-byte load.  The one-launch
// forward prefetches a step into registers and transposes it on the way to shared memory; the others bring theirs by
// asynchronous copies through a ring of stages.  The summation order is fixed (ascending reduction index inside one
// thread), so results are bit-reproducible run to run and, range for range, the same from all of them.
#include "common.cuh"

namespace sfb {
namespace {

constexpr int BK = 16;
constexpr int F32_MIN_LARGE_TILES = 100;   // fewer tiles of 128 x 128, and the one-launch forward takes 64 x 64

__device__ __forceinline__ float4 ld4_left(const float* p, int left, bool vec_ok) {
  if (vec_ok && left > 3) return *reinterpret_cast<const float4*>(p);
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  if (left > 0) r.x = p[0];
  if (left > 1) r.y = p[1];
  if (left > 2) r.z = p[2];
  if (left > 3) r.w = p[3];
  return r;
}

// PACKED: the multiply-adds as packed fp32 pairs (two independent round-to-nearest FMAs per instruction: half
// the issue slots of scalar FFMA for the same arithmetic, bit-identical results).  It pays in the apply kernels;
// the forward kernel, which also holds its operand prefetch in registers, measured slower with it.
template <int MI, int NI, bool PACKED>
__device__ __forceinline__ void mma_tile(const float (*As)[64 * MI + 4], const float (*Bs)[64 * NI + 4], int ty,
                                         int tx, float2 (&acc)[4 * MI][2 * NI]) {
#pragma unroll
  for (int k = 0; k < BK; ++k) {
    float a[4 * MI], b[4 * NI];
#pragma unroll
    for (int mi = 0; mi < MI; ++mi) {
      float4 t = *reinterpret_cast<const float4*>(&As[k][mi * 64 + ty * 4]);
      a[mi * 4 + 0] = t.x; a[mi * 4 + 1] = t.y; a[mi * 4 + 2] = t.z; a[mi * 4 + 3] = t.w;
    }
#pragma unroll
    for (int ni = 0; ni < NI; ++ni) {
      float4 t = *reinterpret_cast<const float4*>(&Bs[k][ni * 64 + tx * 4]);
      b[ni * 4 + 0] = t.x; b[ni * 4 + 1] = t.y; b[ni * 4 + 2] = t.z; b[ni * 4 + 3] = t.w;
    }
#pragma unroll
    for (int m = 0; m < 4 * MI; ++m) {
      const float2 aa = make_float2(a[m], a[m]);
#pragma unroll
      for (int n = 0; n < 2 * NI; ++n) {
        if (PACKED) {
          acc[m][n] = __ffma2_rn(aa, make_float2(b[2 * n], b[2 * n + 1]), acc[m][n]);
        } else {
          acc[m][n].x = fmaf(a[m], b[2 * n], acc[m][n].x);
          acc[m][n].y = fmaf(a[m], b[2 * n + 1], acc[m][n].y);
        }
      }
    }
  }
}

// ------------------------------------------------------------------------------------------ forward, one launch
// For the shapes that forward_f32_plan gives it, and where the pair difference is formed on the way and not kept (DML
// factors without v, sfb_loss).  blockIdx.z takes the reduction range [z d_per_range, + d_per_range) and writes its partial products
// range_stride bytes after the previous range's.
// Tile rows = samples i (BM = 64*MI), tile columns = classes j (BN = 64*NI), reduction over d.
// Both operands are contiguous along d, so tiles are transposed while being stored to shared memory.
// PAIR: A = X - Xb.
template <int MI, int NI, bool PAIR>
__global__ void __launch_bounds__(256, MI == 1 ? 3 : 2) forward_f32_kernel(const float* W, const float* X,
                                                          const float* Xb, int K, int J, int D,
                                                          RowMap z, RowMap v, int d_per_range, long long range_stride,
                                                          const int* only_if) {
  chain_wait();
  if (only_if != nullptr && *only_if == 0) return;
  constexpr int BM = 64 * MI, BN = 64 * NI;
  __shared__ __align__(16) float As[BK][BM + 4];
  __shared__ __align__(16) float Bs[BK][BN + 4];
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int jt = (J + BN - 1) / BN;              // tiles one after the other in grid.x: K has no limit of grid.y
  const int i0 = (int)(blockIdx.x / jt) * BM, j0 = (int)(blockIdx.x % jt) * BN;
  const bool vec_ok = (D & 3) == 0;
  const bool write_v = (v.base != nullptr) && (j0 == 0);
  const int lr = tid >> 2, lc = (tid & 3) * 4;   // loader: row within 64, first of 4 reduction columns

  float2 acc[4 * MI][2 * NI];
#pragma unroll
  for (int m = 0; m < 4 * MI; ++m)
#pragma unroll
    for (int n = 0; n < 2 * NI; ++n) acc[m][n] = make_float2(0.f, 0.f);

  float4 pa[MI], pb[NI];
  const float* xr = X + (size_t)(i0 + lr) * D + lc;
  const float* wr = W + (size_t)(j0 + lr) * D + lc;
  auto fetch = [&](int d0) {   // (the stores of v last: no load waits behind them)
    const int left = D - d0 - lc;
    float4 sb[PAIR ? MI : 1];
#pragma unroll
    for (int q = 0; q < NI; ++q)
      pb[q] = (j0 + lr + 64 * q < J) ? ld4_left(wr + (size_t)(64 * q) * D + d0, left, vec_ok) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < MI; ++q) {
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
      if (PAIR) sb[PAIR ? q : 0] = a;
      if (i0 + lr + 64 * q < K) {
        const float* x = xr + (size_t)(64 * q) * D + d0;
        a = ld4_left(x, left, vec_ok);
        if (PAIR) sb[PAIR ? q : 0] = ld4_left(x + (Xb - X), left, vec_ok);
      }
      pa[q] = a;
    }
    if (PAIR) {
#pragma unroll
      for (int q = 0; q < MI; ++q) {
        const float4 a = pa[q], b = sb[PAIR ? q : 0];
        pa[q] = make_float4(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z), __fsub_rn(a.w, b.w));
      }
    }
    if (write_v && d0 + lc < v.ld) {
#pragma unroll
      for (int q = 0; q < MI; ++q)
        if (i0 + lr + 64 * q < K) *reinterpret_cast<float4*>(v.row(i0 + lr + 64 * q) + (size_t)(d0 + lc) * 4) = pa[q];
    }
  };
  auto stash = [&]() {
#pragma unroll
    for (int q = 0; q < MI; ++q) {
      As[lc + 0][lr + 64 * q] = pa[q].x; As[lc + 1][lr + 64 * q] = pa[q].y;
      As[lc + 2][lr + 64 * q] = pa[q].z; As[lc + 3][lr + 64 * q] = pa[q].w;
    }
#pragma unroll
    for (int q = 0; q < NI; ++q) {
      Bs[lc + 0][lr + 64 * q] = pb[q].x; Bs[lc + 1][lr + 64 * q] = pb[q].y;
      Bs[lc + 2][lr + 64 * q] = pb[q].z; Bs[lc + 3][lr + 64 * q] = pb[q].w;
    }
  };

  const int d_lo = blockIdx.z * d_per_range, d_hi = min(D, d_lo + d_per_range);
  fetch(d_lo);
  for (int d0 = d_lo; d0 < d_hi; d0 += BK) {
    stash();
    __syncthreads();
    if (d0 + BK < d_hi) fetch(d0 + BK);
    mma_tile<MI, NI, false>(As, Bs, ty, tx, acc);
    __syncthreads();
  }
  // The factor v has pad columns [D, ldv): the last loader step wrote zeros there only when
  // D..ldv falls inside a fetched float4, which holds because ldv = D rounded up to 4.

#pragma unroll
  for (int mi = 0; mi < MI; ++mi)
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int i = i0 + mi * 64 + ty * 4 + a;
      if (i >= K) continue;
      float* zr = reinterpret_cast<float*>(z.row(i) + blockIdx.z * range_stride);
#pragma unroll
      for (int ni = 0; ni < NI; ++ni) {
        const int j = j0 + ni * 64 + tx * 4;
        if (j < z.ld)   // ld is a multiple of 4, so the whole float4 is inside the row; columns >= J hold 0
          *reinterpret_cast<float4*>(zr + j) = make_float4(acc[mi * 4 + a][ni * 2].x, acc[mi * 4 + a][ni * 2].y,
                                                           acc[mi * 4 + a][ni * 2 + 1].x, acc[mi * 4 + a][ni * 2 + 1].y);
      }
    }
}

// ---- large tiles with operands whose rows run along the OUTPUT indices: C[m][n] (+)= sum_k A[k][m] * B[k][n].
// The rows go to shared memory as they are, fetched with 16-byte asynchronous copies (zero-filled beyond the
// reduction range, M and N) through a ring of PIPE stages: one barrier per reduction step, no staging registers.
//   OUT 0 (apply):   A = factor rows u_i (k = sample, m = row j of W), B = v_i; W[m][n] -= eta * C[m][n].
//   OUT 1 (forward): A = X^T (k = feature d, m = sample i), B = W^T (n = class j), both made by a transposing
//                    pass; the products of reduction range blockIdx.z are stored to z rows (+ range stride).
constexpr int PIPE = 4;
constexpr int PIPE_STAGE_FLOATS = 2 * BK * (128 + 4);

__device__ __forceinline__ void cp_async16_zfill(float* dst_smem, const void* src, int src_bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst_smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int OUT>
__global__ void __launch_bounds__(256, 2) sgemm_pipe_kernel(float* W, RowMap u, RowMap v, int K, int J,
                                                         int D, float eta, const int* dev_status,
                                                         RowMap z, int k_per_range, long long range_stride,
                                                         const int* row_idx, const int* n_rows, const int* only_if,
                                                         int full_if) {
  chain_wait();
  if (OUT == 0 && only_if != nullptr) {
    const int word = *only_if;
    if (word == 0) return;
    if (word & full_if) row_idx = n_rows = nullptr;
  }
  constexpr int BM = 128, BN = 128;
  extern __shared__ __align__(16) float ring[];
  if (OUT == 0 && dev_status != nullptr && (*dev_status & SFB_DEV_BAD_HEADER)) return;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int j0 = blockIdx.y * BM, d0 = blockIdx.x * BN;
  const int k_lo = (OUT == 1) ? blockIdx.z * k_per_range : 0;
  // OUT 0 with a row list: the reduction runs over the listed factor rows only (the others are all zeros)
  const int k_hi = (OUT == 1) ? min(K, k_lo + k_per_range) : (n_rows != nullptr ? min(K, *n_rows) : K);
  const int lr = tid >> 5, lc = (tid & 31) * 4;   // loader: factor rows lr and lr + 8 of the step, 4 columns at lc
  // bytes of this thread's 16-byte piece that exist (the rest is zero-filled); a piece with nothing to read
  // still needs a valid aligned address: column 0 of a valid row
  const int ju = j0 + lc, dv = d0 + lc;
  const int u_bytes = max(0, min(16, (J - ju) * 4)), v_bytes = max(0, min(16, (D - dv) * 4));
  const size_t u_off = u_bytes > 0 ? (size_t)ju * 4 : 0, v_off = v_bytes > 0 ? (size_t)dv * 4 : 0;

  auto issue = [&](int stage, int k0) {
    float* As = ring + stage * PIPE_STAGE_FLOATS;
    float* Bs = As + BK * (BM + 4);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = lr + 8 * h, i = k0 + r;
      const bool ok = i < k_hi;
      const int ii = ok ? ((OUT == 0 && row_idx != nullptr) ? row_idx[i] : i) : 0;
      cp_async16_zfill(As + r * (BM + 4) + lc, u.row(ii) + u_off, ok ? u_bytes : 0);
      cp_async16_zfill(Bs + r * (BN + 4) + lc, v.row(ii) + v_off, ok ? v_bytes : 0);
    }
  };

  float2 acc[8][4];
#pragma unroll
  for (int m = 0; m < 8; ++m)
#pragma unroll
    for (int n = 0; n < 4; ++n) acc[m][n] = make_float2(0.f, 0.f);

  const int nk = (k_hi - k_lo + BK - 1) / BK;
#pragma unroll
  for (int st = 0; st < PIPE - 1; ++st) {
    if (st < nk) issue(st, k_lo + st * BK);
    cp_async_commit();
  }
  for (int kt = 0; kt < nk; ++kt) {
    cp_async_wait<PIPE - 2>();       // this thread's pieces of step kt have landed
    __syncthreads();                 // ... everybody's have, and everybody is done with step kt - 1
    const int nxt = kt + PIPE - 1;
    if (nxt < nk) issue(nxt % PIPE, k_lo + nxt * BK);
    cp_async_commit();
    const float* As = ring + (kt % PIPE) * PIPE_STAGE_FLOATS;
    mma_tile<2, 2, true>(reinterpret_cast<const float(*)[BM + 4]>(As), reinterpret_cast<const float(*)[BN + 4]>(As + BK * (BM + 4)),
                   ty, tx, acc);
  }
  cp_async_wait<0>();

  if (OUT == 1) {   // rows of z: m = sample, n = class; z.ld is a multiple of 4 and columns J .. z.ld - 1 get zeros
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const int i = j0 + mi * 64 + ty * 4 + a;
        if (i >= J) continue;
        float* zr = reinterpret_cast<float*>(z.row(i) + blockIdx.z * range_stride);
#pragma unroll
        for (int ni = 0; ni < 2; ++ni) {
          const int n = d0 + ni * 64 + tx * 4;
          if (n < z.ld)
            *reinterpret_cast<float4*>(zr + n) = make_float4(acc[mi * 4 + a][ni * 2].x, acc[mi * 4 + a][ni * 2].y,
                                                             acc[mi * 4 + a][ni * 2 + 1].x, acc[mi * 4 + a][ni * 2 + 1].y);
        }
      }
    return;
  }

  const bool vec_ok = (D & 3) == 0;
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int j = j0 + mi * 64 + ty * 4 + a;
      if (j >= J) continue;
      float* wr = W + (size_t)j * D;
#pragma unroll
      for (int ni = 0; ni < 2; ++ni) {
        const int d = d0 + ni * 64 + tx * 4;
        const float c[4] = {acc[mi * 4 + a][ni * 2].x, acc[mi * 4 + a][ni * 2].y, acc[mi * 4 + a][ni * 2 + 1].x,
                            acc[mi * 4 + a][ni * 2 + 1].y};
        if (vec_ok && d + 3 < D) {
          float4 w = *reinterpret_cast<float4*>(wr + d);
          w.x = fmaf(-eta, c[0], w.x); w.y = fmaf(-eta, c[1], w.y);
          w.z = fmaf(-eta, c[2], w.z); w.w = fmaf(-eta, c[3], w.w);
          *reinterpret_cast<float4*>(wr + d) = w;
        } else {
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (d + b < D) wr[d + b] = fmaf(-eta, c[b], wr[d + b]);
        }
      }
    }
}

// ---- 64 x 64 tiles, 4 x 4 outputs per thread, the same ring: for problems whose 128 x 128 tiles leave the chip idle.
//   OUT 0 (apply):   as above (16-byte copies; the row list too).
//   OUT 1 (forward): A = sample rows (m = sample i), B = rows of W (n = class j), both contiguous along k = feature d, read
//                    in place: 4-byte asynchronous copies transpose them on the way into shared memory (sixteen lanes
//                    take 64 contiguous bytes of a row; any D), no transposing pass.  Where the factor v is a copy of the
//                    sample rows, the blocks of a row of tiles write it from shared memory, each its share of the rows.
// Bound: the latency of a step's copies (0.9 us for 16 steps of the forward with a block per SM), hence many short
// ranges.  A step of 100 x 800, K = 160: 98 -> 19 us, of 40 x 15000, K = 800: 312 -> 132, of 300 x 3000, K = 400: 107 -> 69
// (64 x 64 tiles without a ring, 128 x 128 tiles in 512-step ranges before).
constexpr int SMALL_STAGE_FLOATS = 2 * BK * (64 + 4);

__device__ __forceinline__ void cp_async4_zfill(float* dst_smem, const void* src, int src_bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst_smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(src_bytes) : "memory");
}

struct SmallArgs {
  float* W;                 // OUT 0: updated in place; OUT 1: the B operand
  RowMap a, b;              // OUT 0: u and v rows; OUT 1: a = sample rows
  int K, M, N, ldw;         // reduction length; output rows, columns; row length of W
  float eta;
  const int* dev_status;
  RowMap z, copy;           // OUT 1: products (+ range stride); optional second destination of the sample rows
  int k_per_range;
  long long range_stride;
  const int* row_idx;       // OUT 0, optional: the factor rows to take
  const int* n_rows;
  const int* only_if;       // OUT 0, optional: do nothing where this is 0
  int full_if;              // ... and take all rows where it has a bit of this
};

template <int OUT>
__global__ void __launch_bounds__(256, 4) sgemm_small_kernel(const __grid_constant__ SmallArgs p) {
  chain_wait();
  constexpr int BT = 64;
  __shared__ __align__(16) float ring[PIPE * SMALL_STAGE_FLOATS];
  __shared__ long long a_off[OUT == 1 ? BT : 1];   // byte offset of the tile's sample rows, -1: no such row
  __shared__ long long c_off[OUT == 1 ? BT : 1];   // ... and of their copies
  const int *row_idx = p.row_idx, *n_rows = p.n_rows;
  if (OUT == 0 && p.only_if != nullptr) {
    const int word = *p.only_if;
    if (word == 0) return;
    if (word & p.full_if) row_idx = n_rows = nullptr;
  }
  if (OUT == 0 && p.dev_status != nullptr && (*p.dev_status & SFB_DEV_BAD_HEADER)) return;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, lane = tid & 31, warp = tid >> 5;
  const int nt = (p.N + BT - 1) / BT;            // tiles one after the other in grid.x: M has no limit of grid.y
  const int n_tile = (int)(blockIdx.x % nt), m0 = (int)(blockIdx.x / nt) * BT, n0 = n_tile * BT;
  const int k_lo = (OUT == 1) ? blockIdx.z * p.k_per_range : 0;
  const int k_hi = (OUT == 1) ? min(p.K, k_lo + p.k_per_range) : (n_rows != nullptr ? min(p.K, *n_rows) : p.K);
  if (OUT == 1) {
    if (tid < BT) {
      a_off[tid] = m0 + tid < p.M ? (long long)(p.a.row(m0 + tid) - p.a.base) : -1;
      c_off[tid] = p.copy.base != nullptr && m0 + tid < p.M ? (long long)(p.copy.row(m0 + tid) - p.copy.base) : -1;
    }
    __syncthreads();
  }
  auto issue = [&](int stage, int k0) {
    float* As = ring + stage * SMALL_STAGE_FLOATS;
    float* Bs = As + BK * (BT + 4);
    if (OUT == 0) {   // thread = (factor row of the step, 4 columns); nothing to read: a valid address all the same
      const int r = tid >> 4, c = (tid & 15) * 4, i = k0 + r;
      const bool ok = i < k_hi;
      const int ii = ok ? (row_idx != nullptr ? row_idx[i] : i) : 0;
      const int ub = max(0, min(16, (p.M - m0 - c) * 4)), vb = max(0, min(16, (p.N - n0 - c) * 4));
      cp_async16_zfill(As + r * (BT + 4) + c, p.a.row(ii) + (ub > 0 ? (size_t)(m0 + c) * 4 : 0), ok ? ub : 0);
      cp_async16_zfill(Bs + r * (BT + 4) + c, p.b.row(ii) + (vb > 0 ? (size_t)(n0 + c) * 4 : 0), ok ? vb : 0);
    } else {
      const int k = lane & 15, half = lane >> 4;
      const bool ok = k0 + k < k_hi;
      const char* abase = p.a.base + (ok ? (size_t)(k0 + k) * 4 : 0);
      const float* wk = p.W + (ok ? k0 + k : 0);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = q * 16 + warp * 2 + half;
        const long long off = a_off[r];
        const bool in = n0 + r < p.N;
        cp_async4_zfill(As + k * (BT + 4) + r, abase + (off >= 0 ? off : 0), ok && off >= 0 ? 4 : 0);
        cp_async4_zfill(Bs + k * (BT + 4) + r, wk + (in ? (size_t)(n0 + r) * p.ldw : 0), ok && in ? 4 : 0);
      }
    }
  };
  float2 acc[4][2];
#pragma unroll
  for (int m = 0; m < 4; ++m) acc[m][0] = acc[m][1] = make_float2(0.f, 0.f);
  const int nk = (k_hi - k_lo + BK - 1) / BK;
#pragma unroll
  for (int st = 0; st < PIPE - 1; ++st) {
    if (st < nk) issue(st, k_lo + st * BK);
    cp_async_commit();
  }
  for (int kt = 0; kt < nk; ++kt) {
    cp_async_wait<PIPE - 2>();
    __syncthreads();
    const int nxt = kt + PIPE - 1;
    if (nxt < nk) issue(nxt % PIPE, k_lo + nxt * BK);
    cp_async_commit();
    const float* As = ring + (kt % PIPE) * SMALL_STAGE_FLOATS;
    if (OUT == 1 && p.copy.base != nullptr) {   // four steps of a row per thread; rows n_tile, + nt, ...
      const int k = (tid & 3) * 4, kk = k_lo + kt * BK + k;
      for (int r = n_tile + nt * (tid >> 2); r < BT; r += nt * 64)
        if (c_off[r] >= 0 && kk < p.copy.ld)
          *reinterpret_cast<float4*>(p.copy.base + c_off[r] + (size_t)kk * 4) =
              make_float4(As[k * (BT + 4) + r], As[(k + 1) * (BT + 4) + r], As[(k + 2) * (BT + 4) + r],
                          As[(k + 3) * (BT + 4) + r]);
    }
    mma_tile<1, 1, true>(reinterpret_cast<const float(*)[BT + 4]>(As),
                         reinterpret_cast<const float(*)[BT + 4]>(As + BK * (BT + 4)), ty, tx, acc);
  }
  cp_async_wait<0>();
  const int n = n0 + tx * 4;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int i = m0 + ty * 4 + m;
    if (i >= p.M) continue;
    const float c[4] = {acc[m][0].x, acc[m][0].y, acc[m][1].x, acc[m][1].y};
    if (OUT == 1) {   // z.ld is a multiple of 4 and columns N .. z.ld - 1 get zeros
      if (n < p.z.ld)
        *reinterpret_cast<float4*>(p.z.row(i) + blockIdx.z * p.range_stride + (size_t)n * 4) = make_float4(c[0], c[1], c[2], c[3]);
      continue;
    }
    float* w = p.W + (size_t)i * p.ldw + n;
    if ((p.ldw & 3) == 0 && n + 3 < p.N) {
      float4 t = *reinterpret_cast<float4*>(w);
      t.x = fmaf(-p.eta, c[0], t.x); t.y = fmaf(-p.eta, c[1], t.y);
      t.z = fmaf(-p.eta, c[2], t.z); t.w = fmaf(-p.eta, c[3], t.w);
      *reinterpret_cast<float4*>(w) = t;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (n + e < p.N) w[e] = fmaf(-p.eta, c[e], w[e]);
    }
  }
}

// dst[c][r] = src row r, column c (R rows of C values behind a row map; dst rows ldr floats long, columns R .. ldr - 1
// zero).  `copy` (optional): the same rows also copied there, pad columns zero (the factor v = x of the MLR model).
__global__ void __launch_bounds__(256) transpose_rows_kernel(RowMap src, float* dst, int R, int C, int ldr,
                                                             RowMap copy) {
  chain_wait();
  __shared__ float tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8
#pragma unroll
  for (int q = 0; q < 32; q += 8) {
    const int r = r0 + ty + q, c = c0 + tx;
    float val = 0.f;
    if (r < R && c < C) val = reinterpret_cast<const float*>(src.row(r))[c];
    tile[ty + q][tx] = val;
    if (copy.base != nullptr && r < R && c < copy.ld) reinterpret_cast<float*>(copy.row(r))[c] = val;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 32; q += 8) {
    const int c = c0 + ty + q, r = r0 + tx;
    if (c < C && r < ldr) dst[(size_t)c * ldr + r] = tile[tx][ty + q];
  }
}

// The same transposition for rows that are whole numbers of 16-byte units (C a multiple of 4, rows 16-byte aligned):
// 64 x 64 tiles, 16-byte global loads and stores on both sides, and both operands of the forward pass in one launch
// (blockIdx.z picks the job).
struct TransposeJob {
  RowMap src;
  float* dst;
  int R, C, ldr;
  RowMap copy;
};
__global__ void __launch_bounds__(256) transpose_rows_vec_kernel(TransposeJob j0, TransposeJob j1) {
  chain_wait();
  __shared__ float tile[64][65];
  const TransposeJob& j = blockIdx.z == 0 ? j0 : j1;
  const int c0 = blockIdx.x * 64, r0 = blockIdx.y * 64;
  if (c0 >= j.C || r0 >= j.ldr) return;
  const int tq = threadIdx.x & 15, tr = threadIdx.x >> 4;   // 16 x 16
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int rr = tr + 16 * q, r = r0 + rr, c = c0 + tq * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < j.R && c < j.C) {
      v = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(j.src.row(r)) + c);
      if (j.copy.base != nullptr) *reinterpret_cast<float4*>(reinterpret_cast<float*>(j.copy.row(r)) + c) = v;
    }
    tile[rr][tq * 4] = v.x; tile[rr][tq * 4 + 1] = v.y; tile[rr][tq * 4 + 2] = v.z; tile[rr][tq * 4 + 3] = v.w;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int cc = tr + 16 * q, c = c0 + cc, r = r0 + tq * 4;
    if (c < j.C && r < j.ldr)
      *reinterpret_cast<float4*>(j.dst + (size_t)c * j.ldr + r) =
          make_float4(tile[tq * 4][cc], tile[tq * 4 + 1][cc], tile[tq * 4 + 2][cc], tile[tq * 4 + 3][cc]);
  }
}

}  // namespace

// How a forward is done, and its reduction ranges.  Estimated microseconds: 64 x 64 tiles run at 40 % of the FMA rate when
// the SMs are full and at 0.9 us per 16 steps when not; 128 x 128 tiles at 70 %, behind a transposing pass at 4.5 TB/s; a
// range's partial products go out and come back.
// Where the transposing pass does not pay (or its workspace is not there), one launch with the operands in place is the
// faster of the two others
//   - on 128 x 128 tiles, where there are enough of them and the samples meet more than one tile's width of classes: 3.28 us
//     per 16 steps for two tiles to an SM, against 0.62 for every 64 x 64 tile (1000 x 256, K = 32768: 569 -> 388 us;
//     300 x 511, K = 65536, rows of no whole 16-byte units: 721 -> 640; 100 x 64, K = 32768: 22.0 -> 17.4; but
//     64 x 256, K = 65536: 84 against 131 us);
//   - for reductions of four stages or less, which would not fill the ring (10 x 64, K = 4096: 5.7 -> 5.1 us);
//   - for pairs also where the difference, formed on the way, would cost more as a pass of its own.
ForwardF32Plan forward_f32_plan(int K, int J, int D, bool pair, int max_ks, bool transposed_ok) {
  if (step_small_fits(K, J, D)) return {F32_IN_PLACE, 1, 0.0};   // (the single-launch step repeats these sums in this order)
  const double fma_us = 128 * 1900.0;
  ForwardF32Plan best = {F32_SMALL, 1, -1.0};
  auto consider = [&](F32Route route, int tile, double rate, double step_us, double before) {
    const double tiles = (double)((K + tile - 1) / tile) * ((J + tile - 1) / tile);
    for (int ks = 1; ks <= max_ks && (ks == 1 || D / ks >= 64); ++ks) {
      const int per = ((D + ks - 1) / ks + BK - 1) / BK * BK;
      const double per_sm = (double)(long long)((tiles * ks + 147) / 148);
      const double work = per_sm * tile * tile * per / (fma_us * rate), chain = per / 16.0 * step_us;
      const double us = before + (work > chain ? work : chain) + (ks > 1 ? ks * (double)J * K * 8 / 6e6 : 0.0);
      if (best.us < 0 || us < best.us) best = {route, ks, us};
    }
  };
  consider(F32_SMALL, 64, 0.40, 0.9, 0.0);
  if (transposed_ok && K >= 128 && J >= 64 && D >= 512)
    consider(F32_TRANSPOSED, 128, 0.70, 0.9, 4.0 + (double)(J + K) * D * 8 / 4.5e6);
  if (best.route != F32_SMALL) return best;
  auto tiles_of = [&](int t) { return (long long)((K + t - 1) / t) * ((J + t - 1) / t); };
  const long long t64 = tiles_of(64), t128 = tiles_of(128);
  const double steps = (D + BK - 1) / BK, steps_ks = ((D + best.ks - 1) / best.ks + BK - 1) / BK;
  const double full = (double)((t64 * best.ks + 147) / 148) * (0.25 + 0.62 * steps_ks), chain = 0.9 * steps_ks;
  const double small_us = 0.5 + (full > chain ? full : chain) + (best.ks > 1 ? best.ks * (double)J * K * 8 / 6e6 : 0.0) +
                          (pair ? 3.0 + (double)K * D * 12 / 5e6 : 0.0);
  const double odd = (D & 3) != 0 ? 1.12 : 1.0;
  double in_place_us = small_us;
  if (J > 64 && t128 >= F32_MIN_LARGE_TILES)
    in_place_us = odd * (t128 > 148 ? (double)((t128 + 295) / 296) * (2.8 + 3.28 * steps) : 2.8 + 2.1 * steps);
  else if (pair) {
    const double f = (double)((t64 + 147) / 148) * (0.45 + 0.70 * steps), c = 0.9 * steps;
    in_place_us = 0.5 + odd * (f > c ? f : c);
  }
  if (in_place_us < small_us || (D <= 4 * BK && t64 <= 296)) return {F32_IN_PLACE, 1, in_place_us < best.us ? in_place_us : best.us};
  return best;
}

// No empty range: the finishing pass would add a partial buffer nobody wrote.
static int range_length(int D, int* ks) {
  const int per = ((D + *ks - 1) / *ks + BK - 1) / BK * BK;
  *ks = (D + per - 1) / per;
  return per;
}

static int forward_in_place(cudaStream_t s, const float* W, const float* X, const float* Xb, int K, int J, int D, RowMap z,
                            RowMap v, int per, long long split_stride, int ks, const int* only_if) {
  const int large = ((J + 127) / 128) * ((K + 127) / 128), small = ((J + 63) / 64) * ((K + 63) / 64);
  auto go = [&](auto kernel, int tiles) {
    launch_chained(kernel, dim3(tiles, 1, ks), 256, 0, s, W, X, Xb, K, J, D, z, v, per, split_stride, only_if);
  };
  if (J > 64 && (long long)large * ks >= F32_MIN_LARGE_TILES) {
    if (Xb != nullptr) go(forward_f32_kernel<2, 2, true>, large);
    else go(forward_f32_kernel<2, 2, false>, large);
  } else {
    if (Xb != nullptr) go(forward_f32_kernel<1, 1, true>, small);
    else go(forward_f32_kernel<1, 1, false>, small);
  }
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

int launch_forward_f32(cudaStream_t s, const float* W, const float* X, const float* Xb, int K, int J, int D, RowMap z,
                       RowMap v, RowMap part, long long split_stride, int ks, int* nsplit_out) {
  const int per = range_length(D, &ks);
  if (nsplit_out != nullptr) *nsplit_out = ks;
  return forward_in_place(s, W, X, Xb, K, J, D, ks > 1 ? part : z, v, per, split_stride, ks, nullptr);
}

int launch_forward_f32_if(cudaStream_t s, const float* W, const float* X, const float* Xb, int K, int J, int D, RowMap z,
                          long long split_stride, int ks, const int* only_if) {
  const int per = ((D + ks - 1) / ks + BK - 1) / BK * BK;
  return forward_in_place(s, W, X, Xb, K, J, D, z, RowMap(), per, split_stride, ks, only_if);
}

int launch_forward_f32_small(cudaStream_t s, const float* W, RowMap src, RowMap copy, int K, int J, int D, RowMap z,
                             RowMap part, long long split_stride, int ks, int* nsplit_out) {
  SmallArgs p = {};
  p.k_per_range = range_length(D, &ks);
  p.W = const_cast<float*>(W);
  p.a = src; p.copy = copy;
  p.K = D; p.M = K; p.N = J; p.ldw = D;
  p.z = ks > 1 ? part : z;
  p.range_stride = split_stride;
  *nsplit_out = ks;
  launch_chained(sgemm_small_kernel<1>, dim3(((J + 63) / 64) * ((K + 63) / 64), 1, ks), 256, 0, s, p);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

int launch_apply_f32(cudaStream_t s, float* W, RowMap u, RowMap v, int K, int J, int D, float eta,
                     const int* dev_status, const int* row_idx, const int* n_rows, const int* only_if, int full_if) {
  const long long big_tiles = (long long)((J + 127) / 128) * ((D + 127) / 128);
  if (big_tiles >= 148) {
    dim3 grid((D + 127) / 128, (J + 127) / 128);
    static PerDeviceOnce attr_once;
    if (!set_up_device(attr_once, [] { return allow_smem(sgemm_pipe_kernel<0>, PIPE * PIPE_STAGE_FLOATS * 4); }))
      return SFB_ERR_CUDA;
    launch_chained(sgemm_pipe_kernel<0>, grid, 256, PIPE * PIPE_STAGE_FLOATS * 4, s, W, u, v, K, J, D, eta, dev_status, RowMap(), 0, 0,
                                                                         row_idx, n_rows, only_if, full_if);
  } else {
    SmallArgs p = {};
    p.W = W;
    p.a = u; p.b = v;
    p.K = K; p.M = J; p.N = D; p.ldw = D;
    p.eta = eta;
    p.dev_status = dev_status;
    p.row_idx = row_idx; p.n_rows = n_rows; p.only_if = only_if; p.full_if = full_if;
    launch_chained(sgemm_small_kernel<0>, ((D + 63) / 64) * ((J + 63) / 64), 256, 0, s, p);
  }
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

// Forward contraction through transposed copies of its operands (workspace: xt [D][ldk], wt [D][ldj] floats with
// ldk, ldj = K, J rounded up to 4): two bandwidth-bound transposing passes, then the pipelined kernel above, which
// runs faster than the kernel that transposes through registers.  src: the operand rows a_i (X rows, or pair
// differences already written as the factor v); copy: optional second destination of those rows (v = x).
long long forward_f32_nn_workspace_floats(int K, int J, int D) {
  return (long long)D * (((K + 3) & ~3) + ((J + 3) & ~3));
}

int launch_forward_f32_nn(cudaStream_t s, const float* W, RowMap src, RowMap copy, int K, int J, int D, float* ws,
                          RowMap z, RowMap part, long long split_stride, int ks, int* nsplit_out) {
  const int ldk = (K + 3) & ~3, ldj = (J + 3) & ~3;
  float* xt = ws;
  float* wt = ws + (size_t)D * ldk;
  RowMap wrows;
  wrows.base = const_cast<char*>(reinterpret_cast<const char*>(W));
  wrows.worker_stride = 0; wrows.ld = D; wrows.B = J > 0 ? J : 1; wrows.es = 4;
  const bool vec = (D & 3) == 0 && (src.ld & 3) == 0 && (reinterpret_cast<uintptr_t>(src.base) & 15) == 0 &&
                   (src.worker_stride & 15) == 0 && (reinterpret_cast<uintptr_t>(W) & 15) == 0 &&
                   (copy.base == nullptr || ((copy.ld & 3) == 0 && (reinterpret_cast<uintptr_t>(copy.base) & 15) == 0 &&
                                             (copy.worker_stride & 15) == 0));
  int transposes = 2;
  if (vec) {   // both operands in one launch
    TransposeJob jx, jw;
    jx.src = src; jx.dst = xt; jx.R = K; jx.C = D; jx.ldr = ldk; jx.copy = copy;
    jw.src = wrows; jw.dst = wt; jw.R = J; jw.C = D; jw.ldr = ldj; jw.copy = RowMap();
    const int ry = ((ldk > ldj ? ldk : ldj) + 63) / 64;
    launch_chained(transpose_rows_vec_kernel, dim3((D + 63) / 64, ry, 2), 256, 0, s, jx, jw);
    transposes = 1;
  } else {
    launch_chained(transpose_rows_kernel, dim3((D + 31) / 32, (ldk + 31) / 32), 256, 0, s, src, xt, K, D, ldk, copy);
    launch_chained(transpose_rows_kernel, dim3((D + 31) / 32, (ldj + 31) / 32), 256, 0, s, wrows, wt, J, D, ldj, RowMap());
  }
  const int per = range_length(D, &ks);
  *nsplit_out = ks;
  RowMap a, b;
  a.base = reinterpret_cast<char*>(xt); a.worker_stride = 0; a.ld = ldk; a.B = D; a.es = 4;
  b.base = reinterpret_cast<char*>(wt); b.worker_stride = 0; b.ld = ldj; b.B = D; b.es = 4;
  static PerDeviceOnce attr_once;
  if (!set_up_device(attr_once, [] { return allow_smem(sgemm_pipe_kernel<1>, PIPE * PIPE_STAGE_FLOATS * 4); }))
    return SFB_ERR_CUDA;
  // rows of the output tile = samples (M = K), columns = classes (N = J), reduction over the D features
  dim3 grid((J + 127) / 128, (K + 127) / 128, ks);
  launch_chained(sgemm_pipe_kernel<1>, grid, 256, PIPE * PIPE_STAGE_FLOATS * 4, s, nullptr, a, b, D, K, ldj, 0.f, nullptr,
                                                                       ks > 1 ? part : z, per, split_stride, nullptr, nullptr, nullptr, 0);
  return cudaGetLastError() == cudaSuccess ? transposes + 1 : SFB_ERR_CUDA;
}

}  // namespace sfb
