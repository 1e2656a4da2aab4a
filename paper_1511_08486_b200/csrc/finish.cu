// Bandwidth-bound passes of the factor computation: the model epilogues that turn the products
// z_i = W a_i into the factor u_i, row copies, and the fp32 -> bf16 cast of W.
//
//   MLR  u_i = softmax(z_i) - onehot(y_i)   (chain rule on the multiclass logistic loss; Section 2.1)
//   DML  u_i = +z_i (similar pair) | -z_i * [|z_i|^2 < margin] (dissimilar pair)   (Section 2, DML)
//
// One thread block per sample row; the row is staged once in shared memory (when it fits) so HBM
// sees one read and one write per value; reductions over the J entries use warp shuffles.
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace sfb {
namespace {

constexpr int ROW_CACHE_FLOATS = 48 * 1024;   // 192 KB of dynamic shared memory

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Block-wide reductions with a fixed combination order (bit-reproducible).
__device__ float block_max(float v, float* red) {
  v = warp_max(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  float r = (l < (int)(blockDim.x >> 5)) ? red[l] : -INFINITY;
  return warp_max(r);
}
__device__ float block_sum(float v, float* red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  float r = (l < (int)(blockDim.x >> 5)) ? red[l] : 0.f;
  return warp_sum(r);
}

// Four products starting at column j: the sum, in split order, of the partial products of a reduction
// that the GEMM cut in `nsplit` ranges (partial s lives `stride` floats after partial s - 1).
__device__ __forceinline__ float4 ldz4(const float* zr, int j, int nsplit, long long stride) {
  float4 t = *reinterpret_cast<const float4*>(zr + j);
  for (int s = 1; s < nsplit; ++s) {
    const float4 q = *reinterpret_cast<const float4*>(zr + s * stride + j);
    t.x += q.x; t.y += q.y; t.z += q.z; t.w += q.w;
  }
  return t;
}

// Stores 4 consecutive values starting at column j (j % 4 == 0, j + 3 < ld).
__device__ __forceinline__ void store_u4(char* row, int j, float4 v, int es) {
  if (es == 4) {
    *reinterpret_cast<float4*>(row + (size_t)j * 4) = v;
  } else {
    __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    uint2 p;
    p.x = *reinterpret_cast<uint32_t*>(&lo);
    p.y = *reinterpret_cast<uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(row + (size_t)j * 2) = p;
  }
}

// 16 bytes of row i at unit q, copied from src to dst (columns from `cols` on as zeros), with their correction operands.
__device__ __forceinline__ void copy_unit(const RowMap& src, const RowMap& dst, int i, int q, int cols, const CorrOut& corr) {
  const int per = 16 / dst.es, c = q * per;
  uint4 val = make_uint4(0u, 0u, 0u, 0u);
  if (c < cols && c < src.ld) {
    val = *reinterpret_cast<const uint4*>(src.row(i) + (size_t)q * 16);
    if (c + per > cols) {   // mask the tail beyond `cols`
      if (dst.es == 4) {
        uint32_t* w = reinterpret_cast<uint32_t*>(&val);
        for (int e = 0; e < 4; ++e)
          if (c + e >= cols) w[e] = 0u;
      } else {
        uint16_t* h = reinterpret_cast<uint16_t*>(&val);
        for (int e = 0; e < 8; ++e)
          if (c + e >= cols) h[e] = 0;
      }
    }
  }
  *reinterpret_cast<uint4*>(dst.row(i) + (size_t)q * 16) = val;
  if (corr.mn != nullptr || corr.km != nullptr)   // fp32 rows only (the compensated path)
    corr_store4(corr, i, dst.B, c, make_float4(__uint_as_float(val.x), __uint_as_float(val.y), __uint_as_float(val.z),
                                               __uint_as_float(val.w)));
}

// The first header_blocks blocks of a finishing pass write the header and the directory; the others take a row each, and
// row i of the copy.  (In the block of a row they would be on the pass's critical path, and with many workers the longest
// part of it: 4096 workers of one sample, 64 x 512 in tf32: 77.9 us a step, 53.2 with blocks of their own.)
__device__ __forceinline__ bool header_block(const FinishExtra& x) {
  if (x.take_bad != nullptr && blockIdx.x == 0 && threadIdx.x == 0) {
    if (x.give_bad != nullptr) *x.give_bad = *x.take_bad;
    *x.take_bad = 0;
  }
  if ((int)blockIdx.x >= x.header_blocks) return false;
  write_header(x.commit, blockIdx.x * blockDim.x + threadIdx.x, x.header_blocks * blockDim.x);
  return true;
}
int header_blocks(const FinishExtra& x) {
  if (x.commit.buf == nullptr) return 0;
  const long long words = (long long)(x.commit.h.streams_off / 4);
  return (int)(words / 2048 < 1 ? 1 : (words / 2048 > 148 ? 148 : words / 2048));
}
__device__ __forceinline__ void finish_extra(const FinishExtra& x, int i) {
  if (x.dst.base != nullptr)
    for (int q = threadIdx.x; q < x.dst.ld * x.dst.es / 16; q += blockDim.x) copy_unit(x.src, x.dst, i, q, x.cols, CorrOut());
}

// Row i of u written: does it hold a nonzero wire value?  (any: this thread's values do)
__device__ __forceinline__ void flag_row(const FinishExtra& x, int i, bool any) {
  if (x.nonzero == nullptr) return;
  any = __syncthreads_or(any);
  if (threadIdx.x == 0) x.nonzero[i] = any ? 1 : 0;
}
__device__ __forceinline__ bool wire_nonzero4(const float4& t, int es) {
  if (es == 4) return t.x != 0.f || t.y != 0.f || t.z != 0.f || t.w != 0.f;
  const __nv_bfloat162 lo = __floats2bfloat162_rn(t.x, t.y), hi = __floats2bfloat162_rn(t.z, t.w);
  return ((*reinterpret_cast<const uint32_t*>(&lo) | *reinterpret_cast<const uint32_t*>(&hi)) & 0x7fff7fffu) != 0u;
}

// z rows are fp32 with ld a multiple of 4; values beyond J inside the last float4 are ignored.
template <int T, int BLOCKS>
__global__ void __launch_bounds__(T, BLOCKS) finish_mlr_kernel(RowMap z, RowMap u, const int32_t* labels,
                                                                 int K, int J, int cache_floats, int* dev_status, int nsplit, long long zstride,
                                                                 float* dual, float sdca_step, CorrOut corr, const __grid_constant__ FinishExtra extra) {
  if (extra.next_early) chain_next();
  chain_wait();
  extern __shared__ __align__(16) float cache[];
  __shared__ float red[32];
  if (header_block(extra)) return;
  const int i = blockIdx.x - extra.header_blocks;
  if (i >= K) return;
  const int y = labels[i];   // (early: its latency passes beside the row's)
  finish_extra(extra, i);
  const float* zr = reinterpret_cast<const float*>(z.row(i));
  char* ur = u.row(i);
  const int J4 = (J + 3) >> 2;
  const bool cached = (J4 * 4) <= cache_floats;
  const float kLog2e = 1.4426950408889634f;

  float m = -INFINITY;
  for (int q = threadIdx.x; q < J4; q += T) {
    float4 t = ldz4(zr, q * 4, nsplit, zstride);
    const int j = q * 4;
    if (j + 1 >= J) t.y = -INFINITY;
    if (j + 2 >= J) t.z = -INFINITY;
    if (j + 3 >= J) t.w = -INFINITY;
    if (cached) *reinterpret_cast<float4*>(cache + j) = t;
    m = fmaxf(fmaxf(fmaxf(m, t.x), fmaxf(t.y, t.z)), t.w);
  }
  m = block_max(m, red);

  float s = 0.f;
  const float mb = m * kLog2e;
  for (int q = threadIdx.x; q < J4; q += T) {
    const int j = q * 4;
    float4 t;
    if (cached) {
      t = *reinterpret_cast<const float4*>(cache + j);
    } else {
      t = ldz4(zr, j, nsplit, zstride);
      if (j + 1 >= J) t.y = -INFINITY;
      if (j + 2 >= J) t.z = -INFINITY;
      if (j + 3 >= J) t.w = -INFINITY;
    }
    t.x = exp2f(fmaf(t.x, kLog2e, -mb)); t.y = exp2f(fmaf(t.y, kLog2e, -mb));
    t.z = exp2f(fmaf(t.z, kLog2e, -mb)); t.w = exp2f(fmaf(t.w, kLog2e, -mb));
    if (cached) *reinterpret_cast<float4*>(cache + j) = t;
    s += (t.x + t.y) + (t.z + t.w);
  }
  s = block_sum(s, red);
  const float inv = 1.0f / s;

  const bool bad = (y < 0) || (y >= J);
  if (bad && threadIdx.x == 0) atomicOr(dev_status, SFB_DEV_BAD_LABEL);
  const int ld4 = u.ld >> 2;   // u.ld is a multiple of 4 (fp32) or 8 (bf16)
  bool any = false;
  for (int q = threadIdx.x; q < ld4; q += T) {
    const int j = q * 4;
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    if (q < J4 && !bad) {
      if (cached) {
        t = *reinterpret_cast<const float4*>(cache + j);
      } else {
        t = ldz4(zr, j, nsplit, zstride);
        t.x = exp2f(fmaf(t.x, kLog2e, -mb)); t.y = exp2f(fmaf(t.y, kLog2e, -mb));
        t.z = exp2f(fmaf(t.z, kLog2e, -mb)); t.w = exp2f(fmaf(t.w, kLog2e, -mb));
      }
      t.x *= inv; t.y *= inv; t.z *= inv; t.w *= inv;
      if (y == j) t.x -= 1.f;
      if (y == j + 1) t.y -= 1.f;
      if (y == j + 2) t.z -= 1.f;
      if (y == j + 3) t.w -= 1.f;
      if (j + 1 >= J) t.y = 0.f;
      if (j + 2 >= J) t.z = 0.f;
      if (j + 3 >= J) t.w = 0.f;
    }
    if (dual != nullptr && q < J4) t = sdca_step4(dual + (size_t)i * (J4 * 4), j, J, t, sdca_step, bad);
    store_u4(ur, j, t, u.es);
    any |= wire_nonzero4(t, u.es);
    if (corr.mn != nullptr) corr_store4(corr, i, u.B, j, t);
  }
  flag_row(extra, i, any);
}

template <int T, int BLOCKS>
__global__ void __launch_bounds__(T, BLOCKS) finish_dml_kernel(RowMap z, RowMap u, const uint8_t* similar,
                                                                 float margin, int K, int J, int cache_floats, int nsplit, long long zstride,
                                                                 uint8_t* active, CorrOut corr, const __grid_constant__ FinishExtra extra) {
  if (extra.next_early) chain_next();
  chain_wait();
  extern __shared__ __align__(16) float cache[];
  __shared__ float red[32];
  if (header_block(extra)) return;
  const int i = blockIdx.x - extra.header_blocks;
  if (i >= K) return;
  const bool sim = similar[i] != 0;   // (early: its latency passes beside the row's)
  finish_extra(extra, i);
  const float* zr = reinterpret_cast<const float*>(z.row(i));
  char* ur = u.row(i);
  const int J4 = (J + 3) >> 2;
  const bool cached = (J4 * 4) <= cache_floats;

  float n = 0.f;
  for (int q = threadIdx.x; q < J4; q += T) {
    float4 t = ldz4(zr, q * 4, nsplit, zstride);
    const int j = q * 4;
    if (j + 1 >= J) t.y = 0.f;
    if (j + 2 >= J) t.z = 0.f;
    if (j + 3 >= J) t.w = 0.f;
    if (cached) *reinterpret_cast<float4*>(cache + j) = t;
    n += (t.x * t.x + t.y * t.y) + (t.z * t.z + t.w * t.w);
  }
  n = block_sum(n, red);
  const float g = sim ? 1.f : ((n < margin) ? -1.f : 0.f);   // strict hinge: inactive at equality
  if (active != nullptr && threadIdx.x == 0) active[i] = (g != 0.f) ? 1 : 0;   // u_i is all zeros otherwise

  const int ld4 = u.ld >> 2;
  bool any = false;
  for (int q = threadIdx.x; q < ld4; q += T) {
    const int j = q * 4;
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    if (q < J4 && g != 0.f) {
      t = cached ? *reinterpret_cast<const float4*>(cache + j) : ldz4(zr, j, nsplit, zstride);
      t.x *= g; t.y *= g; t.z *= g; t.w *= g;
      if (j + 1 >= J) t.y = 0.f;
      if (j + 2 >= J) t.z = 0.f;
      if (j + 3 >= J) t.w = 0.f;
    }
    store_u4(ur, j, t, u.es);
    any |= wire_nonzero4(t, u.es);
    if (corr.mn != nullptr) corr_store4(corr, i, u.B, j, t);
  }
  flag_row(extra, i, any);
}

// Second half of the fused multiclass-logistic epilogue.  The forward GEMM left e[j] = exp(z[j] - m_p)
// in the u row (p = the half tile that holds class j) and (m_p, s_p = sum of those exps) per part.
// Here: m = max_p m_p, s = sum_p s_p exp(m_p - m), u[j] = e[j] * exp(m_p - m) / s - [j == label], in place.
template <int ES>
__global__ void __launch_bounds__(256) finish_mlr_fused_kernel(RowMap u, const float2* stats, int n_parts,
                                                               int part_cols, const int32_t* labels, int K,
                                                               int J, int* dev_status, float* dual,
                                                               float sdca_step, const __grid_constant__ FinishExtra extra) {
  if (extra.next_early) chain_next();
  chain_wait();
  extern __shared__ float scale[];   // [n_parts]
  __shared__ float red[32];
  if (header_block(extra)) return;
  const int i = blockIdx.x - extra.header_blocks;
  if (i >= K) return;
  const int y = labels[i];   // (early: its latency passes beside the row's)
  finish_extra(extra, i);
  const float kLog2e = 1.4426950408889634f;
  const float2* st = stats + (size_t)i * n_parts;
  float m = -INFINITY;
  for (int q = threadIdx.x; q < n_parts; q += 256) m = fmaxf(m, st[q].x);
  m = block_max(m, red);
  float ssum = 0.f;
  for (int q = threadIdx.x; q < n_parts; q += 256) {
    const float2 ps = st[q];
    const float f = (ps.x == -INFINITY) ? 0.f : exp2f((ps.x - m) * kLog2e);
    scale[q] = f;
    ssum += ps.y * f;
  }
  ssum = block_sum(ssum, red);   // also orders the writes of scale[] before the reads below
  const float inv = 1.0f / ssum;
  const bool bad = (y < 0) || (y >= J);
  if (bad && threadIdx.x == 0) atomicOr(dev_status, SFB_DEV_BAD_LABEL);
  char* ur = u.row(i);
  constexpr int PER = 16 / ES;          // values per 16-byte unit (part_cols is a multiple of it)
  const int units = u.ld / PER;
  bool any = false;
  for (int q = threadIdx.x; q < units; q += 256) {
    const int j = q * PER;
    uint4 raw = *reinterpret_cast<const uint4*>(ur + (size_t)q * 16);
    float vals[PER];
    if (ES == 4) {
      const float* f = reinterpret_cast<const float*>(&raw);
#pragma unroll
      for (int e = 0; e < PER; ++e) vals[e] = f[e];
    } else {
      const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&raw);
#pragma unroll
      for (int e = 0; e < PER; ++e) vals[e] = __bfloat162float(h[e]);
    }
    const float f = (j < J && !bad) ? scale[j / part_cols] * inv : 0.f;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      float r = vals[e] * f;
      if (j + e == y) r -= 1.f;
      if (j + e >= J || bad) r = 0.f;
      vals[e] = r;
    }
    if (dual != nullptr && j < J) {   // SDCA: the factor becomes the dual step, the dual variables move by it
      float* drow = dual + (size_t)i * (((J + 3) >> 2) * 4);
#pragma unroll
      for (int e4 = 0; e4 < PER; e4 += 4) {
        if (j + e4 < J) {
          const float4 du = sdca_step4(drow, j + e4, J, make_float4(vals[e4], vals[e4 + 1], vals[e4 + 2], vals[e4 + 3]),
                                       sdca_step, bad);
          vals[e4] = du.x; vals[e4 + 1] = du.y; vals[e4 + 2] = du.z; vals[e4 + 3] = du.w;
        }
      }
    }
    if (ES == 4) {
      float* f4 = reinterpret_cast<float*>(&raw);
#pragma unroll
      for (int e = 0; e < PER; ++e) f4[e] = vals[e];
    } else {
      __nv_bfloat16* h = reinterpret_cast<__nv_bfloat16*>(&raw);
#pragma unroll
      for (int e = 0; e < PER; ++e) h[e] = __float2bfloat16_rn(vals[e]);
    }
    any |= ((raw.x | raw.y | raw.z | raw.w) & (ES == 4 ? 0x7fffffffu : 0x7fff7fffu)) != 0u;
    *reinterpret_cast<uint4*>(ur + (size_t)q * 16) = raw;
  }
  flag_row(extra, i, any);
}

// Unit-ball projection of the columns of W (sparse-coding prox).  A cluster of CTAs owns a slab of 32 consecutive
// columns: eight lanes hold a row's 128-byte segment, a CTA takes every 32nd row of its share of the rows and keeps up to
// PROX_HELD of them per thread in registers between the norm and the rescaling (rows beyond that are read again, from
// L2).  Squared norms are combined in a fixed order: rows of a thread, threads, CTAs.  Units of four columns none of
// which is rescaled are not written.
// shadow (optional): W's correction operand of the compensated tf32 path, [row][atom of 32 columns][32 values | 32
// remainders]; a slab is one atom, so its line is rewritten from the registers that hold the new W.
// Bound: HBM, W read once and written once.  (One block per slab with one 4-byte load in flight per thread and a second
// pass over the slab took 206 us at 4096 x 10000, 1.6 TB/s on its 328 MB; this takes 61 us, 5.4 TB/s, and as long with
// the 164 MB of the operand, whose stand-alone rebuild before the next forward pass took 45 us.)
constexpr int PROX_HELD = 16, PROX_THREADS = 256, PROX_ROWS = PROX_THREADS / 8;
template <bool VEC>
__global__ void __launch_bounds__(PROX_THREADS, VEC ? 2 : 1) prox_unit_columns_kernel(float* W, int J, int D,
                                                                            int rows_per_cta, __nv_bfloat16* shadow) {
  chain();
  __shared__ float4 part[PROX_ROWS][9];
  __shared__ float cta_sum[32];
  cg::cluster_group cluster = cg::this_cluster();
  const int lq = threadIdx.x & 7, lr = threadIdx.x >> 3;
  const int ctas = cluster.num_blocks(), slab = blockIdx.x / ctas;
  const int d = slab * 32 + lq * 4;
  const int j_lo = (int)cluster.block_rank() * rows_per_cta, j_hi = min(J, j_lo + rows_per_cta);
  auto load = [&](int j) {
    const float* w = W + (size_t)j * D + d;
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    if (VEC) {
      if (d < D) t = *reinterpret_cast<const float4*>(w);
    } else {
      if (d < D) t.x = w[0];
      if (d + 1 < D) t.y = w[1];
      if (d + 2 < D) t.z = w[2];
      if (d + 3 < D) t.w = w[3];
    }
    return t;
  };
  float4 held[PROX_HELD];
#pragma unroll
  for (int q = 0; q < PROX_HELD; ++q) {
    const int j = j_lo + lr + q * PROX_ROWS;
    held[q] = j < j_hi ? load(j) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add = [&](const float4& t) {
    acc.x = fmaf(t.x, t.x, acc.x); acc.y = fmaf(t.y, t.y, acc.y);
    acc.z = fmaf(t.z, t.z, acc.z); acc.w = fmaf(t.w, t.w, acc.w);
  };
#pragma unroll
  for (int q = 0; q < PROX_HELD; ++q) add(held[q]);
  for (int j = j_lo + lr + PROX_HELD * PROX_ROWS; j < j_hi; j += PROX_ROWS) add(load(j));
  part[lr][lq] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    float n = 0.f;
#pragma unroll
    for (int r = 0; r < PROX_ROWS; ++r) n += reinterpret_cast<const float*>(&part[r][0])[threadIdx.x];
    cta_sum[threadIdx.x] = n;
  }
  cluster.sync();
  float sc[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float n2 = 0.f;
    for (int c = 0; c < ctas; ++c) n2 += cluster.map_shared_rank(cta_sum, c)[lq * 4 + e];
    sc[e] = (n2 > 1.0f) ? 1.0f / sqrtf(n2) : 1.0f;
  }
  cluster.sync();   // nobody leaves while its sums may still be read
  if (sc[0] == 1.0f && sc[1] == 1.0f && sc[2] == 1.0f && sc[3] == 1.0f) return;
  const int atoms = gridDim.x / ctas;
  auto store = [&](int j, float4 t) {
    t.x *= sc[0]; t.y *= sc[1]; t.z *= sc[2]; t.w *= sc[3];
    float* w = W + (size_t)j * D + d;
    if (VEC) {
      if (d < D) *reinterpret_cast<float4*>(w) = t;
    } else {
      if (d < D) w[0] = t.x;
      if (d + 1 < D) w[1] = t.y;
      if (d + 2 < D) w[2] = t.z;
      if (d + 3 < D) w[3] = t.w;
    }
    if (VEC && shadow != nullptr && d < D) {
      uint2 val, rem;
      split4(t, val, rem);
      uint2* dst = reinterpret_cast<uint2*>(shadow + ((size_t)j * atoms + slab) * 64) + lq;
      dst[0] = val;
      dst[8] = rem;
    }
  };
#pragma unroll
  for (int q = 0; q < PROX_HELD; ++q) {
    const int j = j_lo + lr + q * PROX_ROWS;
    if (j < j_hi) store(j, held[q]);
  }
  for (int j = j_lo + lr + PROX_HELD * PROX_ROWS; j < j_hi; j += PROX_ROWS) store(j, load(j));
}

// 16-byte-vectorised row copy; rows are whole numbers of 16-byte units on both sides.
__global__ void __launch_bounds__(256) copy_rows_kernel(RowMap src, RowMap dst, int K, int cols, CorrOut corr) {
  chain();
  const int units_dst = dst.ld * dst.es / 16;
  const long long total = (long long)K * units_dst;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x)
    copy_unit(src, dst, (int)(g / units_dst), (int)(g % units_dst), cols, corr);
}

// u and v rows into their streams, and the header, in one launch.
__global__ void __launch_bounds__(256) pack_rows_kernel(RowMap u_src, RowMap u_dst, int J, RowMap v_src, RowMap v_dst, int D,
                                                        int K, const __grid_constant__ Commit commit) {
  chain();
  if (blockIdx.x == 0) write_header(commit, threadIdx.x, 256);
  const int uu = u_dst.ld * u_dst.es / 16, units = uu + v_dst.ld * v_dst.es / 16;
  const long long total = (long long)K * units;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(g / units), q = (int)(g % units);
    if (q < uu) copy_unit(u_src, u_dst, i, q, J, CorrOut());
    else copy_unit(v_src, v_dst, i, q - uu, D, CorrOut());
  }
}

// v rows = Xa - Xb (one fp32 subtraction per element), pad columns zero; 4 values per thread.
__global__ void __launch_bounds__(256) diff_rows_kernel(const float* Xa, const float* Xb, RowMap v,
                                                        int K, int D, CorrOut corr) {
  chain();
  const int units = v.ld >> 2;
  const long long total = (long long)K * units;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(g / units), c = (int)(g % units) * 4;
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c + 3 < D && (D & 3) == 0) {
      const float4 a = *reinterpret_cast<const float4*>(Xa + (size_t)i * D + c);
      const float4 b = *reinterpret_cast<const float4*>(Xb + (size_t)i * D + c);
      r = make_float4(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z), __fsub_rn(a.w, b.w));
    } else {
      float* e = reinterpret_cast<float*>(&r);
      for (int q = 0; q < 4; ++q)
        if (c + q < D) e[q] = __fsub_rn(Xa[(size_t)i * D + c + q], Xb[(size_t)i * D + c + q]);
    }
    *reinterpret_cast<float4*>(v.row(i) + (size_t)c * 4) = r;
    if (corr.mn != nullptr || corr.km != nullptr) corr_store4(corr, i, v.B, c, r);
  }
}

__global__ void __launch_bounds__(256) cast_bf16_kernel(const float* W, __nv_bfloat16* Wb,
                                                        long long n4) {
  chain();
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < n4; g += (long long)gridDim.x * blockDim.x) {
    const float4 t = reinterpret_cast<const float4*>(W)[g];
    __nv_bfloat162 lo = __floats2bfloat162_rn(t.x, t.y), hi = __floats2bfloat162_rn(t.z, t.w);
    uint2 p;
    p.x = *reinterpret_cast<uint32_t*>(&lo);
    p.y = *reinterpret_cast<uint32_t*>(&hi);
    reinterpret_cast<uint2*>(Wb)[g] = p;
  }
}

// Threads and blocks per SM of a finishing pass.  Long rows take a whole SM's worth of shared memory, so one block must
// supply all the memory parallelism.  Other rows take 256 threads and the registers that keep a thread's loads of a row, or
// of its partial products, in flight together, unless there is nothing of the kind (up to 1024 values, one range) and more
// rows than two waves of such blocks: then the number of rows at work counts, and the registers are held down for it, in
// half-size blocks where 512 values suffice (same order of the sums: the other warps would add zeros).
// 10 x 64, K = 65536: 248 us for the factors with 63 registers a thread and 256 threads, 100 with 40 and 128; but 200 x 8000,
// one sample in 16 ranges: 13.9 us with 63, 17.3 with 40.
template <typename F>
int by_rows(int K, int J, int nsplit, F&& go) {
  if (J >= 8192) return go(std::integral_constant<int, 1024>(), std::integral_constant<int, 1>());
  if (J > 1024 || nsplit > 1 || K <= 8 * 148) return go(std::integral_constant<int, 256>(), std::integral_constant<int, 4>());
  if (J > 512) return go(std::integral_constant<int, 256>(), std::integral_constant<int, 6>());
  return go(std::integral_constant<int, 128>(), std::integral_constant<int, 12>());
}

int fin_cache_floats(int J) {
  const int need = ((J + 3) / 4) * 4;
  return need <= ROW_CACHE_FLOATS ? need : 0;
}

}  // namespace

int launch_finish_mlr(cudaStream_t s, RowMap z, RowMap u, const int32_t* labels, int K, int J, int* dev_status,
                      int nsplit, long long split_stride_bytes, float* dual, float sdca_step, CorrOut corr,
                      const FinishExtra& extra_in) {
  FinishExtra extra = extra_in;
  extra.header_blocks = header_blocks(extra);
  const int cf = fin_cache_floats(J);
  return by_rows(K, J, nsplit, [&](auto threads, auto blocks) -> int {
    auto kernel = finish_mlr_kernel<threads(), blocks()>;
    static PerDeviceOnce attr_once;
    if (threads() == 1024 && !set_up_device(attr_once, [&] { return allow_smem(kernel, ROW_CACHE_FLOATS * 4); }))
      return SFB_ERR_CUDA;
    launch_chained(kernel, K + extra.header_blocks, threads(), (size_t)cf * 4, s, z, u, labels, K, J, cf, dev_status, nsplit, split_stride_bytes / 4,
                   dual, sdca_step, corr, extra);
    return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
  });
}

// idx[0 .. n) = the samples i < K with active[i] != 0, in ascending order; *n_out = n.  One block, ordered.
__global__ void __launch_bounds__(1024) compact_active_kernel(const uint8_t* active, int K, int* idx,
                                                              int* n_out) {
  chain_wait();
  __shared__ int warp_cnt[32];
  __shared__ int base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) base = 0;
  __syncthreads();
  for (int start = 0; start < K; start += 1024) {
    const int i = start + threadIdx.x;
    const bool f = i < K && active[i] != 0;
    const unsigned m = __ballot_sync(0xffffffffu, f);
    const int before = __popc(m & ((1u << lane) - 1u));
    if (lane == 0) warp_cnt[warp] = __popc(m);
    __syncthreads();
    int off = 0;
    for (int w = 0; w < warp; ++w) off += warp_cnt[w];
    if (f) idx[base + off + before] = i;
    __syncthreads();
    if (threadIdx.x == 0) {
      int t = 0;
      for (int w = 0; w < 32; ++w) t += warp_cnt[w];
      base += t;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *n_out = base;
}

int launch_compact_active(cudaStream_t s, const uint8_t* active, int K, int* idx, int* n_out) {
  launch_chained(compact_active_kernel, 1, 1024, 0, s, active, K, idx, n_out);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

int launch_finish_dml(cudaStream_t s, RowMap z, RowMap u, const uint8_t* similar, float margin, int K, int J,
                      int nsplit, long long split_stride_bytes, uint8_t* active, CorrOut corr, const FinishExtra& extra_in) {
  FinishExtra extra = extra_in;
  extra.header_blocks = header_blocks(extra);
  const int cf = fin_cache_floats(J);
  return by_rows(K, J, nsplit, [&](auto threads, auto blocks) -> int {
    auto kernel = finish_dml_kernel<threads(), blocks()>;
    static PerDeviceOnce attr_once;
    if (threads() == 1024 && !set_up_device(attr_once, [&] { return allow_smem(kernel, ROW_CACHE_FLOATS * 4); }))
      return SFB_ERR_CUDA;
    launch_chained(kernel, K + extra.header_blocks, threads(), (size_t)cf * 4, s, z, u, similar, margin, K, J, cf, nsplit, split_stride_bytes / 4,
                   active, corr, extra);
    return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
  });
}

int launch_finish_mlr_fused(cudaStream_t s, RowMap u, const float2* stats, int n_parts, int part_cols,
                            const int32_t* labels, int K, int J, int* dev_status, float* dual, float sdca_step,
                            const FinishExtra& extra_in) {
  FinishExtra extra = extra_in;
  extra.header_blocks = header_blocks(extra);
  const size_t smem = (size_t)n_parts * sizeof(float);
  if (smem > 48 * 1024) return SFB_ERR_SHAPE;
  if (u.es == 4)
    launch_chained(finish_mlr_fused_kernel<4>, K + extra.header_blocks, 256, smem, s, u, stats, n_parts, part_cols, labels, K, J, dev_status, dual, sdca_step, extra);
  else
    launch_chained(finish_mlr_fused_kernel<2>, K + extra.header_blocks, 256, smem, s, u, stats, n_parts, part_cols, labels, K, J, dev_status, dual, sdca_step, extra);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

int launch_prox_unit_columns(cudaStream_t s, float* W, int J, int D, __nv_bfloat16* shadow) {
  // CTAs per slab: as many as hold the slab in registers, or as are needed to give every SM two, up to eight
  const int slabs = (D + 31) / 32;
  int ctas = 1;
  while (ctas < 8 && (ctas * PROX_HELD * PROX_ROWS < J || (slabs * ctas < 296 && ctas * 2 * PROX_ROWS < J))) ctas *= 2;
  const int rows = (J + ctas - 1) / ctas;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ctas; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(ctas * slabs);
  cfg.blockDim = dim3(PROX_THREADS);
  cfg.stream = s;
  cfg.attrs = at; cfg.numAttrs = 2;
  const cudaError_t e = (D & 3) == 0 ? cudaLaunchKernelEx(&cfg, prox_unit_columns_kernel<true>, W, J, D, rows, shadow)
                                     : cudaLaunchKernelEx(&cfg, prox_unit_columns_kernel<false>, W, J, D, rows, shadow);
  return e == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

int launch_pack_rows(cudaStream_t s, RowMap u_src, RowMap u_dst, int J, RowMap v_src, RowMap v_dst, int D, int K,
                     const Commit& commit) {
  const long long total = (long long)K * ((u_dst.ld + v_dst.ld) * (long long)u_dst.es / 16);
  const int blocks = (int)((total + 255) / 256 < 148LL * 16 ? (total + 255) / 256 : 148LL * 16);
  launch_chained(pack_rows_kernel, blocks, 256, 0, s, u_src, u_dst, J, v_src, v_dst, D, K, commit);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

int launch_copy_rows(cudaStream_t s, RowMap src, RowMap dst, int K, int cols, CorrOut corr) {
  const long long total = (long long)K * (dst.ld * dst.es / 16);
  if (total == 0) return 0;
  const int blocks = (int)((total + 255) / 256 < 148LL * 16 ? (total + 255) / 256 : 148LL * 16);
  launch_chained(copy_rows_kernel, blocks, 256, 0, s, src, dst, K, cols, corr);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

int launch_diff_rows(cudaStream_t s, const float* Xa, const float* Xb, RowMap v, int K, int D, CorrOut corr) {
  const long long total = (long long)K * (v.ld >> 2);
  const int blocks = (int)((total + 255) / 256 < 148LL * 16 ? (total + 255) / 256 : 148LL * 16);
  launch_chained(diff_rows_kernel, blocks, 256, 0, s, Xa, Xb, v, K, D, corr);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

int launch_cast_bf16(cudaStream_t s, const float* W, __nv_bfloat16* Wb, long long n) {
  const long long n4 = n / 4;   // J*D is a multiple of 4 on the bf16 path (D % 8 == 0 is required there)
  const int blocks = (int)((n4 + 255) / 256 < 148LL * 16 ? (n4 + 255) / 256 : 148LL * 16);
  launch_chained(cast_bf16_kernel, blocks, 256, 0, s, W, Wb, n4);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

}  // namespace sfb
