// A whole step of a small dense fp32 problem in one launch of one thread block: factors, commit to the SF buffer, apply.
//
// Everything fits in one SM's shared memory, so the step costs one launch and one pass over global memory instead of
// three dependent launches.  Every sum is formed in the order the separate kernels use (products over ascending d,
// softmax and norm sums by the same tree, the update over ascending i), so the results are theirs bit for bit.
//
// Bound: latency of the launch and of the loads.  J = 10, D = 64, K = 32: 16.4 us a step as three launches, 8.1 as one.
#include "common.cuh"

namespace sfb {
namespace {

constexpr int T = 512;

struct SmallStep {
  float* W;
  const float* X;
  const float* Xb;          // DML
  const int32_t* labels;    // MLR
  const uint8_t* similar;   // DML
  float* dual;              // MLR, optional
  float sdca_step, margin, eta;
  RowMap u, v;
  int K, Ka, J, D;          // samples; samples whose pairs are applied
  int dp, jp;               // shared-memory row lengths of X / W rows and u rows: odd numbers of 16-byte units
  int* dev_status;
  Commit commit;
};

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

__global__ void __launch_bounds__(T) step_small_kernel(const __grid_constant__ SmallStep p) {
  chain();
  extern __shared__ __align__(16) float smem[];
  float* Xs = smem;                       // [K][dp]
  float* Ws = Xs + p.K * p.dp;            // [J][dp]
  float* Us = Ws + p.J * p.dp;            // [K][jp]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int K = p.K, J = p.J, D = p.D;
  const bool apply = (*p.dev_status & SFB_DEV_BAD_HEADER) == 0;   // as the apply kernels: a bad header stays until read

  // operands into shared memory, zeros behind D; the factor v on the way
  const int d4 = (D + 3) >> 2;
  const bool vec = (D & 3) == 0;
  auto row4 = [&](const float* row, int c) {
    if (vec) return *reinterpret_cast<const float4*>(row + c);
    float4 r = make_float4(row[c], 0.f, 0.f, 0.f);
    if (c + 1 < D) r.y = row[c + 1];
    if (c + 2 < D) r.z = row[c + 2];
    if (c + 3 < D) r.w = row[c + 3];
    return r;
  };
  for (int t = tid; t < K * d4; t += T) {
    const int i = t / d4, c = (t - i * d4) * 4;
    float4 a = row4(p.X + (size_t)i * D, c);
    if (p.Xb != nullptr) {
      const float4 b = row4(p.Xb + (size_t)i * D, c);
      a = make_float4(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z), __fsub_rn(a.w, b.w));
    }
    *reinterpret_cast<float4*>(Xs + i * p.dp + c) = a;
    *reinterpret_cast<float4*>(p.v.row(i) + (size_t)c * 4) = a;    // ldv = D rounded up to 4
  }
  for (int t = tid; t < J * d4; t += T) {
    const int j = t / d4, c = (t - j * d4) * 4;
    *reinterpret_cast<float4*>(Ws + j * p.dp + c) = row4(p.W + (size_t)j * D, c);
  }
  write_header(p.commit, tid, T);
  __syncthreads();

  // z_i = W a_i: one thread per (sample, row of W)
  for (int t = tid; t < K * J; t += T) {
    const int i = t / J, j = t - i * J;
    const float* x = Xs + i * p.dp;
    const float* w = Ws + j * p.dp;
    float z = 0.f;
#pragma unroll 4
    for (int c = 0; c < d4; ++c) {
      const float4 a = *reinterpret_cast<const float4*>(x + 4 * c), b = *reinterpret_cast<const float4*>(w + 4 * c);
      z = fmaf(a.x, b.x, z); z = fmaf(a.y, b.y, z); z = fmaf(a.z, b.z, z); z = fmaf(a.w, b.w, z);
    }
    Us[i * p.jp + j] = z;
  }
  __syncthreads();

  // u_i: one warp per sample, four rows of W per lane (J <= 128)
  const int j = lane * 4;
  for (int i = warp; i < K; i += T / 32) {
    float t[4], g[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) t[e] = j + e < J ? Us[i * p.jp + j + e] : 0.f;
    if (p.labels != nullptr) {
      const float kLog2e = 1.4426950408889634f;
      float m = -INFINITY;
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j + e < J) m = fmaxf(m, t[e]);
      m = warp_max(m);
      const float mb = m * kLog2e;
#pragma unroll
      for (int e = 0; e < 4; ++e) t[e] = j + e < J ? exp2f(fmaf(t[e], kLog2e, -mb)) : 0.f;
      const float inv = 1.0f / warp_sum((t[0] + t[1]) + (t[2] + t[3]));
      const int y = p.labels[i];
      const bool bad = y < 0 || y >= J;
      if (bad && lane == 0) atomicOr(p.dev_status, SFB_DEV_BAD_LABEL);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float r = t[e] * inv;
        if (y == j + e) r -= 1.f;
        g[e] = (bad || j + e >= J) ? 0.f : r;
      }
      if (p.dual != nullptr && j < J) {   // SDCA: the factor is the dual step, the dual variables move by it
        const float4 du = sdca_step4(p.dual + (size_t)i * ((J + 3) & ~3), j, J, make_float4(g[0], g[1], g[2], g[3]),
                                     p.sdca_step, bad);
        g[0] = du.x; g[1] = du.y; g[2] = du.z; g[3] = du.w;
      }
    } else {
      const float n = warp_sum((t[0] * t[0] + t[1] * t[1]) + (t[2] * t[2] + t[3] * t[3]));
      const float s = p.similar[i] != 0 ? 1.f : ((n < p.margin) ? -1.f : 0.f);   // strict hinge
#pragma unroll
      for (int e = 0; e < 4; ++e) g[e] = s != 0.f && j + e < J ? t[e] * s : 0.f;
    }
    __syncwarp();
    if (j < p.u.ld) {   // ldu = J rounded up to 4
      *reinterpret_cast<float4*>(p.u.row(i) + (size_t)j * 4) = make_float4(g[0], g[1], g[2], g[3]);
      *reinterpret_cast<float4*>(Us + i * p.jp + j) = make_float4(g[0], g[1], g[2], g[3]);
    }
  }
  __syncthreads();
  if (!apply) return;

  // W[j .. j + 3][d]: one thread per column and four rows
  const int j4 = (J + 3) >> 2;
  for (int t = tid; t < j4 * D; t += T) {
    const int jj = (t / D) * 4, d = t - (t / D) * D;
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll 8
    for (int i = 0; i < p.Ka; ++i) {
      const float4 u = *reinterpret_cast<const float4*>(Us + i * p.jp + jj);
      const float x = Xs[i * p.dp + d];
      a0 = fmaf(u.x, x, a0); a1 = fmaf(u.y, x, a1); a2 = fmaf(u.z, x, a2); a3 = fmaf(u.w, x, a3);
    }
    const float a[4] = {a0, a1, a2, a3};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (jj + e < J) p.W[(size_t)(jj + e) * D + d] = fmaf(-p.eta, a[e], Ws[(jj + e) * p.dp + d]);
  }
}

int odd_units(int n) {   // n floats rounded up to an odd number of 16-byte units
  const int u = (n + 3) / 4;
  return (u | 1) * 4;
}
size_t smem_bytes(int K, int J, int D) {
  return ((size_t)(K + J) * odd_units(D) + (size_t)K * odd_units(J)) * 4;
}
constexpr size_t SMEM_MAX = 96 * 1024;

}  // namespace

// One SM does all of it, so the time grows with K J D (4 us from 2^14 to 2^16) while three launches that spread over the
// chip start at 14 us: at 2^16 10.5-11.8 us (J 100 / 16, D 64) against about 17, at 2^18 the two would meet.
bool step_small_fits(int K, int J, int D) {
  return J <= 128 && (long long)K * J * D <= (1 << 16) && smem_bytes(K, J, D) <= SMEM_MAX;
}

int launch_step_small(cudaStream_t s, const sfb_desc& d, float* W, const float* X, const sfb_aux* aux, RowMap u, RowMap v,
                      int K, int K_apply, float eta, int* dev_status, const Commit& commit) {
  static PerDeviceOnce attr_once;
  if (!set_up_device(attr_once, [] { return allow_smem(step_small_kernel, SMEM_MAX); })) return SFB_ERR_CUDA;
  SmallStep p = {};
  p.W = W; p.X = X;
  if (d.model == SFB_DML) {
    p.Xb = reinterpret_cast<const float*>(aux->Xb);
    p.similar = aux->similar;
  } else {
    p.labels = aux->labels;
    p.dual = reinterpret_cast<float*>(aux->dual);
    p.sdca_step = aux->sdca_step;
  }
  p.margin = d.margin; p.eta = eta;
  p.u = u; p.v = v;
  p.K = K; p.Ka = K_apply; p.J = d.J; p.D = d.D;
  p.dp = odd_units(d.D); p.jp = odd_units(d.J);
  p.dev_status = dev_status;
  p.commit = commit;
  launch_chained(step_small_kernel, 1, T, smem_bytes(K, d.J, d.D), s, p);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

}  // namespace sfb
