// Shared declarations of the SF hot-path kernels (internal; the public boundary is include/sfb.h).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "per_device.cuh"
#include "sfb.h"

namespace sfb {

// Where the K factor rows of one operand live: row i of worker p = i / B sits at
// base + p * worker_stride + (i % B) * ld * elem_size.  Covers both caller-side [K][ld] arrays
// (worker_stride = B * ld * elem_size) and the U / V blocks of the SF buffer's worker streams.
struct RowMap {
  char* base;
  long long worker_stride;  // bytes
  int ld;                   // values per row (padded)
  int B;                    // rows per worker
  int es;                   // bytes per value (4 = fp32, 2 = bf16)
  __host__ __device__ __forceinline__ char* row(int i) const {
    return base + (long long)(i / B) * worker_stride + (long long)(i % B) * ld * es;
  }
};

// Byte layout of the SF buffer for one descriptor (see the wire format in include/sfb.h).
struct Layout {
  int es, ldu, ldv, cap_p;
  long long u_bytes, v_bytes, rp_bytes, idx_bytes, val_bytes;
  long long stream_stride, streams_off, total_bytes;
};

static inline long long pad_to(long long n, long long a) { return (n + a - 1) / a * a; }

// Optional extra outputs of a kernel that writes fp32 factor rows on the compensated tf32 path: the rows'
// bf16 correction operands (split.cu), so that no separate pass has to read the rows again.
//   mn: for the apply (MN-major), [block of 32 pairs][64 lines][ldc]; pair (worker w, row r) sits in block
//       w * k_bpw + r / 32, line r % 32 (k_wp == 1: whole blocks per worker), or in block w / k_wp, line
//       (w % k_wp) * k_bb + r (k_bb rows of each of k_wp workers per block); a_side: remainder lines first.
//   km: for the forward (K-major A side), [pair][atom][32 remainders | 32 values].
struct CorrOut {
  char* mn;
  char* km;
  int ldc, k_bb, k_wp, k_bpw, a_side, atoms;
  __host__ __device__ CorrOut() : mn(nullptr), km(nullptr), ldc(0), k_bb(32), k_wp(1), k_bpw(1), a_side(0), atoms(0) {}
};
#ifdef __CUDACC__
// Four fp32 values as bf16, and the bf16 remainders of what the tensor core sees of them (see split.cu).
__device__ __forceinline__ void split4(const float4& t, uint2& val, uint2& rem) {
  const float rx = t.x - __uint_as_float(__float_as_uint(t.x) & 0xFFFFE000u);
  const float ry = t.y - __uint_as_float(__float_as_uint(t.y) & 0xFFFFE000u);
  const float rz = t.z - __uint_as_float(__float_as_uint(t.z) & 0xFFFFE000u);
  const float rw = t.w - __uint_as_float(__float_as_uint(t.w) & 0xFFFFE000u);
  const __nv_bfloat162 v0 = __floats2bfloat162_rn(t.x, t.y), v1 = __floats2bfloat162_rn(t.z, t.w);
  const __nv_bfloat162 r0 = __floats2bfloat162_rn(rx, ry), r1 = __floats2bfloat162_rn(rz, rw);
  val = make_uint2(*reinterpret_cast<const uint32_t*>(&v0), *reinterpret_cast<const uint32_t*>(&v1));
  rem = make_uint2(*reinterpret_cast<const uint32_t*>(&r0), *reinterpret_cast<const uint32_t*>(&r1));
}
// values t of pair i (B pairs per worker) at columns j .. j + 3, j a multiple of 4
__device__ __forceinline__ void corr_store4(const CorrOut& c, int i, int B, int j, float4 t) {
  uint2 val, rem;
  split4(t, val, rem);
  if (c.mn != nullptr && j < c.ldc) {
    const int w = i / B, r = i - w * B;
    long long blk;
    int line;
    if (c.k_wp == 1) { blk = (long long)w * c.k_bpw + (r >> 5); line = r & 31; }
    else { blk = w / c.k_wp; line = (w % c.k_wp) * c.k_bb + r; }
    char* base = c.mn + ((blk * 64) * c.ldc + j) * 2;
    *reinterpret_cast<uint2*>(base + (long long)(c.a_side ? line : 32 + line) * c.ldc * 2) = rem;
    *reinterpret_cast<uint2*>(base + (long long)(c.a_side ? 32 + line : line) * c.ldc * 2) = val;
  }
  if (c.km != nullptr && (j >> 5) < c.atoms) {
    char* atom = c.km + (((long long)i * c.atoms + (j >> 5)) * 64 + (j & 31)) * 2;
    *reinterpret_cast<uint2*>(atom) = rem;
    *reinterpret_cast<uint2*>(atom + 64) = val;
  }
}
#endif

static inline Layout make_layout(const sfb_desc& d) {
  Layout l;
  l.es = (d.path == SFB_PATH_BF16) ? 2 : 4;
  const int unit = 16 / l.es;
  l.ldu = (int)pad_to(d.J, unit);
  l.ldv = (int)pad_to(d.D, unit);
  l.cap_p = d.v_sparse ? (int)(d.nnz_capacity / (uint64_t)d.P) : 0;
  l.u_bytes = pad_to((long long)d.B * l.ldu * l.es, 128);
  if (d.v_sparse) {
    l.rp_bytes = pad_to((long long)(d.B + 1) * 4, 128);
    l.idx_bytes = pad_to((long long)l.cap_p * 4, 128);
    l.val_bytes = pad_to((long long)l.cap_p * l.es, 128);
    l.v_bytes = l.rp_bytes + l.idx_bytes + l.val_bytes;
  } else {
    l.rp_bytes = l.idx_bytes = l.val_bytes = 0;
    l.v_bytes = pad_to((long long)d.B * l.ldv * l.es, 128);
  }
  l.stream_stride = l.u_bytes + l.v_bytes;
  l.streams_off = 128 + pad_to((long long)d.P * 32, 128);
  l.total_bytes = l.streams_off + (long long)d.P * l.stream_stride;
  return l;
}

struct HeaderImage {   // exactly the first 68 bytes of the 128-byte header
  uint32_t magic;
  uint16_t version;
  uint8_t model, dtype;
  uint32_t flags, P, B, J, D, clock, ldu, ldv;
  uint64_t stream_stride, total_bytes, streams_off;
  uint32_t cap_p;
};
static_assert(sizeof(HeaderImage) == 72, "header image is 68 bytes of fields plus 4 of tail padding");

// The check of a buffer's header before it is applied, for whichever kernel of a call does it (buf == nullptr: none).
struct HeaderCheck {
  const char* buf;
  HeaderImage h;
  int* dev_status;
  int* clear;   // optional: a word to clear on the way
  __host__ __device__ HeaderCheck() : buf(nullptr), h(), dev_status(nullptr), clear(nullptr) {}
};
#ifdef __CUDACC__
// Has the check that precedes this kernel refused the buffer it was given (refused: the status word, or nullptr = not
// checked)?  Then nothing in that buffer may be followed: row pointers and offsets could lead anywhere.
__device__ __forceinline__ bool is_refused(const int* refused) {
  return refused != nullptr && (*refused & SFB_DEV_BAD_HEADER) != 0;
}
// Does the buffer's header match the descriptor's?  Every thread for itself: five loads at once, the same for all, against
// the expected words in registers, which a kernel whose other work waits for the answer has fetched before.  (A word per lane
// looks the expected ones up one after the other: 0.5 us of the pass that asks.)
struct HeaderWords { uint32_t w[17]; };
__device__ __forceinline__ HeaderWords expected_header(const HeaderCheck& c) {
  const uint32_t* r = reinterpret_cast<const uint32_t*>(&c.h);
  HeaderWords e;
#pragma unroll
  for (int t = 0; t < 17; ++t) {
    e.w[t] = r[t];
    asm volatile("" : "+r"(e.w[t]));   // (now, not where it is used)
  }
  return e;
}
__device__ __forceinline__ bool header_matches(const HeaderCheck& c, const HeaderWords& e) {
  const uint4* q = reinterpret_cast<const uint4*>(c.buf);
  const uint32_t* r = e.w;
  const uint4 w0 = q[0], w1 = q[1], w2 = q[2], w3 = q[3];
  const uint32_t w16 = reinterpret_cast<const uint32_t*>(c.buf)[16];
  uint32_t d = (w0.x ^ r[0]) | (w0.y ^ r[1]) | ((w0.z & ~2u) ^ r[2]) | (w0.w ^ r[3]);   // flag bit 1 (compacted): either
  d |= (w1.x ^ r[4]) | (w1.y ^ r[5]) | (w1.z ^ r[6]);                                   // word 7 is the clock: any value
  d |= (w2.x ^ r[8]) | (w2.y ^ r[9]) | (w2.z ^ r[10]) | (w2.w ^ r[11]);
  d |= (w3.x ^ r[12]) | (w3.y ^ r[13]) | (w3.z ^ r[14]) | (w3.w ^ r[15]) | (w16 ^ r[16]);
  return d == 0u;
}
// The outcome written down, by one thread.
__device__ __forceinline__ void report_header(const HeaderCheck& c, bool matches) {
  if (c.clear != nullptr) *c.clear = 0;
  if (!matches) atomicOr(c.dev_status, SFB_DEV_BAD_HEADER);
}
#endif

// Header and directory of a buffer, for whichever kernel of a call writes them (buf == nullptr: none).
struct Commit {
  char* buf;
  HeaderImage h;
  long long u_bytes;
  const uint32_t* rowptr;   // global CSR row pointers (sparse v), or nullptr
  __host__ __device__ Commit() : buf(nullptr), h(), u_bytes(0), rowptr(nullptr) {}
};
Commit make_commit(void* sf_buf, const sfb_desc& d, const Layout& l, uint32_t clock, const uint32_t* rowptr);
#ifdef __CUDACC__
// Called by n threads, of one block or of several.
__device__ __forceinline__ void write_header(const Commit& c, int tid, int n) {
  uint32_t* w = reinterpret_cast<uint32_t*>(c.buf);
  const HeaderImage& h = c.h;
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&h);
  for (int t = tid; t < 32; t += n) w[t] = (t < 17) ? src[t] : 0u;
  const int dir_words = (int)((h.streams_off - 128) / 4);
  for (int t = tid; t < dir_words; t += n) {
    const int p = t >> 3, f = t & 7;
    uint32_t val = 0u;
    if (p < (int)h.P) {
      const uint64_t u_off = h.streams_off + (uint64_t)p * h.stream_stride;
      const uint64_t v_off = u_off + (uint64_t)c.u_bytes;
      switch (f) {
        case 0: val = (uint32_t)p; break;
        case 1: val = h.B; break;
        case 2: val = h.clock; break;
        case 3:
          if (c.rowptr != nullptr) {
            const uint32_t m = c.rowptr[(p + 1) * h.B] - c.rowptr[p * h.B];
            val = m < h.cap_p ? m : h.cap_p;
          } else if (h.flags & 1u) {   // no global row pointers: the count the worker's own stream carries
            val = reinterpret_cast<const uint32_t*>(c.buf + v_off)[h.B];
          }
          break;
        case 4: val = (uint32_t)(u_off & 0xffffffffu); break;
        case 5: val = (uint32_t)(u_off >> 32); break;
        case 6: val = (uint32_t)(v_off & 0xffffffffu); break;
        default: val = (uint32_t)(v_off >> 32); break;
      }
    }
    w[32 + t] = val;
  }
}
#endif

// What a finishing pass does beside its own work: the buffer's header, which u rows hold a nonzero wire value (for the
// compaction), and (MLR, small batches) the factor v = x.
struct FinishExtra {
  Commit commit;
  uint8_t* nonzero;  // [rows] or nullptr
  RowMap src, dst;   // dst.base == nullptr: no copy
  int cols;
  bool next_early;   // see chain_next
  int header_blocks; // blocks in front of the rows' that write the header (set by the launcher)
  int* take_bad;     // a word to clear, and (give_bad) another that gets its value first
  int* give_bad;
  FinishExtra() : nonzero(nullptr), src(), dst(), cols(0), next_early(false), header_blocks(0), take_bad(nullptr), give_bad(nullptr) {}
};

#ifdef __CUDACC__
// SDCA (dual != nullptr; Section 2.1, "Stochastic DCA"): the factor is the damped dual step
// du_i = step * (dual_i + g_i) with g_i = softmax(z_i) - onehot(y_i), and dual_i <- dual_i - du_i in place
// (dual rows: fp32, ldd = J rounded up to 4 values per row, pad values written as zeros).
__device__ __forceinline__ float4 sdca_step4(float* dual_row, int j, int J, float4 g, float step, bool bad) {
  float4 d = *reinterpret_cast<const float4*>(dual_row + j);
  float4 du = make_float4(0.f, 0.f, 0.f, 0.f);
  if (!bad) {   // a sample with a bad label takes no step: its dual variables stay as they are
    du.x = step * (d.x + g.x); du.y = step * (d.y + g.y); du.z = step * (d.z + g.z); du.w = step * (d.w + g.w);
    d.x -= du.x; d.y -= du.y; d.z -= du.z; d.w -= du.w;
  }
  if (j + 1 >= J) { du.y = 0.f; d.y = 0.f; }
  if (j + 2 >= J) { du.z = 0.f; d.z = 0.f; }
  if (j + 3 >= J) { du.w = 0.f; d.w = 0.f; }
  *reinterpret_cast<float4*>(dual_row + j) = d;
  return du;
}
#endif

// Chained launches (programmatic dependent launch): a kernel of a call's chain may be scheduled while its predecessor on
// the stream is still running, so that launch latency and set-up overlap with it.  Every such kernel starts with chain(),
// or, where the set-up touches no memory that another kernel writes, chain_next() first and chain_wait() behind it:
// (A kernel that is followed by one of the fp32 GEMMs does not call chain_next, so that its successor is scheduled when
// it ends: their blocks, two to four to an SM, would otherwise crowd onto the SMs that run free first.  40 x 15000,
// K = 800: 318 us a step, 399 with it.)
// Nothing before the wait reads or writes global memory, and every thread waits, so each grid is complete, its writes
// visible, before its successor touches memory, exactly as without the overlap.  That holds for ordinary loads only: the
// read-only path asks for data that does not change while the kernel runs, which here begins before the wait, and the
// compiler may move a load from a __restrict__ pointer above it.  So these kernels declare no pointer __restrict__ and
// use no __ldg, for the caller's arrays neither (their producer may itself have let its successor start early).
#ifdef __CUDACC__
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain() {
  chain_next();
  chain_wait();
}
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#endif

// cudaFuncSetAttribute acts on the current device only.  False: the set-up failed, nothing may be launched that needs it.
template <typename F>
bool set_up_device(PerDeviceOnce& once, F&& setup) {
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && once.ok(dev, setup)) return true;
  cudaGetLastError();
  return false;
}
template <typename K>
bool allow_smem(K* kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

// ---- kernel launchers (each returns the number of kernels it launched, or a negative SFB_ERR_*) ----

// v rows = Xa rows - Xb rows, one fp32 subtraction per element, pad columns zero (the DML factor v).
int launch_diff_rows(cudaStream_t s, const float* Xa, const float* Xb, RowMap v, int K, int D, CorrOut corr = CorrOut());
// Z[i][j] = sum_d A[i][d] * W[j][d] on fp32 CUDA cores, written as fp32 rows through `z`.
// The reduction is cut into ks ranges (*nsplit_out of them exist) whose partial products go to `part` (fp32 rows,
// split_stride bytes between partial buffers) instead of `z` if there is more than one; the finishing pass sums them in
// range order.  The sums do not depend on which of the three kernels forms them.
//   launch_forward_f32, one launch: A = X, or X - Xb (element-wise fp32 subtraction) when Xb != nullptr.  When `v` has a
//   base, the operand rows (X, or the difference) are also written there (the factor v), pad columns zero.
int launch_forward_f32(cudaStream_t s, const float* W, const float* X, const float* Xb, int K, int J, int D,
                       RowMap z, RowMap v, RowMap part = RowMap(), long long split_stride = 0, int ks = 1,
                       int* nsplit_out = nullptr);
//   The others take operand rows a_i behind a row map; copy (optional): those rows also written there.
//   _small: 64 x 64 tiles, operands in place.  _nn: large tiles through transposed copies of both operands; ws:
//   forward_f32_nn_workspace_floats(K, J, D) floats.
// forward_f32_plan: which of the three, and how many ranges to ask for, at most max_ks.  pair: A = X - Xb.
enum F32Route { F32_IN_PLACE, F32_SMALL, F32_TRANSPOSED };
struct ForwardF32Plan {
  F32Route route;
  int ks;
  double us;   // estimated time
};
constexpr int FORWARD_F32_MAX_SPLITS = 32;
ForwardF32Plan forward_f32_plan(int K, int J, int D, bool pair, int max_ks, bool transposed_ok);
// The products only, in exactly ks ranges (range s to z + s * split_stride; ranges beyond D: zeros), if *only_if != 0.
int launch_forward_f32_if(cudaStream_t s, const float* W, const float* X, const float* Xb, int K, int J, int D, RowMap z,
                          long long split_stride, int ks, const int* only_if);
int launch_forward_f32_small(cudaStream_t s, const float* W, RowMap src, RowMap copy, int K, int J, int D, RowMap z,
                             RowMap part, long long split_stride, int ks, int* nsplit_out);
long long forward_f32_nn_workspace_floats(int K, int J, int D);
int launch_forward_f32_nn(cudaStream_t s, const float* W, RowMap src, RowMap copy, int K, int J, int D, float* ws,
                          RowMap z, RowMap part, long long split_stride, int ks, int* nsplit_out);

// W[j][d] -= eta * sum_{i<K} U[i][j] * V[i][d] on fp32 CUDA cores (fixed summation order).
int launch_apply_f32(cudaStream_t s, float* W, RowMap u, RowMap v, int K, int J, int D, float eta,
                     const int* dev_status, const int* row_idx = nullptr, const int* n_rows = nullptr,
                     const int* only_if = nullptr, int full_if = 0);
// only_if (optional, device): nothing is done where it is 0; all K rows instead of the listed ones where it has a bit of full_if.
// row_idx / n_rows (optional, device): apply only the factor rows row_idx[0 .. *n_rows), in that order, instead of
// rows 0 .. K-1 (rows that are known to be all zeros can be left out: the result is bit-identical).

// A whole step (dense fp32, MLR or DML) of a problem that fits in one block: factors of K samples into u and v, header,
// and the update by the first K_apply pairs.  Same bits as the separate kernels.
bool step_small_fits(int K, int J, int D);
int launch_step_small(cudaStream_t s, const sfb_desc& d, float* W, const float* X, const sfb_aux* aux, RowMap u, RowMap v,
                      int K, int K_apply, float eta, int* dev_status, const Commit& commit);

// MLR epilogue: u = softmax(z) - onehot(label).  z rows are fp32; u rows fp32 or bf16 (u.es).
// z may be `nsplit` partial products (split s at z + s * split_stride_bytes), summed in split order.
// dual (optional, SDCA): fp32 dual variables of the K samples, [K][J rounded up to 4], updated in place; the factor
// written to u is then the dual step sdca_step * (dual + softmax - onehot).
int launch_finish_mlr(cudaStream_t s, RowMap z, RowMap u, const int32_t* labels, int K, int J, int* dev_status,
                      int nsplit = 1, long long split_stride_bytes = 0, float* dual = nullptr, float sdca_step = 0.f,
                      CorrOut corr = CorrOut(), const FinishExtra& extra = FinishExtra());

// DML epilogue: u = +z (similar) or -z * [|z|^2 < margin] (dissimilar).
// active (optional, [K] bytes): 1 where the pair contributes (similar, or dissimilar inside the margin), 0 where u_i = 0.
int launch_finish_dml(cudaStream_t s, RowMap z, RowMap u, const uint8_t* similar, float margin, int K, int J,
                      int nsplit = 1, long long split_stride_bytes = 0, uint8_t* active = nullptr, CorrOut corr = CorrOut(),
                      const FinishExtra& extra = FinishExtra());
// idx[0 .. *n_out) = ascending list of the samples i < K with active[i] != 0 (device arrays; one ordered block).
int launch_compact_active(cudaStream_t s, const uint8_t* active, int K, int* idx, int* n_out);

// Copies K rows of `cols` values from src to dst rows (same value type), zero-filling dst pad columns.
int launch_copy_rows(cudaStream_t s, RowMap src, RowMap dst, int K, int cols, CorrOut corr = CorrOut());

// The u rows (J values) and v rows (D values) of K pairs into the streams behind u_dst / v_dst, and the header.
int launch_pack_rows(cudaStream_t s, RowMap u_src, RowMap u_dst, int J, RowMap v_src, RowMap v_dst, int D, int K,
                     const Commit& commit);

// Writes header and directory of the SF buffer.  `rowptr` (global CSR row pointers) only for sparse v.
int launch_write_header(cudaStream_t s, void* sf_buf, const sfb_desc& d, const Layout& l, uint32_t clock,
                        const uint32_t* rowptr);

// Copies the CSR codes of every worker into its stream (local row pointers, zero-filled tail).  commit (optional): header
// and directory written by the same launch.
int launch_pack_csr(cudaStream_t s, void* sf_buf, const sfb_desc& d, const Layout& l, const uint32_t* rowptr,
                    const uint32_t* idx, const float* val, int* dev_status, const Commit& commit = Commit());

// Inactive-pair compaction of a committed dense-v buffer, in place: per worker the pairs with a nonzero u move to
// the front (same order), the slots behind them are cleared, the directory gets the pair counts and the header
// its "compacted" flag.  workspace: compact_workspace_bytes(K, P) bytes.  launch_kept_rows lists the slots
// p * B + r, r < count of worker p, of the first `workers` workers (idx [K], n_out one int; device arrays).
long long compact_workspace_bytes(int K, int P);
int launch_compact(cudaStream_t s, void* sf_buf, const sfb_desc& d, const Layout& l, void* workspace, int first_worker = 0,
                   int n_workers = 0,
                   bool flags_ready = false);   // n_workers > 0: only those workers' streams (a process's shard)
// flags_ready: the finishing pass that wrote the u rows left its flags (FinishExtra::nonzero) in compact_flags(workspace).
uint8_t* compact_flags(void* workspace);
// flags[i] = 1 where row i of u (J values) holds a nonzero one.  refused: see is_refused (the flags stay as they are then).
int launch_row_nonzero(cudaStream_t s, RowMap u, int K, int J, uint8_t* flags, const int* refused = nullptr);
// Rebuilds the directory's pair counts (and the header flag) from streams that arrived already compacted.
int launch_count_pairs(cudaStream_t s, void* sf_buf, const sfb_desc& d, const Layout& l, void* workspace);
int launch_kept_rows(cudaStream_t s, const void* sf_buf, int B, int workers, int* idx, int* n_out, const int* refused = nullptr);

// Sets SFB_DEV_BAD_HEADER in *dev_status unless the buffer's header matches the descriptor.
HeaderCheck make_check(const void* sf_buf, const sfb_desc& d, const Layout& l, int* dev_status);
int launch_check_header(cudaStream_t s, const HeaderCheck& check);

// SC forward: u_i = sum_{(d,a) in code i} a * W[:, d] - x_i, codes read from CSR arrays whose row
// pointers are either global ([K+1]) or per worker stream inside the SF buffer.
struct CsrView {
  const char* base;          // SF buffer base, or nullptr for caller-side global arrays
  const uint32_t* rowptr;    // global arrays (base == nullptr)
  const uint32_t* idx;
  const float* val;
  long long streams_off, stream_stride, v_off, rp_bytes, idx_bytes;  // stream-relative offsets (base != nullptr)
  int B;
  int cap_p;                 // global arrays only: > 0 cuts every worker's rows off after its first cap_p nonzeros
                             // (what pack_csr keeps in the stream); 0 = rows as given
};
// Wt is a caller-provided workspace of sc_forward_workspace_bytes(J, D) bytes (atom-major copy of W).
long long sc_forward_workspace_bytes(int J, int D);
int launch_sc_forward_ws(cudaStream_t s, const float* W, float* Wt, CsrView codes, const float* Xdata, RowMap u, int K,
                         int J, int D, int* dev_status);

// SC apply: W[:, d] -= eta * sum_{i: a_id != 0} a_id * u_i (sparse-v scatter, no float atomics).
// flags: K bytes of scratch.  dev_status: SFB_DEV_BAD_INDEX for rows with entries that are left out; refused: see is_refused.
int launch_sc_apply(cudaStream_t s, float* W, CsrView codes, RowMap u, int K, int J, int D, float eta, uint8_t* flags,
                    int* dev_status, const int* refused = nullptr);

// The same update through an atom-major (CSC) re-sort of the codes and shared-memory u columns (faster;
// needs sc_csc_supported(K) and a workspace of sc_csc_workspace_bytes(K, D, nnz_capacity) bytes).
long long sc_csc_workspace_bytes(int K, int D, long long nnz_capacity);
bool sc_csc_supported(int K);
// In two halves: the re-sort reads only the codes (it can run beside the forward pass), the update needs u and the
// workspace the re-sort filled.
// dev_status (optional): SFB_DEV_BAD_INDEX is set for entries the re-sort leaves out (the same entries the forward
// pass skips).
// refused: see is_refused (no entry is sorted then).
int launch_sc_csc_build(cudaStream_t s, CsrView codes, int K, int D, long long nnz_capacity, void* workspace,
                        int* dev_status = nullptr, const int* refused = nullptr);
int launch_sc_csc_apply(cudaStream_t s, float* W, RowMap u, int K, int J, int D, float eta, long long nnz_capacity,
                        void* workspace, const int* dev_status_ro);

// Dense fp32 rows a_i of the CSR codes (zeros elsewhere), for the tensor-core sparse-coding path.
// round_tf32: values rounded to the nearest tf32 (the plain tf32 path, whose tensor cores would truncate them).
// refused: see is_refused (the rows stay as they are then).
int launch_densify_codes(cudaStream_t s, CsrView codes, RowMap a, int K, int D, int* dev_status, bool round_tf32 = true,
                         const int* refused = nullptr);
// The same (exact values) with the rows' correction operands written beside them; a row of ld floats must fit in
// shared memory (densify_corr_fits).
bool densify_corr_fits(int ld);
int launch_densify_codes_corr(cudaStream_t s, CsrView codes, RowMap a, int K, int D, int* dev_status, CorrOut corr);

// SC epilogue on dense products: u = z - x in place (u rows hold z), pad columns zero.
// z: products (possibly `nsplit` partials); u = sum of partials - x.
int launch_finish_sc(cudaStream_t s, RowMap z, RowMap u, const float* Xdata, int K, int J, int nsplit = 1,
                     long long split_stride_bytes = 0, CorrOut corr = CorrOut());

// Column-norm projection: every column of W with 2-norm above 1 is divided by its norm (in place).
// shadow (optional, D a multiple of 4): W's correction operand of the compensated path, kept in step with W.
int launch_prox_unit_columns(cudaStream_t s, float* W, int J, int D, __nv_bfloat16* shadow = nullptr);
// Minibatch objective: per-sample values from the fp32 rows (z_i for MLR / DML, u_i for SC) into loss_i[K],
// then their fp64 sum into *total (device).  Two launches.
int launch_sample_loss(cudaStream_t s, int model, RowMap rows, const int32_t* labels, const uint8_t* similar, float margin,
                       int K, int J, float* loss_i, double* total, int* dev_status);

// W (fp32) -> bf16 shadow, round to nearest even.
int launch_cast_bf16(cudaStream_t s, const float* W, __nv_bfloat16* Wb, long long n);
// Correction operands of the error-compensated tf32 kernels (split.cu): bf16 [remainder | value] (A side) or
// [value | remainder] (B side) of fp32 rows.  K-major: dst[row][atom][64] over `rows` rows of `cols` values.
// MN-major: dst[block][64][ldc], block = 32 pairs taken as the apply's reduction blocks are (32 rows of one
// worker, or k_bb rows of each of k_wp workers), ldc a multiple of 64.
int launch_split_k(cudaStream_t s, RowMap src, int rows, int cols, void* dst, bool a_side);
struct SplitSide { RowMap src; int cols; void* dst; int ldc; };   // one factor's rows and where they go (dst == nullptr: not)
// check: done on the way; refused: see is_refused (of a check that came before).  Either way the rows of a buffer that does
// not match are not read.
int launch_split_mn(cudaStream_t s, const SplitSide& us, const SplitSide& vs, int workers, int k_bb, int k_wp, int k_bpw,
                    int blocks, const HeaderCheck& check, const int* refused);

}  // namespace sfb
