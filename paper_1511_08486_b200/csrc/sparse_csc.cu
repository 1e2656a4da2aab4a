// Sparse-v scatter apply through an atom-major (CSC) view of the codes.
//
//   W[:, d] -= eta * sum_{i : a_id != 0} a_id * u_i        (Section 3 update with v_i = a_i sparse)
//
// The codes arrive sample-major (CSR, the factor v_i of each sample).  Per step they are re-sorted by
// (slice of samples, atom) with a counting sort that is deterministic: per (chunk of 32 samples, atom) a mask of the
// samples that use the atom (atomic or), prefix sums of the masks' populations over chunks and atoms, and every entry's
// place follows from the bits below its own, so inside a column the entries are in sample order whatever the thread
// schedule.  Every column of a slice is padded with zero entries to a multiple of four, so that a warp reads the entries
// of consecutive atoms as one stream of groups of four.
// The sort runs beside the forward pass, but below some 1000 x 3000 weights the forward is the shorter of the two: there
// the latency of its steps counts, hence no loop over samples in any of them (counts per chunk of 8 samples, placed one
// sample after the other, and a scan of 1024 sums at a time, made the step 65.0 us
// against 42.3 at 500 x 3000, K = 320, 5 % density, 46.4 against 30.2 at 100 x 400, K = 40, 2 %).
// The apply gives each thread block 32 rows of W at a time and keeps the matching 32 columns of a slice of the
// u_i in shared memory (the samples are taken in as few slices as fit).  A warp takes 8 consecutive
// atoms: it starts the loads of the next part of W, walks the atoms' entries (coalesced loads staged through a
// small per-warp strip), accumulating a_id * u_i[j0 + 4 q .. + 3] from shared memory, parks the sums
// in a private 8 x 36 tile, and finally updates W with 32-byte row segments.
// U is read once and W once per slice; no floating-point atomics; every element of W has one owner and a fixed
// summation order (bit-reproducible); atoms nobody uses get W + (-eta * 0) = W, bit-identical.
#include "common.cuh"

namespace sfb {
namespace {

constexpr int CSC_CHUNK = 32;   // samples per chunk of the counting sort: the bits of a mask

struct CsrRow2 {
  const uint32_t* idx;
  const float* val;
  int len;
};
__device__ __forceinline__ CsrRow2 csr_row2(const CsrView& c, int i) {
  CsrRow2 r;
  if (c.base == nullptr) {
    uint32_t s = c.rowptr[i], e = c.rowptr[i + 1];
    if (c.cap_p > 0) {   // what the worker's stream can hold: the same truncation as pack_csr
      const uint32_t lim = c.rowptr[(size_t)(i / c.B) * c.B] + (uint32_t)c.cap_p;
      s = min(s, lim); e = min(e, lim);
    }
    r.idx = c.idx + s; r.val = c.val + s; r.len = (int)(e - s);
  } else {
    const int p = i / c.B, l = i % c.B;
    const char* vb = c.base + c.streams_off + (long long)p * c.stream_stride + c.v_off;
    const uint32_t* rp = reinterpret_cast<const uint32_t*>(vb);
    const uint32_t s = rp[l], e = rp[l + 1];
    r.idx = reinterpret_cast<const uint32_t*>(vb + c.rp_bytes) + s;
    r.val = reinterpret_cast<const float*>(vb + c.rp_bytes + c.idx_bytes) + s;
    r.len = (int)(e - s);
  }
  return r;
}

// An entry counts only if its atom exists and exceeds its predecessor's: the rule of the forward pass
// (sc_forward_kernel), so that forward and apply agree on malformed rows.  In a row that is strictly ascending no atom
// is repeated; in another one an atom may count more than once (5, 3, 5: the fill adds both values, as the forward does).
__device__ __forceinline__ bool entry_ok(const CsrRow2& row, int k, int D) {
  const uint32_t d = row.idx[k];
  return d < (uint32_t)D && !(k > 0 && row.idx[k - 1] >= d);
}

// bit i % 32 of mask[i / 32][d]: sample i uses atom d (atomic or: the masks do not depend on the order)
__global__ void __launch_bounds__(256) csc_mask_kernel(CsrView codes, int K, int D, uint32_t* __restrict__ mask,
                                                       int* dev_status, const int* refused) {
  if (is_refused(refused)) return;
  const int i = blockIdx.x;
  const CsrRow2 row = csr_row2(codes, i);
  uint32_t* m = mask + (size_t)(i / CSC_CHUNK) * D;
  bool bad = false;
  for (int k = threadIdx.x; k < row.len; k += 256) {
    if (entry_ok(row, k, D)) atomicOr(m + row.idx[k], 1u << (i % CSC_CHUNK));
    else bad = true;   // the entry is skipped
  }
  if (bad && dev_status != nullptr) atomicOr(dev_status, SFB_DEV_BAD_INDEX);
}

// per atom: populations of the chunks' masks -> offsets of each chunk inside the column's slice; slice totals
__global__ void __launch_bounds__(64) csc_chunk_offsets_kernel(int nchunks, int chunks_per_slice, int D,
                                                               const uint32_t* mask, int* off,
                                                               int* total) {
  chain();
  const int d = blockIdx.x * 64 + threadIdx.x;
  if (d >= D) return;
  int run = 0, slice = 0, left = chunks_per_slice;
  for (int c0 = 0; c0 < nchunks; c0 += 16) {   // sixteen independent loads in flight, then the running sum
    uint32_t t[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) t[q] = (c0 + q < nchunks) ? mask[(size_t)(c0 + q) * D + d] : 0u;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      if (c0 + q < nchunks) {
        off[(size_t)(c0 + q) * D + d] = run;
        run += __popc(t[q]);
        if (--left == 0) {
          total[(size_t)slice * D + d] = run;
          run = 0; ++slice; left = chunks_per_slice;
        }
      }
    }
  }
  if (left < chunks_per_slice) total[(size_t)slice * D + d] = run;
}

// colptr[0 .. n] = exclusive scan of total[0 .. n) rounded up to fours (one block, fixed order; eight sums a thread)
__global__ void __launch_bounds__(1024) csc_scan_kernel(int n, const int* total, int* colptr) {
  chain();
  __shared__ int warp_sum[32];
  constexpr int PER = 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int carry = 0;
  for (int base = 0; base < n; base += 1024 * PER) {
    const int d = base + threadIdx.x * PER;
    int v[PER], sum = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) v[q] = d + q < n ? (total[d + q] + 3) & ~3 : 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) sum += v[q];
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int o_ = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += o_;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    int w = warp_sum[lane];                       // every warp scans the 32 sums for itself
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int o_ = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += o_;
    }
    const int before = __shfl_sync(0xffffffffu, w, max(warp - 1, 0));
    int run = carry + (warp > 0 ? before : 0) + incl - sum;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      if (d + q < n) colptr[d + q] = run;
      run += v[q];
    }
    carry += __shfl_sync(0xffffffffu, w, 31);
    __syncthreads();                              // the sums are no longer read
  }
  if (threadIdx.x == 0) colptr[n] = carry;
}

// Blocks 0 .. K - 1: one sample each, every entry to its place (entry = sample index inside its slice, value); the
// blocks behind them write the zero entries that fill the columns up.
__global__ void __launch_bounds__(256) csc_fill_kernel(CsrView codes, int K, int D, int passes, int chunks_per_slice,
                                                       const uint32_t* mask, const int* off,
                                                       const int* total, const int* colptr,
                                                       int2* ent, const int* refused) {
  chain();
  if (is_refused(refused)) return;   // (every column is empty: no mask was written)
  if (blockIdx.x >= (unsigned)K) {
    const int c = (blockIdx.x - K) * 256 + threadIdx.x;
    if (c < passes * D) {
      const int end = colptr[c + 1];
      for (int e = colptr[c] + total[c]; e < end; ++e) ent[e] = make_int2(0, 0);
    }
    return;
  }
  const int i = blockIdx.x, c = i / CSC_CHUNK, slice = c / chunks_per_slice;
  const int i_in = i - slice * chunks_per_slice * CSC_CHUNK;
  const uint32_t below = (1u << (i % CSC_CHUNK)) - 1u;
  const CsrRow2 row = csr_row2(codes, i);
  auto place = [&](int k) {
    const uint32_t d = row.idx[k];
    const size_t cell = (size_t)c * D + d;
    return ent + colptr[(size_t)slice * D + d] + off[cell] + __popc(mask[cell] & below);
  };
  bool bad = false;
  for (int k = threadIdx.x; k < row.len; k += 256) {
    if (entry_ok(row, k, D)) *place(k) = make_int2(i_in, __float_as_int(row.val[k]));
    else bad = true;
  }
  if (__syncthreads_or(bad)) {   // malformed: an atom that counts twice has one place, its values are added in row order
    for (int k = threadIdx.x; k < row.len; k += 256)
      if (entry_ok(row, k, D)) place(k)->y = 0;
    __syncthreads();
    if (threadIdx.x == 0)
      for (int k = 0; k < row.len; ++k)
        if (entry_ok(row, k, D)) {
          int2* e = place(k);
          e->y = __float_as_int(__int_as_float(e->y) + row.val[k]);
        }
  }
}

constexpr int CSC2_JT = 32;     // rows of W per block, four per lane of a quarter warp
constexpr int CSC2_AB = 8;      // atoms per warp block
constexpr int CSC2_WARPS = 20;
constexpr int CSC2_STRIP = 128; // entries a warp stages at a time
constexpr int CSC2_RS = 32 / CSC2_AB;   // rows of W a warp instruction covers
constexpr int CSC2_TS = 32 + CSC2_RS;    // row length of the tile: 8 atoms x 4 rows fall on 32 banks
constexpr int CSC2_WARP_FLOATS = 2 * CSC2_STRIP + CSC2_AB * CSC2_TS;   // entry strip + [8][36] tile

// The work is the list of (block of 32 rows, block of 8 atoms), rows outermost; every thread block takes an equal run
// of it, so the SMs are loaded evenly whatever J is (a run rarely touches more than two blocks of rows).
// A quarter warp takes every fourth entry: one 8-byte read of the strip (four addresses) and one 512-byte read of u per
// four entries, five wavefronts of shared memory, which bounds this kernel where the codes are dense; the four partial
// sums meet in three shuffles that leave every lane one row.  Where they are sparse the bound is W's way through the
// memory and the latency of a column's few steps: 32 rows (not 64), so that 1408 samples fit beside the tiles and W is read
// and written once; the next block's part of W is in flight while this one's entries are summed; a column's last groups
// are read together; 20 warps (16: 5 % 488 us; 24 or 32, with fewer registers: 461 and 464, small problems 10 % slower).
// 4096 x 10000, K = 1024, against half warps on 64 rows with W loaded when its block begins: 5 % density 514 -> 443 us an
// apply, 2 % 355 -> 274, 1 % 304 -> 206 (3000 x 500, K = 320: 21.9 -> 22.5).
__global__ void __launch_bounds__(CSC2_WARPS * 32) csc_apply_kernel(float* W, RowMap u, int K, int J, int D,
                                                                    float eta, const int* colptr,
                                                                    const int2* ent, int passes, int Kh,
                                                                    const int* status_ro) {
  chain();
  extern __shared__ __align__(16) float smem[];
  if (status_ro != nullptr && (*status_ro & SFB_DEV_BAD_HEADER)) return;
  float* Us = smem;                                   // [Kh][32]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* region = smem + (size_t)Kh * CSC2_JT + warp * CSC2_WARP_FLOATS;
  int2* strip = reinterpret_cast<int2*>(region);
  const int quarter = lane >> 3, q4 = (lane & 7) * 4; // this lane's entries and rows
  const bool up1 = (lane & 16) != 0, up0 = (lane & 8) != 0;
  const int my_row = q4 + (up1 ? 2 : 0) + (up0 ? 1 : 0);   // ... and the row whose sum it ends up with
  float* T = region + 2 * CSC2_STRIP;
  const int nblocks = (D + CSC2_AB - 1) / CSC2_AB;
  const long long work = (long long)((J + CSC2_JT - 1) / CSC2_JT) * nblocks;
  const long long w_lo = work * blockIdx.x / gridDim.x, w_hi = work * (blockIdx.x + 1) / gridDim.x;
  const int n_ent = colptr[(size_t)passes * D];       // padded entries of all slices
  for (long long w0 = w_lo; w0 < w_hi;) {
    const int jb = (int)(w0 / nblocks), ab_lo = (int)(w0 - (long long)jb * nblocks);
    const int ab_hi = (int)min((long long)nblocks, ab_lo + (w_hi - w0));
    w0 += ab_hi - ab_lo;
    const int j0 = jb * CSC2_JT;
    const int jn = min(CSC2_JT, J - j0);
    for (int h = 0; h < passes; ++h) {
      const int i_lo = h * Kh;
      const int i_n = min(Kh, K - i_lo);
      __syncthreads();                                  // the previous slice is no longer read
      // 16-byte asynchronous copies, all in flight together; rows of u are padded to 16 bytes
      for (int t = threadIdx.x; t < i_n * (CSC2_JT / 4); t += CSC2_WARPS * 32) {
        const int i = t / (CSC2_JT / 4), c = (t % (CSC2_JT / 4)) * 4;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(Us + i * CSC2_JT + c);
        const bool in = c < jn;
        const char* src = u.row(i_lo + i) + (in ? (size_t)(j0 + c) * 4 : 0);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      // entries of the warp's next block, on their way while the current one is summed
      constexpr int PRE = CSC2_STRIP / 32;
      int2 pre[PRE];
      auto fetch = [&](int from) {
#pragma unroll
        for (int t = 0; t < PRE; ++t) {
          const int e = from + 32 * t + lane;
          pre[t] = e < n_ent ? ent[e] : make_int2(0, 0);
        }
      };
      // the warp's part of W of a block: lane = atom lane % 8, rows lane / 8 + 4 t
      const int wa = lane & (CSC2_AB - 1), wq = lane / CSC2_AB;
      constexpr int WN = CSC2_JT * CSC2_AB / 32;
      float w_next[WN];
      auto fetch_w = [&](int ab) {
        const int d = ab * CSC2_AB + wa;
        const bool in = ab < ab_hi && d < D;
        const float* wp = W + (size_t)(j0 + wq) * D + (in ? d : 0);
        const size_t step = (size_t)CSC2_RS * D;
        const int rows = in ? jn - wq : 0;
#pragma unroll
        for (int t = 0; t < WN; ++t, wp += step) w_next[t] = CSC2_RS * t < rows ? *wp : 0.f;
      };
      // first entry of the atoms of a block: lane a has atom a's, lanes behind the last atom the end of its column
      const int* cols = colptr + (size_t)h * D;
      auto starts = [&](int ab) { return ab < ab_hi ? cols[ab * CSC2_AB + min(lane, min(CSC2_AB, D - ab * CSC2_AB))] : n_ent; };
      int beg_next = starts(ab_lo + warp);
      fetch_w(ab_lo + warp);
      fetch(__shfl_sync(0xffffffffu, beg_next, 0));
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
      for (int ab = ab_lo + warp; ab < ab_hi; ab += CSC2_WARPS) {
        const int d0 = ab * CSC2_AB;
        const int dn = min(CSC2_AB, D - d0);
        const int beg = beg_next;
        beg_next = starts(ab + CSC2_WARPS);
        int pos = __shfl_sync(0xffffffffu, beg, 0);
        const int end = __shfl_sync(0xffffffffu, beg, dn);
        int strip_lo = pos, strip_hi = pos;             // entries in the strip: [strip_lo, strip_hi)
        auto refill = [&]() {
          __syncwarp();
          // the sample index addresses shared memory: keep it inside the slice whatever the entries hold
#pragma unroll
          for (int t = 0; t < PRE; ++t) strip[32 * t + lane] = make_int2(min(max(pre[t].x, 0), i_n - 1), pre[t].y);
          strip_lo = pos;
          strip_hi = pos + CSC2_STRIP;
          const int nxt = __shfl_sync(0xffffffffu, beg_next, 0);
          fetch(strip_hi < end ? strip_hi : nxt);
          __syncwarp();
        };
        refill();
        float wv[WN];
#pragma unroll
        for (int t = 0; t < WN; ++t) wv[t] = w_next[t];
        fetch_w(ab + CSC2_WARPS);
        for (int dd = 0; dd < dn; ++dd) {
          const int stop = __shfl_sync(0xffffffffu, beg, dd + 1);
          float4 acc0 = make_float4(0.f, 0.f, 0.f, 0.f), acc1 = acc0;
          while (pos < stop) {
            if (pos == strip_hi) refill();              // (warp-uniform)
            auto four = [&](int k, float4& acc) {
              const int2 p = strip[k + quarter];
              const float4 u0 = *reinterpret_cast<const float4*>(Us + p.x * CSC2_JT + q4);
              const float a0 = __int_as_float(p.y);
              acc.x = fmaf(a0, u0.x, acc.x); acc.y = fmaf(a0, u0.y, acc.y);
              acc.z = fmaf(a0, u0.z, acc.z); acc.w = fmaf(a0, u0.w, acc.w);
            };
            const int to = min(stop, strip_hi);         // groups of four never straddle a column or the strip
            int k = pos - strip_lo;
            const int k_end = to - strip_lo;
#pragma unroll 1
            for (; k + 16 <= k_end; k += 16) { four(k, acc0); four(k + 4, acc1); four(k + 8, acc0); four(k + 12, acc1); }
            if (k_end - k == 12) { four(k, acc0); four(k + 4, acc1); four(k + 8, acc0); }
            else if (k_end - k == 8) { four(k, acc0); four(k + 4, acc1); }
            else if (k < k_end) four(k, acc0);
            pos = to;
          }
          acc0.x += acc1.x; acc0.y += acc1.y; acc0.z += acc1.z; acc0.w += acc1.w;
          // quarters 0, 1 go on with rows q4, q4 + 1 and quarters 2, 3 with the other two; then one row each
          float lo = up1 ? acc0.z : acc0.x, hi = up1 ? acc0.w : acc0.y;
          lo += __shfl_xor_sync(0xffffffffu, up1 ? acc0.x : acc0.z, 16);
          hi += __shfl_xor_sync(0xffffffffu, up1 ? acc0.y : acc0.w, 16);
          const float sum = (up0 ? hi : lo) + __shfl_xor_sync(0xffffffffu, up0 ? lo : hi, 8);
          T[dd * CSC2_TS + my_row] = sum;
        }
        __syncwarp();
        // W[j0 + jj][d0 + wa] -= eta * T[wa][jj]: a warp instruction covers four rows x 8 atoms (32-byte segments)
        if (wa < dn) {
          float* wp = W + (size_t)(j0 + wq) * D + d0 + wa;
          const size_t step = (size_t)CSC2_RS * D;
#pragma unroll
          for (int t = 0; t < WN; ++t, wp += step)
            if (CSC2_RS * t < jn - wq) *wp = fmaf(-eta, T[wa * CSC2_TS + CSC2_RS * t + wq], wv[t]);
        }
        __syncwarp();
      }
    }
  }
}

// Slices of the samples: the fewest that let Kh x 128 bytes of u sit beside the warps' tiles.
struct CscSlices {
  int passes, Kh;
};
CscSlices csc_slices(int K) {
  const int tiles = CSC2_WARPS * CSC2_WARP_FLOATS * 4;
  const int kh_max = (220 * 1024 - tiles) / (CSC2_JT * 4) / CSC_CHUNK * CSC_CHUNK;
  CscSlices s;
  s.passes = (K + kh_max - 1) / kh_max;
  s.Kh = ((K + s.passes - 1) / s.passes + CSC_CHUNK - 1) / CSC_CHUNK * CSC_CHUNK;
  s.passes = (K + s.Kh - 1) / s.Kh;
  return s;
}

}  // namespace

// Scratch of the CSC path: masks and offsets [nchunks][D], totals and column starts [slices][D] ints, entries x
// (nnz_capacity + padding).
static long long csc_entries(int K, int D, long long nnz_capacity) {
  return nnz_capacity + 3LL * csc_slices(K).passes * D;
}
static long long csc_ints(int K, int D) {
  const long long nchunks = (K + CSC_CHUNK - 1) / CSC_CHUNK;
  return 2LL * nchunks * D + 2LL * csc_slices(K).passes * D + 1;
}
long long sc_csc_workspace_bytes(int K, int D, long long nnz_capacity) {
  // (a step over the first workers' samples only takes fewer slices of another length: no more entries or ints)
  return pad_to(csc_ints(K, D) * 4, 256) + pad_to(csc_entries(K, D, nnz_capacity) * 8, 256);
}

// The sliced kernel takes any K (more slices); the bound only keeps the chunk tables small.
bool sc_csc_supported(int K) { return K <= (1 << 14); }

namespace {
struct CscScratch {
  uint32_t* mask; int* off; int* total; int* colptr; int2* ent;
};
CscScratch csc_scratch(void* workspace, int K, int D) {
  const int nchunks = (K + CSC_CHUNK - 1) / CSC_CHUNK, passes = csc_slices(K).passes;
  CscScratch w;
  w.mask = reinterpret_cast<uint32_t*>(workspace);
  w.off = reinterpret_cast<int*>(w.mask) + (size_t)nchunks * D;
  w.total = w.off + (size_t)nchunks * D;
  w.colptr = w.total + (size_t)passes * D;
  w.ent = reinterpret_cast<int2*>(reinterpret_cast<char*>(workspace) + pad_to(csc_ints(K, D) * 4, 256));
  return w;
}
}  // namespace

// Atom-major re-sort of the codes into the workspace.  Reads the codes only (not u), so it may run beside
// the forward pass that produces u.
int launch_sc_csc_build(cudaStream_t s, CsrView codes, int K, int D, long long nnz_capacity, void* workspace,
                        int* dev_status, const int* refused) {
  const int nchunks = (K + CSC_CHUNK - 1) / CSC_CHUNK;
  const CscSlices sl = csc_slices(K);
  const CscScratch w = csc_scratch(workspace, K, D);
  const int cps = sl.Kh / CSC_CHUNK, cols = sl.passes * D;
  if (cudaMemsetAsync(w.mask, 0, (size_t)nchunks * D * 4, s) != cudaSuccess) return SFB_ERR_CUDA;
  csc_mask_kernel<<<K, 256, 0, s>>>(codes, K, D, w.mask, dev_status, refused);
  launch_chained(csc_chunk_offsets_kernel, (D + 63) / 64, 64, 0, s, nchunks, cps, D, w.mask, w.off, w.total);
  launch_chained(csc_scan_kernel, 1, 1024, 0, s, cols, w.total, w.colptr);
  launch_chained(csc_fill_kernel, K + (cols + 255) / 256, 256, 0, s, codes, K, D, sl.passes, cps, w.mask, w.off, w.total,
                 w.colptr, w.ent, refused);
  return cudaGetLastError() == cudaSuccess ? 4 : SFB_ERR_CUDA;
}

// The update from a workspace that launch_sc_csc_build filled for the same K, D and codes.
int launch_sc_csc_apply(cudaStream_t s, float* W, RowMap u, int K, int J, int D, float eta, long long nnz_capacity,
                        void* workspace, const int* dev_status_ro) {
  const CscSlices sl = csc_slices(K);
  const CscScratch w = csc_scratch(workspace, K, D);
  static PerDeviceOnce attr_once;
  if (!set_up_device(attr_once, [] { return allow_smem(csc_apply_kernel, 220 * 1024); })) return SFB_ERR_CUDA;
  const long long work = (long long)((J + CSC2_JT - 1) / CSC2_JT) * ((D + CSC2_AB - 1) / CSC2_AB);
  long long blocks = (work + CSC2_WARPS - 1) / CSC2_WARPS;   // at least one block of atoms per warp
  if (blocks > 148) blocks = 148;
  const size_t smem = (size_t)sl.Kh * (CSC2_JT * 4) + (size_t)CSC2_WARPS * CSC2_WARP_FLOATS * 4;
  launch_chained(csc_apply_kernel, (unsigned)blocks, CSC2_WARPS * 32, smem, s, W, u, K, J, D, eta, w.colptr, w.ent, sl.passes, sl.Kh,
                                                                   dev_status_ro);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

}  // namespace sfb
