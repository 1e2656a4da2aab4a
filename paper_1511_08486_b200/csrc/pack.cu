// SF buffer bookkeeping: header and directory, CSR code streams, header validation.
// The buffer is the message the P workers would broadcast at commit() (Section 4.2); the layout is
// the wire format documented in include/sfb.h.  Integer offset arithmetic and copies only.
#include "common.cuh"

namespace sfb {
namespace {

HeaderImage make_header(const sfb_desc& d, const Layout& l, uint32_t clock) {
  HeaderImage h;
  h.magic = 0x31424653u;
  h.version = 1;
  h.model = (uint8_t)d.model;
  h.dtype = (l.es == 2) ? 1 : 0;
  h.flags = d.v_sparse ? 1u : 0u;
  h.P = d.P; h.B = d.B; h.J = d.J; h.D = d.D;
  h.clock = clock;
  h.ldu = l.ldu; h.ldv = l.ldv;
  h.stream_stride = (uint64_t)l.stream_stride;
  h.total_bytes = (uint64_t)l.total_bytes;
  h.streams_off = (uint64_t)l.streams_off;
  h.cap_p = (uint32_t)l.cap_p;
  return h;
}

__global__ void write_header_kernel(const __grid_constant__ Commit c) { chain(); write_header(c, threadIdx.x, blockDim.x); }

__global__ void check_header_kernel(const __grid_constant__ HeaderCheck c) {
  chain();
  report_header(c, header_matches(c, expected_header(c)));
}

// grid.x = P workers; each block copies its worker's CSR rows into the stream.
__global__ void __launch_bounds__(256) pack_csr_kernel(char* buf, long long streams_off, long long stream_stride,
                                                       long long u_bytes, long long rp_bytes, long long idx_bytes,
                                                       int B, int cap_p, int D, const uint32_t* __restrict__ rowptr,
                                                       const uint32_t* __restrict__ idx, const float* __restrict__ val,
                                                       int* dev_status, const __grid_constant__ Commit commit) {
  const int p = blockIdx.x;
  const int part = blockIdx.y, parts = gridDim.y;   // the worker's words are spread over gridDim.y blocks
  if (commit.buf != nullptr && p == 0 && part == 0) write_header(commit, threadIdx.x, 256);
  char* vb = buf + streams_off + (long long)p * stream_stride + u_bytes;
  uint32_t* rp = reinterpret_cast<uint32_t*>(vb);
  uint32_t* ix = reinterpret_cast<uint32_t*>(vb + rp_bytes);
  float* vl = reinterpret_cast<float*>(vb + rp_bytes + idx_bytes);
  const uint32_t base = rowptr[(size_t)p * B];
  const uint32_t nnz_true = rowptr[(size_t)(p + 1) * B] - base;
  const uint32_t nnz = nnz_true < (uint32_t)cap_p ? nnz_true : (uint32_t)cap_p;
  if (nnz_true > (uint32_t)cap_p && threadIdx.x == 0 && part == 0) atomicOr(dev_status, SFB_DEV_CAPACITY);
  const int rp_words = (int)(rp_bytes / 4);
  for (int t = part * blockDim.x + threadIdx.x; t < rp_words; t += parts * blockDim.x) {
    uint32_t r = 0u;
    if (t <= B) {
      r = rowptr[(size_t)p * B + t] - base;
      if (r > nnz) r = nnz;
    }
    rp[t] = r;
  }
  const int idx_words = (int)(idx_bytes / 4);
  bool bad = false;
  for (int t = part * blockDim.x + threadIdx.x; t < idx_words; t += parts * blockDim.x) {
    uint32_t c = 0u;
    float a = 0.f;
    if ((uint32_t)t < nnz) {
      c = idx[base + t];
      a = val[base + t];
      if (c >= (uint32_t)D) bad = true;
    }
    ix[t] = c;
    vl[t] = a;   // val block is padded to the same number of 4-byte words (fp32 values)
  }
  if (bad) atomicOr(dev_status, SFB_DEV_BAD_INDEX);
}

}  // namespace

Commit make_commit(void* sf_buf, const sfb_desc& d, const Layout& l, uint32_t clock, const uint32_t* rowptr) {
  Commit c;
  c.buf = reinterpret_cast<char*>(sf_buf);
  c.h = make_header(d, l, clock);
  c.u_bytes = l.u_bytes;
  c.rowptr = rowptr;
  return c;
}

int launch_write_header(cudaStream_t s, void* sf_buf, const sfb_desc& d, const Layout& l, uint32_t clock,
                        const uint32_t* rowptr) {
  launch_chained(write_header_kernel, 1, 256, 0, s, make_commit(sf_buf, d, l, clock, rowptr));
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

HeaderCheck make_check(const void* sf_buf, const sfb_desc& d, const Layout& l, int* dev_status) {
  HeaderCheck c;
  c.buf = reinterpret_cast<const char*>(sf_buf);
  c.h = make_header(d, l, 0);
  c.dev_status = dev_status;
  return c;
}

int launch_check_header(cudaStream_t s, const HeaderCheck& check) {
  launch_chained(check_header_kernel, 1, 1, 0, s, check);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

int launch_pack_csr(cudaStream_t s, void* sf_buf, const sfb_desc& d, const Layout& l, const uint32_t* rowptr,
                    const uint32_t* idx, const float* val, int* dev_status, const Commit& commit) {
  const int parts = (l.cap_p + 2047) / 2048 < 1 ? 1 : ((l.cap_p + 2047) / 2048 > 64 ? 64 : (l.cap_p + 2047) / 2048);
  pack_csr_kernel<<<dim3(d.P, parts), 256, 0, s>>>(reinterpret_cast<char*>(sf_buf), l.streams_off, l.stream_stride, l.u_bytes,
                                      l.rp_bytes, l.idx_bytes, d.B, l.cap_p, d.D, rowptr, idx, val, dev_status, commit);
  return cudaGetLastError() == cudaSuccess ? 1 : SFB_ERR_CUDA;
}

}  // namespace sfb
