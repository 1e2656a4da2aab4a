// Tensor-core (tcgen05 / TMEM / TMA) side of the SF hot path: interface used by the C-ABI host code.
#pragma once

#include "common.cuh"

namespace sfb {

struct UmmaPlan;   // tensor maps and launch geometry for one descriptor

// Builds the plan for a TF32 or BF16 descriptor.
int umma_plan_create(const sfb_desc& d, const Layout& l, UmmaPlan** out);
void umma_plan_destroy(UmmaPlan* p);

// z = W a on the tensor cores followed by the model epilogue; factors go through u / v row maps.
// for_apply (compensated path): umma_apply of exactly these u / v rows, all K pairs, follows before anything else
// changes them: the kernels that write the factors also write the apply's correction operands (one use).
// workers > 0: only that many workers' samples (X, aux, u, v start at the first of them).
// defer_v: a copy of the factor v that runs on the side stream is left there; the caller calls umma_join on every path.
// extra: what the finishing pass does besides (header, flags of nonzero rows).
int umma_forward(UmmaPlan* p, cudaStream_t s, const void* W, const __nv_bfloat16* w_shadow, const void* X,
                 const sfb_aux* aux, RowMap u, RowMap v, int* dev_status, int workers = 0, bool for_apply = false,
                 const FinishExtra& extra = FinishExtra(), bool defer_v = false);

int umma_join(UmmaPlan* p, cudaStream_t s);

// Z rows (fp32) = A rows (the path's value type) times Wop^T on the tensor cores; no epilogue beyond the store.
// w_corr: on the compensated path, W's correction operand (launch_split_k of W's rows, B side); w_shadow plays
// that part in umma_forward.
int umma_forward_rows(UmmaPlan* p, cudaStream_t s, const void* Wop, RowMap a, RowMap z, int* dev_status,
                      float2* stats = nullptr, int* n_parts_out = nullptr, int* part_cols_out = nullptr,
                      int* k_splits_out = nullptr, int max_splits = 1, long long split_stride = 0, int workers = 0,
                      const void* w_corr = nullptr, bool a_corr_ready = false);

// Sparse coding: u rows = dense code rows `a` (fp32) times W^T minus the data rows Xdata [K][J].
// a_corr: what umma_codes_corr returned, if the kernel that made the rows `a` has written it.
int umma_forward_sc(UmmaPlan* p, cudaStream_t s, const void* W, RowMap a, RowMap u, const float* Xdata, int* dev_status,
                    int workers = 0, const void* w_corr = nullptr, bool for_apply = false, const CorrOut* a_corr = nullptr);
// Compensated path: where the kernel that makes the dense code rows may write their correction operands (the
// forward's; with for_apply also the apply's, for which the code rows are the v rows).  Empty on other paths.
CorrOut umma_codes_corr(UmmaPlan* p, bool for_apply);

// Forgets correction operands a factor stage left for "its" apply (a caller that applies a buffer of its own).
void umma_drop_corr(UmmaPlan* p);

// W <- W - eta * U^T V on the tensor cores with the write-back (and bf16 shadow refresh) fused.
// u_rows / v_rows: the factor rows (normally the U and V blocks of the SF buffer's worker streams).
// directory (optional): the SF buffer's directory (sf_buf + 128) of a compacted buffer, whose rows behind each
// worker's pair count are zeros: reduction blocks that hold only such rows are skipped.
// check (optional, compensated path): the header check of the buffer, done before W is touched.
int umma_apply(UmmaPlan* p, cudaStream_t s, void* W, __nv_bfloat16* w_shadow, RowMap u_rows, RowMap v_rows, float eta,
               int K, const int* dev_status, const void* directory = nullptr, const HeaderCheck* check = nullptr);

// fp32 path, large dense problems: the two contractions on the tensor cores, each fp32 operand as three bf16 parts
// (umma_f32.cu).
struct F32Tc;
// *out = nullptr with SFB_OK: the CUDA cores do it.  A whole step is not estimated to be faster than theirs, whose forward takes
// cores_forward_us, or there is no room for the workspace, or the kernels cannot be set up on this device.
int f32tc_create(const sfb_desc& d, cudaStream_t s, double cores_forward_us, F32Tc** out);
void f32tc_destroy(F32Tc* t);
// Products of K samples (X, or X - Xb) with W, as `nsplit` partial products of rows *z (which are u itself, or the
// workspace), and the samples (differences) into v where v.base != nullptr.
int f32tc_forward(F32Tc* t, cudaStream_t s, const float* W, const float* X, const float* Xb, int K, RowMap u, RowMap v,
                  int* dev_status, RowMap* z, int* nsplit, long long* split_stride);
// Words that say operands hold values which bf16 parts cannot carry (infinities, NaN, 2^36 and more), or that an update has very
// few rows: the CUDA-core kernels then do the work.  The forward's is cleared by the finishing pass behind it, the update's by what precedes it (the finishing pass
// of the same step, which hands the forward's on, or the header check).
int* f32tc_bad_forward(F32Tc* t);
int* f32tc_bad_apply(F32Tc* t);
uint8_t* f32tc_flags(F32Tc* t);         // where the finishing pass leaves which u rows are nonzero
// Lists the rows with nonzero u among the first K: f32tc_apply's when it gets no list of its own.
// active / n_active (optional): how many of these flags are set.  refused: see is_refused (u is not read, the list not to be used).
int f32tc_list(F32Tc* t, cudaStream_t s, RowMap u, int K, bool flags_ready, const uint8_t* active, int* n_active,
               const int* refused);
// W -= eta * sum u_i v_i^T over the listed rows, in that order (idx / n_rows, or f32tc_list's).  The sum depends on the listed
// rows alone, so leaving out zero rows, as a compacted buffer does, changes no bit.
// v_planes: the forward of the same step made v's planes (all K rows).
// left_out: rows that are not listed are not part of the update, whatever their v holds; otherwise a row without a nonzero u
// still makes a NaN of a v that is not finite (the CUDA cores then take all K rows).
// refused: see is_refused (no row is read then).
int f32tc_apply(F32Tc* t, cudaStream_t s, float* W, RowMap u, RowMap v, int K, float eta, int* dev_status, const int* idx,
                const int* n_rows, bool v_planes, bool left_out, const int* refused);

}  // namespace sfb
