// egmla_kernels.h - internal launch interface between the C-ABI layer
// (egmla_api.cu) and the kernels.  Not part of the public ABI.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <mutex>

#include "../../include/egmla.h"

namespace egmla {

// Launch with programmatic stream serialisation: the grid is set up while the
// kernel before it on the stream drains, instead of after it has completed and
// flushed.  What holds the order:
//  - every block of a kernel launched this way executes grid_dependency_wait,
//    and before it touches nothing that a kernel before it writes, and writes
//    nothing, so that a completed kernel stands for everything before it;
//  - before the wait a kernel may read inputs that no kernel of the call writes:
//    the split combine copies W_UV, the fp32 one brings it to L2, the projection
//    GEMM copies its weights.  The caller's kernel before the call may write
//    W_UV: the combine must not start before that one is complete, so the bf16
//    split-KV kernel triggers a separate combine only after its own wait.  (An
//    L2 prefetch reads nothing that could be old.  The first projection's weights
//    must not be written by the kernel directly before the layer call.)
// A kernel lets its successor start early (grid_launch_dependents) where that was
// measured to pay: mostly where the successor's blocks take a whole SM each, since
// smaller blocks, started early, crowd onto the first SMs to free up (the R0
// attention took 42 us instead of 33, the layer's query absorption 13 instead
// of 8); the figures stand at the triggers.  Whole calls against plain launches:
// one 777-token prefill 34.8 -> 26.8 us, the fp32 step 38.9 -> 32.6, 8 x 32K decode
// step 51.2 -> 48.9, 128 ragged sequences 84.2 -> 81.7, the d_c 512 step 188 -> 186,
// a layer of 64 x 8K 119.6 -> 115.1, R0 at 8 x 4K 169.6 -> 164.0.
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// SMs of a GB300: what the tile sizes of the small kernels aim at (their results do
// not depend on it; grids that must cover the device ask it)
constexpr int kSms = 152;

// cuTensorMapEncodeTiled through the runtime's driver entry point (no libcuda link)
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(p);
  });
  return fn;
}

// Map of a bf16 tensor of R dimensions (innermost first) with the strides of the
// outer ones in elements; 128-byte swizzle, elements past an end read as zero and
// are not written.
template <size_t R>
bool encode_map(CUtensorMap* map, const void* base, const uint64_t (&dims)[R], const uint64_t (&strides)[R - 1],
                const uint32_t (&box)[R]) {
  const EncodeFn enc = encode_fn();
  if (enc == nullptr) return false;
  cuuint64_t d[R], s[R - 1];
  cuuint32_t b[R], step[R];
  for (size_t i = 0; i < R; ++i) {
    d[i] = dims[i];
    b[i] = box[i];
    step[i] = 1;
    if (i + 1 < R) s[i] = strides[i] * 2;
  }
  auto encode = [&] {
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, R, const_cast<void*>(base), d, s, b, step,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  };
  CUresult r = encode();
  if (r == CUDA_ERROR_INVALID_CONTEXT) {
    // a host thread that has made no call on the device yet has no current context,
    // which the encoder needs: cudaSetDevice makes the device's own current
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaSetDevice(dev) != cudaSuccess) return false;
    r = encode();
  }
  return r == CUDA_SUCCESS;
}

// Lets `kernel` be launched with up to `most` bytes of dynamic shared memory.  The
// limit belongs to the function, not to the calling thread, so every call of a
// kernel sets the same one, the most that any supported shape needs: a call that
// set its own smaller need would take the launch of another thread's larger call
// from under it.
constexpr size_t kSmemMost = 227 * 1024;   // of a block, on this GPU
template <typename K>
cudaError_t allow_smem(K* kernel, size_t most) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(most));
}

struct AppendArgs {
  void* c_pool;
  void* kr_pool;
  int32_t* id_pool;
  const void* c_new;
  const void* kr_new;
  const int32_t* ids_new;
  const int32_t* block_table;
  int max_pages;
  const int32_t* positions;
  int batch, num_pages, page_size;
  int c_row_bytes, kr_row_bytes;
  int32_t* status;
};

// roles recorded by the decode kernel's event trace (eg_mla_debug_set_trace)
constexpr int kTraceRoles = 5;

struct DecodeArgs {
  // shapes
  int H, d_nope, d_rope, d_v, d_c, page_size, vocab;
  int dtype;  // 0 bf16, 1 fp32
  int gate;      // 0 none, 1 gated (the three gate modes below)
  int gate_add;  // gate by c + g (EG_MLA_GATE_ADD_LN) instead of c (*) g
  int gate_ln;   // LayerNorm after the gate (EG_MLA_GATE_MUL_LN, EG_MLA_GATE_ADD_LN)
  float scale_log2;  // softmax scale * log2(e)
  float eps;
  // tensors
  const void* q;
  const void* c_pool;
  const void* kr_pool;
  const int32_t* id_pool;
  const int32_t* block_table;
  int max_pages;
  const int32_t* seq_lens;
  int max_seq_len;
  int batch, num_pages;
  const void* gate_table;
  const float* ln_gamma;
  const float* ln_beta;
  const void* w_uk;
  const void* w_uv;
  void* out;
  int num_splits;
  int early;   // let the kernel after the split-KV kernel start early (it streams weights of its own)
  void* workspace;
  int32_t* status;
  // cache-read test entry outputs (eg_mla_debug_gather)
  void* dump_c;
  void* dump_kr;
  int32_t* dump_ids;
  void* dump_g;
  // pipeline event trace of the decode kernel (eg_mla_debug_set_trace)
  void* trace;
  int trace_ctas, trace_cap;
  // limit of every pipeline wait (ns), and a withheld page copy of the
  // tensor-core decode kernel (eg_mla_debug_set_fault; stall_cta < 0: none)
  uint64_t wait_ns;
  int stall_cta, stall_tile;
};

cudaError_t launch_append(const AppendArgs& a, cudaStream_t st);
// query absorption and split schedule; with `app` non-null its blocks also
// append the new token of every sequence (the pools are read by no block of it)
// `maps`: W_UK as {d_c, d_nope, H} in boxes of {64, 64, 1} and q^C as {d_nope, H,
// batch} in boxes of {64, 1, absorb_tile}
cudaError_t launch_prologue_tc(const DecodeArgs& a, const AppendArgs* app, const CUtensorMap* maps, cudaStream_t st);
// sequences per block of the absorption
int absorb_tile(int d_c, int batch);
// fp32: absorption (with the append blocks of `app` when it is non-null) and the split-KV kernel
cudaError_t launch_decode_f32(const DecodeArgs& a, const AppendArgs* app, cudaStream_t st);
// `wmap` (tensor-core path): W_UV as {d_c, d_v, H} in boxes of {64, 128, 1}
cudaError_t launch_combine(const DecodeArgs& a, bool tc_path, const CUtensorMap* wmap, cudaStream_t st);
// tensor-core split-KV kernel; `maps` = {c_pool map (3-D box of a tile), kr_pool map}.
// *fused (may be null) is set when the split combine ran inside the kernel
// (cooperative launch); otherwise launch_combine must follow.
cudaError_t launch_decode_tc(const DecodeArgs& a, const CUtensorMap* maps, bool dump, cudaStream_t st,
                             bool* fused);
// true if the bf16 tensor-core path has a kernel for these shapes
bool tc_supported(int d_c, int gate);

// R0 decode (egmla_r0.cu): bf16, 16 heads, d_n = d_v = 128, d_r = 64,
// d_c in {192, 256}
struct R0Args {
  const void* q;
  const void* c_pool;
  const void* kr_pool;
  const int32_t* id_pool;
  const int32_t* block_table;
  const int32_t* seq_lens;
  const void* w_ukv;     // [16 * 256, d_c]: per head its 128 key rows, then its 128 value rows
  const void* gate_r0;   // [vocab, 4096]
  const float* ln_gamma;
  const float* ln_beta;
  void* out;
  void* workspace;
  int32_t* status;
  int d_c, vocab, batch, max_pages, num_pages;
  float eps, scale_log2;
};
size_t r0_workspace_bytes(int batch, int max_pages, int num_pages);
cudaError_t launch_decode_r0(const R0Args& a, cudaStream_t st);
// Prefill (egmla_prefill.cu): bf16, d_n = d_v = 128, d_r = 64, d_c a
// multiple of 64 up to 512, any head count.  Prompts packed row after row
// (cu_seqlens [batch + 1] on the device); the pool pointers may be null (no
// cache write).
struct PrefillArgs {
  const void* q;            // [total, H, d_n + d_r]
  const void* c;            // [total, d_c]
  const void* kr;           // [total, d_r]
  const int32_t* ids;       // [total]
  const int32_t* cu_seqlens;
  const void* gate_table;
  const float* ln_gamma;
  const float* ln_beta;
  const void* w_uk;
  const void* w_uv;
  void* out;                // [total, H, d_v]
  void* c_pool;
  void* kr_pool;
  int32_t* id_pool;
  const int32_t* block_table;
  void* workspace;
  int32_t* status;
  int H, d_c, vocab, batch, total, max_seq_len, max_pages, num_pages;
  int gate, gate_add, gate_ln;
  float eps, scale_log2;
};
size_t prefill_workspace_bytes(int batch, int total_tokens, int H, int d_c);
bool prefill_supported(int d_nope, int d_rope, int d_v, int d_c);
// `mark` (may be null) is called with (stream, true) just before the
// attention kernel's launch and (stream, false) just after it.
cudaError_t launch_prefill(const PrefillArgs& a, cudaStream_t st, void (*mark)(cudaStream_t, bool));
// The gate table G = E W^UE^T (Section 3 Eqs. 3-4 for every vocabulary
// entry): E [vocab, d_e], W^UE [d_c, d_e] bf16 row-major, G [vocab, d_c] bf16;
// d_e a multiple of 64 up to 512, d_c a multiple of 64 (egmla_prefill.cu).
cudaError_t launch_gate_table(const void* emb, const void* w_ue, int vocab, int d_e, int d_c, void* table,
                              int32_t* status, cudaStream_t st);
// out[b][n] = sum_k x[b][k] W[n][k] for b < batch, n < n_out: W [n_out, k] and
// x [batch, k] bf16 row-major (16-byte aligned, k % 8 == 0), out fp32 or
// bf16 with row stride ldo elements (egmla_linear.cu).  Launched with
// programmatic stream serialisation: the weight copies may start while the
// kernel before it on the stream still runs.
cudaError_t launch_linear_tc(const void* w, int n_out, int k, const void* x, int batch, void* out, int ldo,
                             bool out_f32, int32_t* status, cudaStream_t st);
// the launch shape launch_linear_tc picks: cluster size (CTAs splitting k),
// ring stages, and the clusters of that size the device holds at once
cudaError_t linear_tc_plan(int n_out, int k, int batch, int* cluster, int* stages, int* max_clusters);

}  // namespace egmla

// The step inside eg_mla_layer_decode (egmla_api.cu): eg_mla_step (`append`)
// or eg_mla_decode, whose split-KV kernel lets the output projection after it
// start early.  `launch` false: its arguments are checked and nothing is launched.
int egmla_layer_step(const eg_mla_dims* dims, bool append, void* c_pool, void* krope_pool, int32_t* id_pool,
                     const void* c_new, const void* krope_new, const int32_t* ids_new, const int32_t* positions,
                     const void* q, const int32_t* block_table, int32_t max_pages_per_seq, const int32_t* seq_lens,
                     int32_t max_seq_len, int32_t batch, int32_t num_pages, const void* gate_table,
                     const float* ln_gamma, const float* ln_beta, const void* w_uk, const void* w_uv, void* out,
                     int32_t num_splits, void* workspace, size_t workspace_bytes, int32_t* dev_status, void* stream,
                     bool launch);
