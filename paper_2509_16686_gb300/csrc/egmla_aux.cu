// egmla_aux.cu - the small kernels around the tensor-core decode kernel:
//   append_latent_kernel   cache write of the new token (bit-exact copy)
//   prologue_*_kernel      per-step query absorption q^ = W_UK,h^T q^C, the
//                          page prefix sums and split start records of the
//                          split-KV schedule, and (in eg_mla_step) the append
//   combine_*_kernel       log-sum-exp merge of the split partials and the
//                          W_UV,h up-projection of the latent output (fp32 on
//                          CUDA cores, bf16 on tcgen05), for the launches whose
//                          decode kernel does not fuse it
//   decode_f32_kernel      the fp32 specialisation of the split-KV decode
//                          (exact fp32 arithmetic on CUDA cores; bf16 runs on
//                          tcgen05 in egmla_decode_tc.cu)
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "egmla_common.cuh"
#include "egmla_kernels.h"
#include "egmla_ptx.cuh"

namespace egmla {

// ------------------------------------------------------------------ append
// The new token's rows of sequence b, copied by `nthr` threads (this one is
// `thr`); the row copies are 16-byte vectors (the row byte counts allow it for
// every supported shape).
__device__ void append_row(const AppendArgs& a, int b, int thr, int nthr) {
  const int pos = a.positions[b];
  if (pos < 0) return;
  const int lp = pos / a.page_size;
  if (lp >= a.max_pages) {
    if (thr == 0) report_status(a.status, kStatusOutOfRange);
    return;
  }
  const int page = a.block_table[static_cast<size_t>(b) * a.max_pages + lp];
  if (page < 0 || page >= a.num_pages) {
    if (thr == 0) report_status(a.status, kStatusOutOfRange);
    return;
  }
  const size_t row = static_cast<size_t>(page) * a.page_size + pos % a.page_size;
  uint4* cd = reinterpret_cast<uint4*>(static_cast<uint8_t*>(a.c_pool) + row * a.c_row_bytes);
  const uint4* cs = reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(a.c_new) +
                                                   static_cast<size_t>(b) * a.c_row_bytes);
  for (int i = thr; i < a.c_row_bytes / 16; i += nthr) cd[i] = cs[i];
  uint4* kd = reinterpret_cast<uint4*>(static_cast<uint8_t*>(a.kr_pool) + row * a.kr_row_bytes);
  const uint4* ks = reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(a.kr_new) +
                                                   static_cast<size_t>(b) * a.kr_row_bytes);
  for (int i = thr; i < a.kr_row_bytes / 16; i += nthr) kd[i] = ks[i];
  if (a.id_pool != nullptr && a.ids_new != nullptr && thr == 0) a.id_pool[row] = a.ids_new[b];
}

// one block per sequence
__global__ void append_latent_kernel(const AppendArgs a) { append_row(a, blockIdx.x, threadIdx.x, blockDim.x); }

// ------------------------------------------------------------------ helpers
// brings the 128-byte line of p into L2
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<uint64_t>(p)));
}

// v[i] (i < 32) summed over the warp; lane t returns the sum of v[t]
__device__ __forceinline__ float reduce32_transpose(float (&v)[32], int lane) {
#pragma unroll
  for (int o = 16, len = 32; o > 0; o >>= 1, len >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (i < len / 2) {
        const float keep = up ? v[i + len / 2] : v[i];
        const float send = up ? v[i] : v[i + len / 2];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
  }
  return v[0];
}

// ------------------------------------------------------------------ prologue
// Exclusive prefix sum of the schedule units per sequence (its pages plus
// kSegCost when it has any): cu[b] = sum_{b'<b} units_b', cu[batch] = total; a
// scan by the block's first warp, 32 sequences per pass.
__device__ void page_prefix_sums(const int32_t* seq_lens, int batch, int page_size, int32_t* cu) {
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  int32_t carry = 0;
  for (int base = 0; base < batch; base += 32) {
    const int b = base + lane;
    const int L = b < batch ? seq_lens[b] : 0;
    const int np = L > 0 ? (L + page_size - 1) / page_size + kSegCost : 0;
    int incl = np;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (b < batch) cu[b] = carry + incl - np;
    carry += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) cu[batch] = carry;
}

// The same prefix sums by a whole block of 256 threads (a warp scan per 256
// sequences, the warps' totals through shared memory), written to global
// memory and to the block's shared copy cu_s (batch + 1 entries); one load
// round trip per 256 sequences.
__device__ void page_prefix_sums_block(const int32_t* seq_lens, int batch, int page_size, int32_t* cu,
                                       int32_t* cu_s, int32_t* wsum) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x / 32;
  int32_t carry = 0;
  for (int base = 0; base < batch; base += blockDim.x) {
    const int b = base + tid;
    const int L = b < batch ? seq_lens[b] : 0;
    const int np = L > 0 ? (L + page_size - 1) / page_size + kSegCost : 0;
    int incl = np;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < nw; ++w) {
      const int v = wsum[w];
      before += w < warp ? v : 0;
      total += v;
    }
    if (b < batch) {
      const int32_t e = carry + before + incl - np;
      cu[b] = e;
      cu_s[b] = e;
    }
    carry += total;
    __syncthreads();   // wsum is rewritten by the next pass
  }
  if (tid == 0) {
    cu[batch] = carry;
    cu_s[batch] = carry;
  }
}

// Start record of every split (see SplitStart), from the prefix sums this
// block just wrote (its shared copy).  Split c
// owns units [c chunk, (c + 1) chunk); its first sequence is the last one whose
// first unit is at most c chunk (empty sequences skipped), as in the decode
// kernel's walk.
__device__ void split_starts(const int32_t* cu, const int32_t* seq_lens, int batch, int num_splits,
                             const int32_t* __restrict__ block_table, int max_pages, SplitStart* starts) {
  const int total = cu[batch];
  const int chunk = split_chunk(total, num_splits);
  for (int c = threadIdx.x; c < num_splits; c += blockDim.x) {
    SplitStart st;
    const int g0 = c * chunk;
    st.g1 = min(g0 + chunk, total);
    st.b = st.lp = st.lp_end = st.L = st.npages = st.pad = 0;
    st.done = g0 >= st.g1;
    if (!st.done) {
      int lo = 0, hi = batch - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cu[mid] <= g0) lo = mid; else hi = mid - 1;
      }
      while (lo < batch - 1 && cu[lo + 1] <= g0) ++lo;
      const int base = cu[lo] + kSegCost;   // unit of the sequence's first page
      st.b = lo;
      st.lp = max(g0 - base, 0);
      st.lp_end = min(st.g1, cu[lo + 1]) - base;
      st.L = seq_lens[lo];
      st.done = st.lp_end <= st.lp;
      if (!st.done) st.npages = min(kStartPages, min(st.lp_end, max_pages) - st.lp);
    }
    for (int i = 0; i < kStartPages; ++i)
      st.page[i] = i < st.npages ? block_table[static_cast<size_t>(st.b) * max_pages + st.lp + i] : -1;
    const int4* src = reinterpret_cast<const int4*>(&st);
    int4* dst = reinterpret_cast<int4*>(starts + c);
#pragma unroll
    for (int k = 0; k < 4; ++k) dst[k] = src[k];
  }
}

// The schedule, by one block of 256 threads: the combine's counters zeroed, the
// page prefix sums and the splits' start records.  `smem` (`words` ints): the
// prefix sums in shared memory too where they fit, so that the splits'
// searches read them there; `wsum`: eight more ints.
__device__ void schedule_block(const int32_t* seq_lens, int batch, int page_size, int32_t* cu, uint32_t* seq_done,
                               int num_splits, const int32_t* block_table, int max_pages, SplitStart* starts,
                               int32_t* smem, int words, int32_t* wsum) {
  if (seq_done != nullptr)
    for (int i = threadIdx.x; i < batch; i += blockDim.x) seq_done[i] = 0u;
  if (batch + 1 <= words) {
    page_prefix_sums_block(seq_lens, batch, page_size, cu, smem, wsum);
    __syncthreads();   // the prefix sums are visible to the whole block
    split_starts(smem, seq_lens, batch, num_splits, block_table, max_pages, starts);
  } else {
    page_prefix_sums(seq_lens, batch, page_size, cu);
    __syncthreads();
    split_starts(cu, seq_lens, batch, num_splits, block_table, max_pages, starts);
  }
}

// Tensor-core path: the query absorption as a tcgen05 GEMM per head,
//   D[f, b] = q^_{b,h}[f] = sum_n W_UK,h[n][f] q^C_{b,h}[n].
// A block takes (head, 128 features, `nt` sequences): W_UK,h is the M = 128
// operand read MN-major (features contiguous), q^C the K-major N operand, both
// copied by TMA in 64-row / 64-column boxes (rows past d_nope and past the
// batch read as zero; W_UK with an L2 evict-last hint: it stays in L2 across
// steps).  The fp32 accumulator's lanes are features: a lane stores (q^ (*)
// gamma) rounded to bf16 in the prepared query blocks (qop_offset layout), and
// since a warp's quadrant is one chunk of kSumFeatures, the chunk's partials of
// w_h = sum_f bf16(q^ gamma)_f and b_h = q^_h . beta for 16 sequences take one
// transposing reduction of 32 values.  The blocks of the first features also
// copy q^R.  Block 0: the schedule; the blocks after the tiles: the appends, a
// warp per sequence (no block of this kernel reads the pools).
// A block's time is one round of copies, its MMAs and its stores.  On CUDA
// cores the absorption was bound by its shared-memory reads and grew with the
// batch: 13.1 us at 128 sequences with d_c 192 and 18.9 with d_c 512, 8.3 at 64
// with d_c 256; now 4.7, 6.2 and 4.6 (kernel alone, warm); equal at 8.
constexpr int kPmThreads = 256;
constexpr int kPmTile = 128;                    // features per block (the MMA's M)
constexpr uint32_t kPmAtomRow = 128;            // bytes of a swizzled 64-element row
constexpr int kPmMaxSeq = 128;                  // sequences per block, at most (the MMA's N)
constexpr int kPmMaxNope = 256;

struct PmBars {
  uint64_t full[kPmMaxNope / 64];
  uint64_t done;
  uint32_t tmem_base;
  int abort;
};

__host__ __device__ constexpr uint32_t pm_smem(int nk, int nt) {
  return static_cast<uint32_t>(nk) * 64 * kPmAtomRow * 2 + static_cast<uint32_t>(nk) * nt * kPmAtomRow + 1024 +
         sizeof(PmBars);
}

static_assert(pm_smem(kPmMaxNope / 64, kPmMaxSeq) <= kSmemMost, "shared memory");

__global__ void __launch_bounds__(kPmThreads)
prologue_tc_kernel(const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap qmap,
                    const __nv_bfloat16* __restrict__ q, const float* __restrict__ gamma,
                    const float* __restrict__ beta, const int32_t* __restrict__ seq_lens, int batch, int d_nope,
                    int d_rope, int d_c, int page_size, uint8_t* __restrict__ qprep, size_t qstride,
                    int32_t* __restrict__ cu, uint32_t* __restrict__ seq_done, int num_splits,
                    const int32_t* __restrict__ block_table, int max_pages, SplitStart* __restrict__ starts, int nt,
                    uint64_t wait_ns, int32_t* status, const AppendArgs app) {
  extern __shared__ uint8_t pm_raw[];
  uint8_t* smem = pm_raw + ((1024u - (smem_u32(pm_raw) & 1023u)) & 1023u);
  constexpr int H = 16;
  const int mt = (d_c + kPmTile - 1) / kPmTile, nbg = (batch + nt - 1) / nt;
  const int ntiles = q != nullptr ? H * mt * nbg : 0;   // (the cache-read test entry: the schedule only)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (blockIdx.x == 0 || blockIdx.x > static_cast<unsigned>(ntiles)) {
    grid_launch_dependents();
    grid_dependency_wait();
    if (blockIdx.x == 0) {
      int32_t* words = reinterpret_cast<int32_t*>(smem);
      constexpr int kWords = 4096;
      static_assert(pm_smem(1, 16) >= 1024 + (kWords + 8) * 4, "schedule area");
      schedule_block(seq_lens, batch, page_size, cu, seq_done, num_splits, block_table, max_pages, starts, words + 8,
                     kWords, words);
    } else {
      const int b = (static_cast<int>(blockIdx.x) - (ntiles + 1)) * (kPmThreads / 32) + warp;
      if (b < app.batch) append_row(app, b, lane, 32);
    }
    return;
  }
  const int item = static_cast<int>(blockIdx.x) - 1;
  const int h = item % H, fm = (item / H) % mt, b0 = (item / (H * mt)) * nt;
  // the last tile of a latent that is no multiple of 128 starts early and
  // skips the features of the tile before it
  const int f_first = fm * kPmTile, f0 = min(f_first, d_c - kPmTile);
  const int nk = (d_nope + 63) / 64, nb = min(nt, batch - b0);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t atom = static_cast<uint32_t>(nk) * 64 * kPmAtomRow;   // one 64-feature column of W, all rows
  const uint32_t q_off = 2 * atom, q_chunk = static_cast<uint32_t>(nt) * kPmAtomRow;
  PmBars& bars = *reinterpret_cast<PmBars*>(smem + q_off + nk * q_chunk);
  volatile int* abort_flag = &bars.abort;
  uint32_t tmem_cols = 32;
  while (tmem_cols < static_cast<uint32_t>(nt)) tmem_cols <<= 1;
  if (tid == 0) {
    for (int k = 0; k < nk; ++k) mbar_init(smem_u32(&bars.full[k]), 1);
    mbar_init(smem_u32(&bars.done), 1);
    bars.abort = 0;
    fence_mbar_init();
    prefetch_tensormap(&wmap);
    prefetch_tensormap(&qmap);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bars.tmem_base), tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars.tmem_base;
  grid_launch_dependents();
  grid_dependency_wait();
  if (warp == 0) {
    if (elect_one()) {
      const uint64_t keep = policy_evict_last(), once = policy_evict_first();
      for (int k = 0; k < nk; ++k) {
        const uint32_t fb = smem_u32(&bars.full[k]);
        mbar_arrive_expect_tx(fb, 2 * 64 * kPmAtomRow + q_chunk);
        for (int c = 0; c < 2; ++c)
          tma_load_3d(sbase + c * atom + k * 64 * kPmAtomRow, &wmap, f0 + 64 * c, 64 * k, h, fb, keep);
        tma_load_3d(sbase + q_off + k * q_chunk, &qmap, 64 * k, h, b0, fb, once);
      }
      const uint32_t idesc = idesc_bf16(kPmTile, nt, 1, 0);
      const uint64_t wd = smem_desc(sbase, atom, 1024, kSwizzle128B);
      for (int k = 0; k < nk; ++k) {
        // every copy lands before the block can leave (own flag: bounded, not cut short)
        volatile int own = 0;
        if (!mbar_wait(smem_u32(&bars.full[k]), 0, &own, wait_ns)) *abort_flag = 1;
        if (*abort_flag) continue;
        tc_fence_after();
        const uint64_t qd = smem_desc(sbase + q_off + k * q_chunk, 16, 1024, kSwizzle128B);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_bf16_ss(tmem, wd + ((k * 64 * kPmAtomRow + kk * 2048) >> 4), qd + ((kk * 32) >> 4), idesc,
                      (k > 0 || kk > 0) ? 1u : 0u);
      }
      mma_commit(smem_u32(&bars.done));
    }
    __syncwarp();
  } else if (fm == 0) {
    // meanwhile: q^R of the block's sequences, 16 bytes at a time
    const int qrow = d_nope + d_rope, pr = d_rope / 8;
    for (int i = tid - 32; i < nb * pr; i += kPmThreads - 32) {
      const int j = i / pr, r = 8 * (i % pr);
      *reinterpret_cast<uint4*>(qprep + static_cast<size_t>(b0 + j) * qstride + qprep_lat_bytes(d_c) + qop_offset(h, r)) =
          *reinterpret_cast<const uint4*>(q + (static_cast<size_t>(b0 + j) * H + h) * qrow + d_nope + r);
    }
  }
  // ---- epilogue: warp = (lane quadrant, every other group of 16 sequences)
  const int quad = warp & 3, f = f0 + 32 * quad + lane;
  const float gm = gamma ? gamma[f] : 1.f;
  const float bt = beta ? beta[f] : 0.f;
  __syncwarp();
  bool ok = mbar_wait(smem_u32(&bars.done), 0, abort_flag, wait_ns);
  ok = __all_sync(0xffffffffu, ok) && *abort_flag == 0;
  tc_fence_after();
  if (ok && f0 + 32 * quad >= f_first) {   // uniform in the warp
    const int fc = (f0 + 32 * quad) / kSumFeatures;
    for (int c0 = 16 * (warp >> 2); c0 < nb; c0 += 32) {
      float v[16];
      tmem_ld16(tmem + (static_cast<uint32_t>(32 * quad) << 16) + c0, v);
      tmem_wait_ld();
      float part[32];
      uint8_t* qb = qprep + static_cast<size_t>(b0 + c0) * qstride + qlat_offset(h, f, d_c);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const __nv_bfloat16 bq = __float2bfloat16_rn(v[j] * gm);
        part[j] = __bfloat162float(bq);
        part[16 + j] = v[j] * bt;
        if (c0 + j < nb) *reinterpret_cast<__nv_bfloat16*>(qb + j * qstride) = bq;
      }
      const float sum = reduce32_transpose(part, lane);   // lane t: value t
      if (c0 + (lane & 15) < nb) {
        float* sums = reinterpret_cast<float*>(qprep + static_cast<size_t>(b0 + c0 + (lane & 15)) * qstride +
                                               qprep_lat_bytes(d_c) + qprep_rope_bytes(d_rope));
        sums[(fc * 2 + (lane >> 4)) * 16 + h] = sum;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, tmem_cols);
  if (tid == 0 && *abort_flag) report_status(status, kStatusTimeout);
}

// fp32 path: q^ [H, d_c] and q^R [H, d_rope] in fp32, row-major.  Block 0: the
// page prefix sums; then one block per (head, 64 features, group of up to
// kPfBatch sequences); then the append blocks of a step.  A thread takes four
// features of W_UK,h and every 16th of its d_nope rows, each row loaded once
// for all the group's sequences with no load depending on another; the 16
// parts of a sum are added in shared memory.  Bound by the latency of one
// round of loads: 17.5 us for 8 sequences when a thread walked all of d_nope
// for one sequence, 6 us now (ncu, cold caches).
constexpr int kPfBatch = 8, kPfFeat = 64, kPfParts = 16, kPfRows = 8;

__global__ void __launch_bounds__(256)
prologue_f32_kernel(const float* __restrict__ q, const float* __restrict__ w_uk, const int32_t* __restrict__ seq_lens,
                    int batch, int H, int d_nope, int d_rope, int d_c, int page_size, uint8_t* __restrict__ qprep,
                    size_t qstride, int32_t* __restrict__ cu, const AppendArgs app) {
  __shared__ float qn[kPfBatch][256];
  __shared__ __align__(16) float red[kPfParts][kPfBatch][kPfFeat];
  const int nfc = (d_c + kPfFeat - 1) / kPfFeat, nbg = (batch + kPfBatch - 1) / kPfBatch;
  const int nabs = H * nfc * nbg;
  grid_launch_dependents();
  grid_dependency_wait();
  if (blockIdx.x == 0) {
    page_prefix_sums(seq_lens, batch, page_size, cu);
    return;
  }
  if (blockIdx.x > static_cast<unsigned>(nabs)) {   // no block of this kernel reads the pools
    append_row(app, blockIdx.x - (nabs + 1), threadIdx.x, blockDim.x);
    return;
  }
  const int item = static_cast<int>(blockIdx.x) - 1;
  const int h = item % H, fc = (item / H) % nfc, b0 = (item / (H * nfc)) * kPfBatch;
  const int nb = min(kPfBatch, batch - b0), tid = threadIdx.x;
  const int qrow = d_nope + d_rope;
  const int f4 = 4 * (tid % (kPfFeat / 4)), part = tid / (kPfFeat / 4), f = fc * kPfFeat + f4;
  const float* w = w_uk + static_cast<size_t>(h) * d_nope * d_c + f;
  // the first kPfRows rows of this thread, in flight while q is staged
  float4 wv[kPfRows];
  auto load_rows = [&](int n0) {
#pragma unroll
    for (int k = 0; k < kPfRows; ++k) {
      const int n = n0 + kPfParts * k;
      wv[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (f < d_c && n < d_nope) wv[k] = __ldg(reinterpret_cast<const float4*>(w + static_cast<size_t>(n) * d_c));
    }
  };
  load_rows(part);
  for (int i = tid; i < kPfBatch * d_nope; i += 256) {
    const int j = i / d_nope, n = i % d_nope;
    qn[j][n] = j < nb ? q[(static_cast<size_t>(b0 + j) * H + h) * qrow + n] : 0.f;
  }
  __syncthreads();
  float4 acc[kPfBatch];
#pragma unroll
  for (int j = 0; j < kPfBatch; ++j) acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int n0 = part; n0 < d_nope; n0 += kPfParts * kPfRows) {
    if (n0 != part) load_rows(n0);
#pragma unroll
    for (int k = 0; k < kPfRows; ++k) {
      const int n = n0 + kPfParts * k;
      if (n >= d_nope) break;
#pragma unroll
      for (int j = 0; j < kPfBatch; ++j) {
        const float x = qn[j][n];
        acc[j].x = fmaf(wv[k].x, x, acc[j].x);
        acc[j].y = fmaf(wv[k].y, x, acc[j].y);
        acc[j].z = fmaf(wv[k].z, x, acc[j].z);
        acc[j].w = fmaf(wv[k].w, x, acc[j].w);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < kPfBatch; ++j) *reinterpret_cast<float4*>(&red[part][j][f4]) = acc[j];
  __syncthreads();
  for (int i = tid; i < nb * kPfFeat; i += 256) {
    const int j = i / kPfFeat, e = i % kPfFeat;
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < kPfParts; ++k) sum += red[k][j][e];
    if (fc * kPfFeat + e < d_c)
      reinterpret_cast<float*>(qprep + static_cast<size_t>(b0 + j) * qstride)[static_cast<size_t>(h) * d_c +
                                                                              fc * kPfFeat + e] = sum;
  }
  if (fc == 0) {
    for (int i = tid; i < nb * d_rope; i += 256) {
      const int j = i / d_rope, r = i % d_rope;
      reinterpret_cast<float*>(qprep + static_cast<size_t>(b0 + j) * qstride)[static_cast<size_t>(H) * d_c +
                                                                              static_cast<size_t>(h) * d_rope + r] =
          q[(static_cast<size_t>(b0 + j) * H + h) * qrow + d_nope + r];
    }
  }
}

// ------------------------------------------------------------------ merge of the split partials
// For head h and the sequences b0 .. b0 + nt - 1 of a block of T threads: the
// splits that covered sequence b are the CTAs c0..c1 of the page schedule, their
// partials sit in slots c + b, and with M = max_s m_s (log2 units)
//   o = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s,
// 0 for a sequence of length 0.
//  - weights: a warp takes a sequence, its lanes the slots: M, then 2^(m_s - M)
//    into shared memory, kCombineSlots at a time, and the denominator;
//  - sums: thread t takes (sequence, 4 features) pairs t, t + T, .. (PPT of them
//    at most), with several slots of each in flight; where the block has fewer
//    pairs than threads, the slots are dealt to groups of threads whose sums are
//    added in group order.  The time is then a few round trips to L2 whatever
//    the number of slots.
// emit(j, f, o) is called for features f .. f + 3 of sequence b0 + j, by one
// thread; the caller's next __syncthreads makes what it stored visible.
constexpr int kCombineSlots = 128;
constexpr int kMergeMaxSeq = 16;         // sequences per block, at most

template <int T>
struct MergeShared {
  float wts[kMergeMaxSeq][kCombineSlots];
  float inv_l[kMergeMaxSeq];
  int slots[kMergeMaxSeq], slot0[kMergeMaxSeq];
  float4 red[T];
};

// the fewest sequences per block (a power of two up to `most`) that leave at most
// one block per SM
int merge_group(int H, int batch, int most) {
  int nt = 1;
  while (nt < most && H * ((batch + nt - 1) / nt) > kSms) nt *= 2;
  return nt;
}

template <int PPT, int T, int TS, typename Emit>
__device__ void merge_partials(MergeShared<TS>& sh, const int32_t* cu, const float* part_ml, const float* part_o,
                               int batch, int H, int h, int b0, int nt, int d_c, int num_splits, Emit emit) {
  static_assert(T <= TS, "threads");
  constexpr int kFlight = PPT >= 4 ? 4 : 8;   // slots of a pair in flight
  constexpr int kWarps = T / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nb = min(nt, batch - b0), ncol = d_c / 4, pairs = nt * ncol;
  const int chunk = split_chunk(cu[batch], num_splits);
  const size_t mlstride = static_cast<size_t>(H) * 2, sstride = static_cast<size_t>(H) * d_c;
  // the slots of this warp's sequences (warp, warp + kWarps) and their maxima
  int n[2] = {0, 0};
  float M[2] = {-INFINITY, -INFINITY}, lsum[2] = {0.f, 0.f};
  const float* pml[2] = {part_ml, part_ml};
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int j = warp + kWarps * e;
    if (j >= nb) continue;
    const int b = b0 + j, p0 = cu[b] + kSegCost, p1 = cu[b + 1], c0 = p0 / chunk;   // units of the sequence's pages
    n[e] = p1 > p0 ? (p1 - 1) / chunk - c0 + 1 : 0;
    pml[e] += (static_cast<size_t>(c0 + b) * H + h) * 2;
    if (lane == 0) {
      sh.slots[j] = n[e];
      sh.slot0[j] = c0 + b;
    }
    for (int k = lane; k < n[e]; k += 32) M[e] = fmaxf(M[e], pml[e][k * mlstride]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M[e] = fmaxf(M[e], __shfl_xor_sync(0xffffffffu, M[e], o));
  }
  // this thread's pairs, and its group where the slots are dealt out
  const int groups = pairs < T ? T / pairs : 1;
  const int grp = groups > 1 ? tid / pairs : 0;
  int pj[PPT], pf[PPT];
  const float* po[PPT];
  float4 acc[PPT];
  __syncthreads();
  int nmax = 0;
  for (int j = 0; j < nb; ++j) nmax = max(nmax, sh.slots[j]);
#pragma unroll
  for (int u = 0; u < PPT; ++u) {
    const int i = groups > 1 ? tid - grp * pairs : tid + u * T;
    const int j = i / ncol;
    const bool live = grp < groups && j < nb && (groups == 1 || u == 0);
    pj[u] = live ? j : -1;
    pf[u] = 4 * (i - j * ncol);
    acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    po[u] = part_o + (static_cast<size_t>(live ? sh.slot0[j] : 0) * H + h) * d_c + pf[u];
  }
  for (int k0 = 0; k0 < nmax; k0 += kCombineSlots) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int j = warp + kWarps * e;
      if (j >= nb) continue;
      for (int k = lane; k < kCombineSlots; k += 32) {
        float wk = 0.f;
        if (k0 + k < n[e]) {
          const float2 ml = *reinterpret_cast<const float2*>(pml[e] + (k0 + k) * mlstride);
          wk = exp2f(ml.x - M[e]);
          lsum[e] = fmaf(wk, ml.y, lsum[e]);
        }
        sh.wts[j][k] = wk;
      }
    }
    __syncthreads();
    const int kn = min(kCombineSlots, nmax - k0);
    for (int k = grp; k < kn; k += groups * kFlight) {
      float4 v[PPT][kFlight];
#pragma unroll
      for (int u = 0; u < PPT; ++u)
#pragma unroll
        for (int e = 0; e < kFlight; ++e) {
          const int kk = k + e * groups;
          v[u][e] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (pj[u] >= 0 && kk < kn && k0 + kk < sh.slots[pj[u]])
            v[u][e] = *reinterpret_cast<const float4*>(po[u] + (k0 + kk) * sstride);
        }
#pragma unroll
      for (int u = 0; u < PPT; ++u)
#pragma unroll
        for (int e = 0; e < kFlight; ++e) {
          const int kk = k + e * groups;
          const float w = pj[u] >= 0 && kk < kn ? sh.wts[pj[u]][kk] : 0.f;   // 0 past the sequence's slots
          acc[u].x = fmaf(w, v[u][e].x, acc[u].x);
          acc[u].y = fmaf(w, v[u][e].y, acc[u].y);
          acc[u].z = fmaf(w, v[u][e].z, acc[u].z);
          acc[u].w = fmaf(w, v[u][e].w, acc[u].w);
        }
    }
    __syncthreads();   // the weights are read: the next slots' may overwrite them
  }
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int j = warp + kWarps * e;
    if (j >= nb) continue;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lsum[e] += __shfl_xor_sync(0xffffffffu, lsum[e], o);
    if (lane == 0) sh.inv_l[j] = n[e] > 0 ? 1.f / lsum[e] : 0.f;
  }
  if (groups > 1) sh.red[tid] = acc[0];
  __syncthreads();
#pragma unroll
  for (int u = 0; u < PPT; ++u) {
    if (pj[u] < 0 || grp > 0) continue;
    float4 a = acc[u];
    for (int g = 1; g < groups; ++g) {
      const float4 r = sh.red[tid + g * pairs];
      a = make_float4(a.x + r.x, a.y + r.y, a.z + r.z, a.w + r.w);
    }
    const float il = sh.inv_l[pj[u]];
    emit(pj[u], pf[u], make_float4(a.x * il, a.y * il, a.z * il, a.w * il));
  }
}

// ------------------------------------------------------------------ combine, fp32
// Block per (head h, `nt` sequences; blockIdx.y: a part of the d_v output rows,
// each part repeating the merge), 256 threads: the merge, then u = W_UV,h o: warp
// w takes groups of four W_UV,h rows; a lane loads its 16-byte pieces of the four
// rows once and multiplies them into all the group's merged vectors (shared
// memory), then the 32 sums (sequence, row) are reduced across the lanes by a
// transposing butterfly (31 shuffles), after which lane t holds sequence t / 4,
// row t % 4.  8 sequences of 100 to 3000 tokens (up to 47 slots each) took 60 us
// with a warp per sequence, one slot after another; 10 us now (ncu, cold
// caches).
constexpr int kCombineThreads = 256;
constexpr int kCombineGroup = 8;        // sequences per block, at most
constexpr int kCombineMaxDc = 512;
constexpr int kCombineBlocks = 2 * kSms;

template <int PPT>
__global__ void __launch_bounds__(kCombineThreads)
combine_kernel(const int32_t* __restrict__ cu, const float* __restrict__ part_ml, const float* __restrict__ part_o,
               const float* __restrict__ w_uv, float* __restrict__ out, int batch, int H, int d_c, int d_v,
               int num_splits, int nt) {
  __shared__ __align__(16) float olat[kCombineGroup][kCombineMaxDc];
  __shared__ __align__(16) MergeShared<kCombineThreads> sh;
  const int h = blockIdx.x % H, b0 = (blockIdx.x / H) * nt;
  const int nb = min(nt, batch - b0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kCombineThreads / 32;
  const float* wh = w_uv + static_cast<size_t>(h) * d_v * d_c;
  // this block's rows of W_UV,h (groups of 4 kWarps, one in gridDim.y) on their way to L2 meanwhile
  for (int v = 4 * kWarps * blockIdx.y; v < d_v; v += 4 * kWarps * gridDim.y)
    for (int i = 32 * tid; i < min(4 * kWarps, d_v - v) * d_c; i += 32 * kCombineThreads)
      prefetch_l2(wh + static_cast<size_t>(v) * d_c + i);
  grid_dependency_wait();
  merge_partials<PPT, kCombineThreads>(sh, cu, part_ml, part_o, batch, H, h, b0, nt, d_c, num_splits,
                                       [&](int j, int f, const float4& o) { *reinterpret_cast<float4*>(&olat[j][f]) = o; });
  __syncthreads();
  // u[j][v] = sum_f W_UV[h][v][f] olat[j][f]
  constexpr int VEC = 4;
  const int npieces = d_c / VEC;   // d_c is a multiple of 4
  for (int v0 = 4 * (warp + kWarps * blockIdx.y); v0 < d_v; v0 += 4 * kWarps * gridDim.y) {
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.f;
    for (int pc = lane; pc < npieces; pc += 32) {
      float wf[4][VEC];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float4 raw = make_float4(0.f, 0.f, 0.f, 0.f);
        if (v0 + r < d_v) raw = *reinterpret_cast<const float4*>(wh + static_cast<size_t>(v0 + r) * d_c + pc * VEC);
        wf[r][0] = raw.x;
        wf[r][1] = raw.y;
        wf[r][2] = raw.z;
        wf[r][3] = raw.w;
      }
#pragma unroll
      for (int j = 0; j < kCombineGroup; ++j) {
        if (j < nb) {
          float o[VEC];
#pragma unroll
          for (int i = 0; i < VEC; i += 4) {
            const float4 q = *reinterpret_cast<const float4*>(&olat[j][pc * VEC + i]);
            o[i] = q.x;
            o[i + 1] = q.y;
            o[i + 2] = q.z;
            o[i + 3] = q.w;
          }
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int i = 0; i < VEC; ++i) acc[4 * j + r] = fmaf(wf[r][i], o[i], acc[4 * j + r]);
        }
      }
    }
    const float sum = reduce32_transpose(acc, lane);
    const int j = lane >> 2, v = v0 + (lane & 3);
    if (j < nb && v < d_v) out[(static_cast<size_t>(b0 + j) * H + h) * d_v + v] = sum;
  }
}

// ------------------------------------------------------------------ combine, bf16
// The merge and W_UV of the tensor-core path, for the launches whose decode
// kernel does not fuse them.  A block takes (head h, `nt` sequences, 128 output
// rows):
//  - W_UV,h's rows (the MMA's M = 128 operand, K = d_c) are copied by TMA before
//    the block waits for the decode kernel (which lets it start only when all that
//    comes before that kernel is complete);
//  - merge as in combine_kernel: weights per (sequence, slot) in shared memory,
//    then thread t takes (sequence, 4 features) pairs; where the block has fewer
//    pairs than threads, the slots are dealt to groups of threads whose sums
//    are added in group order;
//  - the merged fp32 vector is split into three bf16 pieces, its significand's
//    three bytes (o = o1 + o2 + o3 exactly; an infinite or NaN o is its first
//    piece), which become three columns of the N operand, so that
//    u = W_UV,h o1 + W_UV,h o2 + W_UV,h o3 keeps the fp32 value of o (the weights
//    are bf16 as stored), accumulated in fp32;
//  - u: lanes are output rows; a sequence's three columns are added, rounded to
//    bf16 and stored.
// Bound by the merge's reads of the partials from L2 and the latency of its
// phases: 7 us at 128 sequences with d_c 192 (the merge at the end of the
// decode kernel, on CUDA cores after a grid-wide wait, and the cooperative
// launch it needs cost that step 8 us more), and 8 us against 18 on CUDA cores
// with d_c 512 (kernel alone, warm).
constexpr int kCtMaxThreads = 512;
constexpr uint32_t kCtAtom = 128 * 128;  // 128 rows x 64 bf16

// the N operand's rows: three per sequence, a multiple of the MMA's 16
__host__ __device__ constexpr int ct_cols(int nt) { return (3 * nt + 15) / 16 * 16; }

struct CtShared {
  MergeShared<kCtMaxThreads> merge;
  uint64_t afull, done;
  uint32_t tmem_base;
  int abort;
};
__host__ __device__ constexpr uint32_t ct_smem(int d_c, int nt) {
  return static_cast<uint32_t>(d_c / 64) * (kCtAtom + ct_cols(nt) * 128) + sizeof(CtShared) + 1024;
}

static_assert(ct_smem(kCombineMaxDc, kMergeMaxSeq) <= kSmemMost, "shared memory");

// PPT: (sequence, 4 features) pairs per thread, at most; T threads (512 where
// that is more than one pair each: more of the partials in flight, 128 ragged
// sequences 69.3 -> 67.7 us, 128 at d_c 512 123.6 -> 118.9; 256 otherwise, 32 x 4K
// 37.5 against 38.1)
template <int PPT, int kCtThreads>
__global__ void __launch_bounds__(kCtThreads)
combine_tc_kernel(const __grid_constant__ CUtensorMap wmap, const int32_t* __restrict__ cu,
                  const float* __restrict__ part_ml, const float* __restrict__ part_o, __nv_bfloat16* __restrict__ out,
                  int batch, int d_c, int d_v, int num_splits, int nt, int early, uint64_t wait_ns, int32_t* status) {
  constexpr int H = 16;
  extern __shared__ uint8_t ct_raw[];
  uint8_t* smem = ct_raw + ((1024u - (smem_u32(ct_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  const int nkc = d_c / 64, cols = ct_cols(nt);
  const uint32_t o_off = static_cast<uint32_t>(nkc) * kCtAtom, o_chunk = static_cast<uint32_t>(cols) * 128;
  CtShared& sh = *reinterpret_cast<CtShared*>(smem + o_off + nkc * o_chunk);
  volatile int* abort_flag = &sh.abort;
  const int h = blockIdx.x % H, b0 = (blockIdx.x / H) * nt, v0 = blockIdx.y * 128;
  const int nb = min(nt, batch - b0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    mbar_init(smem_u32(&sh.afull), 1);
    mbar_init(smem_u32(&sh.done), 1);
    sh.abort = 0;
    fence_mbar_init();
    prefetch_tensormap(&wmap);
    const uint64_t keep = policy_evict_last();
    mbar_arrive_expect_tx(smem_u32(&sh.afull), static_cast<uint32_t>(nkc) * kCtAtom);
    for (int kc = 0; kc < nkc; ++kc) tma_load_3d(sbase + kc * kCtAtom, &wmap, 64 * kc, v0, h, smem_u32(&sh.afull), keep);
  }
  if (early) grid_launch_dependents();   // the layer's output projection, which streams weights of its own
  const uint32_t tmem_cols = cols <= 32 ? 32u : 64u;
  if (warp == 1) {
    tmem_alloc(smem_u32(&sh.tmem_base), tmem_cols);
    tmem_relinquish();
  }
  grid_dependency_wait();
  // the merged vectors as three bf16 pieces, rows j, nt + j and 2 nt + j of the N
  // operand (K-major, 128-byte swizzle)
  merge_partials<PPT, kCtThreads>(sh.merge, cu, part_ml, part_o, batch, H, h, b0, nt, d_c, num_splits,
                                  [&](int j, int f, const float4& o) {
    float x[4] = {o.x, o.y, o.z, o.w};
    const int kc = f / 64, unit = (f % 64) / 8;
#pragma unroll
    for (int piece = 0; piece < 3; ++piece) {
      const int row = piece * nt + j;
      uint32_t w[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint32_t lo = __float_as_uint(x[2 * e]), hi = __float_as_uint(x[2 * e + 1]);
        w[e] = __byte_perm(lo, hi, 0x7632);   // the upper halves
#pragma unroll
        for (int k = 2 * e; k < 2 * e + 2; ++k) {
          const float rest = x[k] - __uint_as_float(__float_as_uint(x[k]) & 0xffff0000u);
          x[k] = fabsf(x[k]) < INFINITY ? rest : 0.f;
        }
      }
      *reinterpret_cast<uint2*>(smem + o_off + kc * o_chunk + row * 128 + ((unit ^ (row & 7)) << 4) + (f & 4) * 2) =
          make_uint2(w[0], w[1]);
    }
  });
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;
  if (tid == 0) {
    volatile int own = 0;   // the copies land before the block can leave
    if (!mbar_wait(smem_u32(&sh.afull), 0, &own, wait_ns)) {
      *abort_flag = 1;
    } else {
      tc_fence_after();
      const uint32_t idesc = idesc_bf16(128, cols, 0, 0);
      for (int kc = 0; kc < nkc; ++kc) {
        const uint64_t ad = smem_desc(sbase + kc * kCtAtom, 16, 1024, kSwizzle128B);
        const uint64_t bd = smem_desc(sbase + o_off + kc * o_chunk, 16, 1024, kSwizzle128B);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_bf16_ss(tmem, ad + ((kk * 32) >> 4), bd + ((kk * 32) >> 4), idesc, (kc > 0 || kk > 0) ? 1u : 0u);
      }
    }
    mma_commit(smem_u32(&sh.done));
  }
  __syncwarp();
  bool ok = mbar_wait(smem_u32(&sh.done), 0, abort_flag, wait_ns);
  ok = __all_sync(0xffffffffu, ok) && *abort_flag == 0;
  tc_fence_after();
  // ---- u: warp (of the first eight) = (lane quadrant, every other sequence)
  if (ok && warp < 8) {
    float d[48];
    const uint32_t ta = tmem + (static_cast<uint32_t>(32 * (warp & 3)) << 16);
#pragma unroll
    for (int c = 0; c < 48; c += 16)
      if (c < cols) tmem_ld16(ta + c, *reinterpret_cast<float(*)[16]>(&d[c]));
    tmem_wait_ld();
    const int v = v0 + 32 * (warp & 3) + lane;
    // (nt is a power of two: the columns of a sequence by a compile-time switch)
    auto store = [&](auto nt_c) {
      constexpr int NT = decltype(nt_c)::value;
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        // (an infinite first column, of an infinite o or weight, is the sum: the
        // other pieces may be zero, and their product with such a weight no number)
        const float u = fabsf(d[j]) < INFINITY ? d[j] + (d[NT + j] + d[2 * NT + j]) : d[j];
        if ((NT == 1 ? warp < 4 : (j & 1) == warp >> 2) && j < nb && v < d_v)
          out[(static_cast<size_t>(b0 + j) * H + h) * d_v + v] = __float2bfloat16_rn(u);
      }
    };
    if (nt == 1) store(std::integral_constant<int, 1>{});
    else if (nt == 2) store(std::integral_constant<int, 2>{});
    else if (nt == 4) store(std::integral_constant<int, 4>{});
    else if (nt == 8) store(std::integral_constant<int, 8>{});
    else store(std::integral_constant<int, 16>{});
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, tmem_cols);
  if (tid == 0 && *abort_flag) report_status(status, kStatusTimeout);
}

// p[f .. f + 3] (`none` without p), one load where p allows it
__device__ __forceinline__ float4 load_features4(const float* p, int f, float none) {
  if (p == nullptr) return make_float4(none, none, none, none);
  if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) return __ldg(reinterpret_cast<const float4*>(p + f));
  return make_float4(__ldg(p + f), __ldg(p + f + 1), __ldg(p + f + 2), __ldg(p + f + 3));
}

// ------------------------------------------------------------------ fp32 decode
// One block of 16 warps per split, one 64-token page per tile:
//   gate    warp w takes tokens w, w + 16, ..: c~ = LN(c (*) G[id]) (two-pass mean
//           and variance) into shared memory with the RoPE key behind it, the
//           loads of several tokens issued together;
//   scores  warp = (8 heads, one of 8 parts of d_c + d_rope), lane = tokens
//           lane and lane + 32: each shared-memory value read meets 8 heads or
//           2 tokens;
//   softmax warp = head: the parts added, the tile's maximum, P and the
//           running max and denominator;
//   output  thread = (4 features, 4 heads, every n-th token), accumulated in
//           registers, the token groups added at the segment's end.
// All sums are fp32 on CUDA cores.  A tile's four phases cost five block
// barriers for 64 tokens; processing one token at a time cost 36 barriers per
// token, 651 us for 8 sequences of 100 to 3000 tokens (d_c 256, 16 heads)
// against 17 us now (ncu, cold caches).  At that size a split holds one
// page, so the time is the latency of one tile's phases: the sequence found by
// one round of loads, the page requested before the query block, the tokens of
// the output dealt to groups of threads where d_c leaves threads without work,
// W_UK requested before q is staged and W_UV brought to L2 before the combine
// waits took the step from 28.4 to 26.4 us, gamma and beta in 16-byte loads to
// 25.8.
constexpr int kF32Threads = 512, kF32Warps = kF32Threads / 32;
constexpr int kF32Parts = 8;      // parts of a dot product
constexpr int kF32Heads = 16;     // heads, at most
constexpr int kF32MaxRope = 64;   // d_rope, at most

// row stride of the tile in floats: a multiple of 4 and an odd number of 16-byte
// units, so that the lanes' rows start in different bank groups
__host__ __device__ constexpr int f32_row(int d) { return (d / 4) % 2 ? d : d + 4; }
__host__ __device__ constexpr size_t f32_smem_floats(int d_c, int d_rope) {
  const int d = d_c + d_rope;
  return static_cast<size_t>(kF32Heads) * d + static_cast<size_t>(kPage) * f32_row(d) +
         kF32Parts * kF32Heads * kPage + kPage * kF32Heads + kF32Heads;
}

static_assert(f32_smem_floats(512, kF32MaxRope) * sizeof(float) <= kSmemMost, "shared memory");

// NV: 16-byte units of a latent row per lane (d_c <= 128 NV)
template <int NV>
__global__ void __launch_bounds__(kF32Threads, 1)
decode_f32_kernel(const float* __restrict__ c_pool, const float* __restrict__ kr_pool,
                  const int32_t* __restrict__ id_pool, const int32_t* __restrict__ block_table,
                  int max_pages, const int32_t* __restrict__ seq_lens, int batch, int num_pages,
                  const float* __restrict__ gate_table, const float* __restrict__ gamma,
                  const float* __restrict__ beta, const uint8_t* __restrict__ qprep, size_t qstride,
                  const int32_t* __restrict__ cu, float* __restrict__ part_ml, float* __restrict__ part_o,
                  int H, int d_c, int d_rope, int vocab, int gate, int gate_add, int gate_ln, float scale_log2,
                  float eps,
                  int32_t* status) {
  constexpr int kTok = kPage / kF32Warps;            // tokens of a page per warp
  constexpr int kBatch = NV <= 2 ? kTok : kTok / 2;  // .. whose rows are in flight together
  const int d = d_c + d_rope, row_f = f32_row(d), ncol = d_c / 4;
  extern __shared__ __align__(16) float sm[];
  float* qs = sm;                                    // [16][d]: q^_h, then q^R_h (0 past H)
  float* ct = qs + kF32Heads * d;                    // [64][row_f]: c~, then k^R
  float* sp = ct + kPage * row_f;                    // [8 parts][16 heads][64 tokens]
  float* pw = sp + kF32Parts * kF32Heads * kPage;    // [64 tokens][16 heads]
  float* al = pw + kPage * kF32Heads;                // [16]

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the combine may start (with this trigger / without: 64 short sequences 38.4 / 38.9
  // us, but 8 of 100 to 3000 tokens 25.2 / 24.2 and one of 3000 22.6 / 21.8); before
  // its wait it only brings W_UV to L2
  grid_launch_dependents();
  grid_dependency_wait();
  const int total = cu[batch];
  const int chunk = split_chunk(total, gridDim.x);
  const int g0 = blockIdx.x * chunk;
  const int g1 = min(g0 + chunk, total);
  if (g0 >= g1) return;
  // the sequence of unit g0: the last that starts at or before it, by one round of loads
  int b = batch <= kF32Threads ? __syncthreads_count(tid < batch && cu[min(tid, batch)] <= g0) - 1
                               : find_sequence(cu, batch, g0);
  int g = g0;
  // output: features 4 ocol .., heads 4 ohg .., every og-th token of ogroups
  const int ocols = ncol * (kF32Heads / 4), ogroups = min(kF32Threads / ocols, 8);
  const int ocol = tid % ncol, ohg = tid % ocols / ncol, og = tid / ocols;
  const bool oact = og < ogroups && 4 * ohg < H;
  // a page past the block table's row is out of range like any other bad id
  auto page_of = [&](int lp) { return lp < max_pages ? block_table[static_cast<size_t>(b) * max_pages + lp] : -1; };
  while (g < g1) {
    const int pend = min(g1, cu[b + 1]);
    const int L = seq_lens[b];
    const int s0 = cu[b] + kSegCost;   // unit of the sequence's first page
    const int lp0 = max(g - s0, 0), lp1 = pend - s0;
    if (min(lp1 * kPage, L) <= lp0 * kPage) break;   // the range ends inside the sequence's start cost
    int page = page_of(lp0);   // (requested before the query block)
    {
      // warp = head
      const float* qsrc = reinterpret_cast<const float*>(qprep + static_cast<size_t>(b) * qstride);
      float4 qv[NV], qr = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int u = lane + 32 * i;
        qv[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (warp < H && u < ncol) qv[i] = reinterpret_cast<const float4*>(qsrc + static_cast<size_t>(warp) * d_c)[u];
      }
      if (warp < H && lane < d_rope / 4)
        qr = reinterpret_cast<const float4*>(qsrc + static_cast<size_t>(H) * d_c + warp * d_rope)[lane];
      float* qd = qs + warp * d;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int u = lane + 32 * i;
        if (u < ncol) *reinterpret_cast<float4*>(qd + 4 * u) = qv[i];
      }
      if (lane < d_rope / 4) *reinterpret_cast<float4*>(qd + d_c + 4 * lane) = qr;
    }
    float4 acc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    float mrun = -INFINITY, lrun = 0.f;   // head `warp`, the same in every lane
    for (int lp = lp0; lp < lp1; ++lp) {
      const int ntok = min(kPage, L - lp * kPage);
      if (lp > lp0) page = page_of(lp);
      const bool page_ok = page >= 0 && page < num_pages;
      if (!page_ok && tid == 0) report_status(status, kStatusOutOfRange);
      const size_t row0 = static_cast<size_t>(page_ok ? page : 0) * kPage;
      // ---- gate and LayerNorm
#pragma unroll
      for (int k0 = 0; k0 < kTok; k0 += kBatch) {
        float4 z[kBatch][NV], gv[kBatch][NV], kr[kBatch];
        int id[kBatch];
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
          const int t = warp + kF32Warps * (k0 + k);
          id[k] = gate && t < ntok ? id_pool[row0 + t] : 0;
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
          const int t = warp + kF32Warps * (k0 + k);
          if (id[k] < 0 || id[k] >= vocab) {
            if (lane == 0) report_status(status, kStatusOutOfRange);
            id[k] = 0;
          }
#pragma unroll
          for (int i = 0; i < NV; ++i) {
            const int u = lane + 32 * i;
            z[k][i] = make_float4(0.f, 0.f, 0.f, 0.f);
            gv[k][i] = z[k][i];
            if (t < ntok && u < ncol) {
              z[k][i] = __ldg(reinterpret_cast<const float4*>(c_pool + (row0 + t) * d_c) + u);
              if (gate) gv[k][i] = __ldg(reinterpret_cast<const float4*>(gate_table + static_cast<size_t>(id[k]) * d_c) + u);
            }
          }
          kr[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (t < ntok && lane < d_rope / 4)
            kr[k] = __ldg(reinterpret_cast<const float4*>(kr_pool + (row0 + t) * d_rope) + lane);
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
          const int t = warp + kF32Warps * (k0 + k);
          float* row = ct + t * row_f;
          if (gate) {
            float s1 = 0.f;
#pragma unroll
            for (int i = 0; i < NV; ++i) {
              float4& v = z[k][i];
              const float4 w = gv[k][i];
              v = gate_add ? make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w)
                           : make_float4(v.x * w.x, v.y * w.y, v.z * w.z, v.w * w.w);
              s1 += (v.x + v.y) + (v.z + v.w);
            }
            if (gate_ln) {
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) s1 += __shfl_xor_sync(0xffffffffu, s1, o);
              const float mean = s1 / d_c;
              float s2 = 0.f;
#pragma unroll
              for (int i = 0; i < NV; ++i) {
                float4& v = z[k][i];
                if (lane + 32 * i < ncol) {
                  v = make_float4(v.x - mean, v.y - mean, v.z - mean, v.w - mean);
                  s2 = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, s2))));
                }
              }
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
              const float rstd = rsqrtf(s2 / d_c + eps);
#pragma unroll
              for (int i = 0; i < NV; ++i) {
                const int f = 4 * (lane + 32 * i);
                if (f < d_c) {
                  float4& v = z[k][i];
                  const float4 gm = load_features4(gamma, f, 1.f), bt = load_features4(beta, f, 0.f);
                  v.x = v.x * rstd * gm.x + bt.x;
                  v.y = v.y * rstd * gm.y + bt.y;
                  v.z = v.z * rstd * gm.z + bt.z;
                  v.w = v.w * rstd * gm.w + bt.w;
                }
              }
            }
          }
#pragma unroll
          for (int i = 0; i < NV; ++i) {
            const int u = lane + 32 * i;
            if (u < ncol) *reinterpret_cast<float4*>(row + 4 * u) = z[k][i];
          }
          if (lane < d_rope / 4) *reinterpret_cast<float4*>(row + d_c + 4 * lane) = kr[k];
        }
      }
      __syncthreads();
      // ---- scores
      {
        const int h0 = 8 * (warp / kF32Parts), part = warp % kF32Parts;
        const int u0 = d / 4 * part / kF32Parts, u1 = d / 4 * (part + 1) / kF32Parts;
        float sa[2][8];
#pragma unroll
        for (int j = 0; j < 8; ++j) sa[0][j] = sa[1][j] = 0.f;
        if (h0 < H) {
          const float *r0 = ct + lane * row_f, *r1 = ct + (lane + 32) * row_f, *qh = qs + h0 * d;
          for (int u = u0; u < u1; ++u) {
            const float4 x0 = *reinterpret_cast<const float4*>(r0 + 4 * u);
            const float4 x1 = *reinterpret_cast<const float4*>(r1 + 4 * u);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float4 y = *reinterpret_cast<const float4*>(qh + j * d + 4 * u);
              sa[0][j] = fmaf(y.x, x0.x, fmaf(y.y, x0.y, fmaf(y.z, x0.z, fmaf(y.w, x0.w, sa[0][j]))));
              sa[1][j] = fmaf(y.x, x1.x, fmaf(y.y, x1.y, fmaf(y.z, x1.z, fmaf(y.w, x1.w, sa[1][j]))));
            }
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            sp[(part * kF32Heads + h0 + j) * kPage + lane] = sa[0][j];
            sp[(part * kF32Heads + h0 + j) * kPage + lane + 32] = sa[1][j];
          }
        }
      }
      __syncthreads();
      // ---- softmax of head `warp`
      if (warp < H) {
        float s[2], mx = mrun;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int t = lane + 32 * e;
          float v = 0.f;
#pragma unroll
          for (int k = 0; k < kF32Parts; ++k) v += sp[(k * kF32Heads + warp) * kPage + t];
          s[e] = t < ntok ? v * scale_log2 : -INFINITY;
          mx = fmaxf(mx, s[e]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        float ps = 0.f;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float pv = lane + 32 * e < ntok ? exp2f(s[e] - mx) : 0.f;
          pw[(lane + 32 * e) * kF32Heads + warp] = pv;
          ps += pv;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, o);
        const float a = exp2f(mrun - mx);
        lrun = lrun * a + ps;
        mrun = mx;
        if (lane == 0) al[warp] = a;
      } else {
        pw[lane * kF32Heads + warp] = 0.f;
        pw[(lane + 32) * kF32Heads + warp] = 0.f;
        if (lane == 0) al[warp] = 1.f;
      }
      __syncthreads();
      // ---- output
      if (oact) {
        const float4 a4 = *reinterpret_cast<const float4*>(al + 4 * ohg);
        const float a[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          acc[k].x *= a[k];
          acc[k].y *= a[k];
          acc[k].z *= a[k];
          acc[k].w *= a[k];
        }
        const float* zc = ct + 4 * ocol;
        const float* pc = pw + 4 * ohg;
#pragma unroll 4
        for (int t = og; t < ntok; t += ogroups) {
          const float4 x = *reinterpret_cast<const float4*>(zc + t * row_f);
          const float4 p4 = *reinterpret_cast<const float4*>(pc + t * kF32Heads);
          const float pk[4] = {p4.x, p4.y, p4.z, p4.w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            acc[k].x = fmaf(pk[k], x.x, acc[k].x);
            acc[k].y = fmaf(pk[k], x.y, acc[k].y);
            acc[k].z = fmaf(pk[k], x.z, acc[k].z);
            acc[k].w = fmaf(pk[k], x.w, acc[k].w);
          }
        }
      }
      __syncthreads();   // the tile is read: the next one may overwrite it
    }
    const size_t slot = blockIdx.x + b;
    if (ogroups > 1) {   // the token groups' sums, added in order (the scores' space is free)
      float4* red = reinterpret_cast<float4*>(sp);
#pragma unroll
      for (int k = 0; k < 4; ++k) red[k * kF32Threads + tid] = acc[k];
      __syncthreads();
      if (og == 0) {
        for (int i = 1; i < ogroups; ++i)
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float4 r = red[k * kF32Threads + tid + i * ocols];
            acc[k] = make_float4(acc[k].x + r.x, acc[k].y + r.y, acc[k].z + r.z, acc[k].w + r.w);
          }
      }
    }
    if (oact && og == 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * ohg + k < H)
          *reinterpret_cast<float4*>(part_o + (slot * H + 4 * ohg + k) * d_c + 4 * ocol) = acc[k];
    }
    if (warp < H && lane == 0) {
      part_ml[(slot * H + warp) * 2] = mrun;
      part_ml[(slot * H + warp) * 2 + 1] = lrun;
    }
    g = pend;
    ++b;
    while (b < batch && cu[b + 1] <= g) ++b;
  }
}

// ------------------------------------------------------------------ launchers
cudaError_t launch_append(const AppendArgs& a, cudaStream_t st) {
  if (a.batch == 0) return cudaSuccess;
  append_latent_kernel<<<a.batch, 64, 0, st>>>(a);
  return cudaGetLastError();
}

// The fewest sequences per block (a multiple of the MMA's 16) that leave at
// most one block per SM, so that the blocks' epilogues are short.
int absorb_tile(int d_c, int batch) {
  const int mt = (d_c + kPmTile - 1) / kPmTile;
  int nt = 16;
  while (nt < kPmMaxSeq && 16 * mt * ((batch + nt - 1) / nt) > kSms) nt *= 2;
  return nt;
}

cudaError_t launch_prologue_tc(const DecodeArgs& a, const AppendArgs* app, const CUtensorMap* maps, cudaStream_t st) {
  const WorkspaceLayout wl = workspace_layout(a.batch, a.num_splits, 16, a.d_c, a.d_rope, true);
  uint8_t* ws = static_cast<uint8_t*>(a.workspace);
  // with the gate off the latent is used as cached: no LayerNorm affine to fold into q^
  const float* gamma = a.gate && a.gate_ln ? a.ln_gamma : nullptr;
  const float* beta = a.gate && a.gate_ln ? a.ln_beta : nullptr;
  AppendArgs none;
  std::memset(&none, 0, sizeof(none));
  const AppendArgs& ap = app != nullptr ? *app : none;
  const int nt = absorb_tile(a.d_c, a.batch), mt = (a.d_c + kPmTile - 1) / kPmTile, nk = (a.d_nope + 63) / 64;
  const int tiles = a.q != nullptr ? 16 * mt * ((a.batch + nt - 1) / nt) : 0;
  const int blocks = tiles + 1 + (ap.batch + kPmThreads / 32 - 1) / (kPmThreads / 32);
  const size_t smem = pm_smem(nk, nt);
  const cudaError_t e = allow_smem(prologue_tc_kernel, pm_smem(kPmMaxNope / 64, kPmMaxSeq));
  if (e != cudaSuccess) return e;
  return launch_chained(
      prologue_tc_kernel, dim3(blocks), dim3(kPmThreads), smem, st, maps[0], maps[1],
      static_cast<const __nv_bfloat16*>(a.q), gamma, beta, a.seq_lens, a.batch, a.d_nope, a.d_rope, a.d_c,
      a.page_size, ws + wl.off_qprep, wl.qprep_stride, reinterpret_cast<int32_t*>(ws + wl.off_cu),
      reinterpret_cast<uint32_t*>(ws + wl.off_done), a.num_splits, a.block_table, a.max_pages,
      reinterpret_cast<SplitStart*>(ws + wl.off_start), nt, kWaitLimitNs, a.status, ap);
}

namespace {
template <int NV>
cudaError_t launch_decode_f32_t(const DecodeArgs& a, const WorkspaceLayout& wl, cudaStream_t st) {
  uint8_t* ws = static_cast<uint8_t*>(a.workspace);
  const size_t smem = f32_smem_floats(a.d_c, a.d_rope) * sizeof(float);
  const cudaError_t e = allow_smem(decode_f32_kernel<NV>, f32_smem_floats(128 * NV, kF32MaxRope) * sizeof(float));
  if (e != cudaSuccess) return e;
  return launch_chained(
      decode_f32_kernel<NV>, dim3(a.num_splits), dim3(kF32Threads), smem, st,
      static_cast<const float*>(a.c_pool), static_cast<const float*>(a.kr_pool), a.id_pool, a.block_table,
      a.max_pages, a.seq_lens, a.batch, a.num_pages, static_cast<const float*>(a.gate_table), a.ln_gamma,
      a.ln_beta, ws + wl.off_qprep, wl.qprep_stride, reinterpret_cast<const int32_t*>(ws + wl.off_cu),
      reinterpret_cast<float*>(ws + wl.off_ml), reinterpret_cast<float*>(ws + wl.off_o), a.H, a.d_c, a.d_rope,
      a.vocab, a.gate, a.gate_add, a.gate_ln, a.scale_log2, a.eps, a.status);
}
}  // namespace

cudaError_t launch_decode_f32(const DecodeArgs& a, const AppendArgs* app, cudaStream_t st) {
  const WorkspaceLayout wl = workspace_layout(a.batch, a.num_splits, a.H, a.d_c, a.d_rope, false);
  uint8_t* ws = static_cast<uint8_t*>(a.workspace);
  AppendArgs none;
  std::memset(&none, 0, sizeof(none));
  const AppendArgs& ap = app != nullptr ? *app : none;
  const int absorb =
      a.H * ((a.d_c + kPfFeat - 1) / kPfFeat) * ((a.batch + kPfBatch - 1) / kPfBatch);
  const cudaError_t e = launch_chained(
      prologue_f32_kernel, dim3(absorb + 1 + ap.batch), dim3(256), 0, st,
      static_cast<const float*>(a.q), static_cast<const float*>(a.w_uk), a.seq_lens, a.batch, a.H, a.d_nope,
      a.d_rope, a.d_c, a.page_size, ws + wl.off_qprep, wl.qprep_stride,
      reinterpret_cast<int32_t*>(ws + wl.off_cu), ap);
  if (e != cudaSuccess) return e;
  if (a.d_c <= 128) return launch_decode_f32_t<1>(a, wl, st);
  if (a.d_c <= 256) return launch_decode_f32_t<2>(a, wl, st);
  return launch_decode_f32_t<4>(a, wl, st);
}

namespace {
template <int PPT, int T>
cudaError_t launch_combine_tc(const DecodeArgs& a, const CUtensorMap* wmap, const int32_t* cu, const float* ml,
                              const float* po, int nt, cudaStream_t st) {
  const size_t smem = ct_smem(a.d_c, nt);
  const cudaError_t e = allow_smem(combine_tc_kernel<PPT, T>, ct_smem(kCombineMaxDc, kMergeMaxSeq));
  if (e != cudaSuccess) return e;
  return launch_chained(combine_tc_kernel<PPT, T>, dim3(16 * ((a.batch + nt - 1) / nt), (a.d_v + 127) / 128),
                        dim3(T), smem, st, *wmap, cu, ml, po, static_cast<__nv_bfloat16*>(a.out), a.batch,
                        a.d_c, a.d_v, a.num_splits, nt, a.early, kWaitLimitNs, a.status);
}
}  // namespace

cudaError_t launch_combine(const DecodeArgs& a, bool tc_path, const CUtensorMap* wmap, cudaStream_t st) {
  const WorkspaceLayout wl = workspace_layout(a.batch, a.num_splits, a.H, a.d_c, a.d_rope, tc_path);
  uint8_t* ws = static_cast<uint8_t*>(a.workspace);
  const int32_t* cu = reinterpret_cast<const int32_t*>(ws + wl.off_cu);
  const float* ml = reinterpret_cast<const float*>(ws + wl.off_ml);
  const float* po = reinterpret_cast<const float*>(ws + wl.off_o);
  if (tc_path) {
    const int nt = merge_group(16, a.batch, kMergeMaxSeq);
    const int pairs = nt * (a.d_c / 4);
    if (pairs <= 256) return launch_combine_tc<1, 256>(a, wmap, cu, ml, po, nt, st);
    if (pairs <= 512) return launch_combine_tc<1, 512>(a, wmap, cu, ml, po, nt, st);
    if (pairs <= 1024) return launch_combine_tc<2, 512>(a, wmap, cu, ml, po, nt, st);
    return launch_combine_tc<4, 512>(a, wmap, cu, ml, po, nt, st);
  }
  // small batches: the output rows spread over more blocks (a pass of the block's
  // warps covers 32 rows), so that most SMs read a part of W_UV
  const int nt = merge_group(a.H, a.batch, kCombineGroup), pairs = nt * (a.d_c / 4);
  const int groups = a.H * ((a.batch + nt - 1) / nt), passes = (a.d_v + 31) / 32;
  int parts = kCombineBlocks / groups;
  parts = parts < 1 ? 1 : parts > passes ? passes : parts;
  auto launch = [&](auto kernel) {
    return launch_chained(kernel, dim3(groups, parts), dim3(kCombineThreads), 0, st, cu, ml, po,
                          static_cast<const float*>(a.w_uv), static_cast<float*>(a.out), a.batch, a.H, a.d_c, a.d_v,
                          a.num_splits, nt);
  };
  if (pairs <= kCombineThreads) return launch(combine_kernel<1>);
  if (pairs <= 2 * kCombineThreads) return launch(combine_kernel<2>);
  return launch(combine_kernel<4>);
}

}  // namespace egmla
