// egmla_r0.cu - decode with the paper-literal gate placement (R0): the gate
// and the LayerNorm act on the up-projected keys and values of all heads,
// kv~ = LN_{H(d_n + d_v)}((W^UKV c) (*) g) (Section 3 Eq. 5 applied after
// Eq. 2, as the Appendix E listing does), split per head into k^C, v^C
// (Eq. 6), then attention as in Eqs. 11-13 without absorption (the gate in
// the 4096-wide space cannot be folded into the query).
//
// The LayerNorm needs all 4096 features of a token before any head's key or
// value is final, but the scores do not need the normalised keys:
//   q . k~ = r (q gamma) . z_k - r mu sum(q gamma) + q . beta,
// so the up-projection computes every head's raw dot (q gamma) . z_k while
// it has z_k in registers and keeps only the gated values.  Two kernels:
//   r0_project_kernel  (tcgen05, CTA pairs) one tile of two cache pages (128
//                      tokens) per CTA of the walk over every sequence's
//                      pages; the two CTAs of a cluster share the MMAs (M = 256
//                      rows, both tiles): for each head h, D = C W^UKV_h^T (N =
//                      256 = d_n + d_v features, K = d_c) with each CTA holding
//                      half of W^UKV_h's rows, in one of two TMEM accumulators,
//                      so that the epilogue of head h overlaps the MMAs of head
//                      h + 1.  Epilogue: four groups of four warps, one row per
//                      lane (its R0 gate values G_R0[id] of head h + 1 requested
//                      a quarter at a time while head h is processed): the key
//                      groups gate their 64 features each, round z to bf16 and
//                      add (q gamma) . z to the row's head dots; the value
//                      groups gate and round their 64 features and store them
//                      head-major through a per-warp shared-memory tile (128
//                      contiguous bytes per row).  All add z and z^2 of the
//                      rounded values into the row's statistics.  After the last
//                      head: (mu, 1/sqrt(var + eps)) and every head's logit
//                        s = scale log2(e) (r ((q gamma) . z_k - mu sum(q gamma)) + q . beta + q^R . k^R).
//                      Bound by the epilogue's latency (a warp's chain per head:
//                      accumulator, gate values, conversions, statistics): eight
//                      warps took 133 us for 8 x 4096 tokens whether each CTA
//                      copied all of W^UKV or half of it, sixteen with packed
//                      fp32 pairs about 110 (256 tiles are two waves on 152 SMs).
//   r0_attend_kernel   one block per (sequence, head): an online softmax over
//                      the logits and, with P' = p r,
//                        o = gamma_v ((sum P' z_v - sum P' mu) / sum p) + beta_v,
//                      streaming 256 bytes of gated values per token.
// The gated values (H d_v bf16 per pool row, head-major) are identical for
// every sequence that holds a page, so a page shared by two sequences is
// written twice with the same bytes; the logits are per (sequence, position).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>

#include "egmla_common.cuh"
#include "egmla_kernels.h"
#include "egmla_ptx.cuh"

namespace egmla {
namespace {

constexpr int kR0Heads = 16;
constexpr int kR0Feat = 256;                    // d_n + d_v per head
constexpr int kR0Half = 128;                    // d_n = d_v
constexpr int kR0Rope = 64;
constexpr int kR0Width = kR0Heads * kR0Feat;    // 4096
constexpr int kR0Rows = 2 * kPage;              // tile rows: two pages (the MMA's M)
constexpr int kR0Chunk = 64;                    // K elements per operand chunk (128-byte swizzle atom)
constexpr uint32_t kR0AChunkBytes = kR0Rows * kR0Chunk * 2;   // 16 KB
constexpr uint32_t kR0APageBytes = kPage * kR0Chunk * 2;      // 8 KB: one page's rows of a chunk
// the CTAs of a pair hold half of a head's 256 rows of W^UKV each (rank 0 its key
// rows, rank 1 its value rows)
constexpr uint32_t kR0BChunkBytes = kR0Half * kR0Chunk * 2;   // 16 KB
constexpr int kR0BStages = 5;
// epilogue: four groups of four warps (one TMEM lane quadrant each): the first
// and last 64 key features, the first and last 64 value features of a head
constexpr int kR0Groups = 4;
constexpr int kR0GroupFeat = kR0Feat / kR0Groups;   // 64
constexpr int kR0EpiWarps = 4 * kR0Groups;
constexpr int kR0Threads = 32 * (2 + kR0EpiWarps);   // warp 0 TMA, warp 1 MMA, warps 2-17 epilogue
constexpr uint32_t kR0TmemCols = 512;           // two 256-column accumulators
constexpr int kR0S1Stride = kR0Heads + 1;       // row stride of the head dots (no bank conflicts)
constexpr int kR0EpiBar = 1;                    // named barrier of the epilogue warps
constexpr uint32_t kR0RowBytes = kR0Half * 2;   // one row's gated values of a head: 256 bytes
constexpr uint32_t kR0GroupBytes = kR0GroupFeat * 2;   // .. and a value group's part of it

// shared memory after the latent tile and the W^UKV stages
struct R0Smem {
  float qg[2][kR0Heads][kR0Half];       // q_h (*) gamma_k,h of the tile's two sequences
  __nv_bfloat16 qr[2][kR0Heads][kR0Rope];   // q^R_h
  float2 wb[2][kR0Heads];               // (sum_f q gamma, q . beta)
  float s1[2][kR0Rows][kR0S1Stride];    // (q gamma) . z_k per row and head, of each key group
  float2 sums[kR0Groups][kR0Rows];      // each group's (sum z, sum z^2) per row
  uint8_t vstage[8][32 * kR0GroupBytes];   // per value warp: its 32 rows, 16-byte chunks swizzled by row
  int tile_b[2], tile_lp[2], tile_page[2], tile_n[2];
  int pair_live;
  uint64_t afull;
  uint64_t bfull[kR0BStages], bempty[kR0BStages];
  uint64_t dfull[2], dfree[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};

constexpr int kR0MaxChunks = 4;   // d_c 256
__host__ __device__ constexpr size_t r0_smem(int nkc) {
  return nkc * kR0AChunkBytes + kR0BStages * kR0BChunkBytes + sizeof(R0Smem) + 1024;
}
static_assert(r0_smem(kR0MaxChunks) <= kSmemMost, "shared memory");

struct R0ProjParams {
  const __nv_bfloat16* q;        // [B, 16, d_n + d_r]
  const __nv_bfloat16* kr_pool;  // [pool rows, d_r]
  const int32_t* id_pool;
  const int32_t* block_table;
  const int32_t* seq_lens;
  const __nv_bfloat16* gate;     // [vocab, 4096]
  const float* gamma;            // [4096] or null
  const float* beta;
  __nv_bfloat16* zv;             // [16][pool rows][d_v]
  float2* stats;                 // [pool rows]: (mu, r)
  float* logit;                  // [B][max_pages * 64][16]
  int batch, max_pages, pool_rows, num_pages, vocab, nkc;
  float eps, scale_log2;
  uint64_t wait_ns;
  int32_t* status;
};

__device__ __forceinline__ bool warp_all_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                              uint64_t limit_ns) {
  __syncwarp();
  const bool ok = mbar_wait(bar, parity, abort_flag, limit_ns);
  return __all_sync(0xffffffffu, ok);
}

__device__ __forceinline__ void epi_sync() {
  asm volatile("barrier.cta.sync %0, %1;" ::"r"(kR0EpiBar), "r"(32 * kR0EpiWarps) : "memory");
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2::evict_last [%0];" ::"l"(reinterpret_cast<uint64_t>(p)));
}

__device__ __forceinline__ float bf(const __nv_bfloat16 x) { return __bfloat162float(x); }

__device__ __forceinline__ float2 widen2(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// Pages 2t and 2t + 1 (t = blockIdx.x) of the walk over the sequences' pages
// (sequence by sequence, each in logical order), found by warp 0: a prefix
// sum of the page counts over the lanes, 32 sequences at a time.  A half with
// no page (past the last) has n = 0 and repeats the other half's page (page 0
// where neither has one: the other CTA of the pair may still have a tile).
// pair_live: the walk reaches the pair's first page.
__device__ void find_tile(const R0ProjParams& p, R0Smem& sm, int lane) {
  const int g0 = 2 * static_cast<int>(blockIdx.x);
  int fb[2] = {-1, -1}, flp[2] = {0, 0}, fl[2] = {0, 0};
  int base = 0;
  const int max_len = p.max_pages * kPage;
  for (int b0 = 0; b0 < p.batch && fb[1] < 0; b0 += 32) {
    const int b = b0 + lane;
    // positions past the block table are not read (the attention kernel reports them)
    const int L = b < p.batch ? min(p.seq_lens[b], max_len) : 0;
    const int np = L > 0 ? (L + kPage - 1) / kPage : 0;
    int inc = np;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    const int excl = base + inc - np;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (fb[k] >= 0) continue;   // uniform
      const int g = g0 + k;
      const unsigned m = __ballot_sync(0xffffffffu, np > 0 && g >= excl && g < excl + np);
      if (m != 0u) {
        const int src = __ffs(m) - 1;
        fb[k] = b0 + src;
        flp[k] = g - __shfl_sync(0xffffffffu, excl, src);
        fl[k] = __shfl_sync(0xffffffffu, L, src);
      }
    }
    base += __shfl_sync(0xffffffffu, inc, 31);
  }
  if (lane == 0) {
    // (base: the pages counted; the loop ends early only past this tile's pages)
    sm.pair_live = base > 4 * static_cast<int>(blockIdx.x / 2) ? 1 : 0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      int page = -1, n = 0;
      if (fb[k] >= 0) {
        page = p.block_table[static_cast<size_t>(fb[k]) * p.max_pages + flp[k]];
        if (page < 0 || page >= p.num_pages) {
          report_status(p.status, kStatusOutOfRange);
          page = -1;
        } else {
          n = min(kPage, fl[k] - flp[k] * kPage);
        }
      }
      sm.tile_b[k] = fb[k];
      sm.tile_lp[k] = flp[k];
      sm.tile_page[k] = page;
      sm.tile_n[k] = n;
    }
    // a half without a page of its own reads the other's (its results are not stored)
    if (sm.tile_page[0] < 0) sm.tile_page[0] = sm.tile_page[1];
    if (sm.tile_page[1] < 0) sm.tile_page[1] = sm.tile_page[0];
    if (sm.tile_b[0] < 0) sm.tile_b[0] = sm.tile_b[1];
    if (sm.tile_b[1] < 0) sm.tile_b[1] = sm.tile_b[0];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      sm.tile_page[k] = max(sm.tile_page[k], 0);
      sm.tile_b[k] = max(sm.tile_b[k], 0);
    }
  }
}

// WIDE: the gate's rows are 32-byte aligned and read in 32-byte pieces, otherwise
// in 16-byte ones (all that the contract asks for)
template <bool WIDE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kR0Threads, 1)
    r0_project_kernel(const __grid_constant__ CUtensorMap cmap, const __grid_constant__ CUtensorMap wmap,
                      const R0ProjParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t b_off = static_cast<uint32_t>(p.nkc) * kR0AChunkBytes;
  R0Smem& sm = *reinterpret_cast<R0Smem*>(smem + b_off + kR0BStages * kR0BChunkBytes);
  volatile int* abort_flag = &sm.abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  const uint32_t rank = cluster_rank();
  if (tid == 0) {
    mbar_init(smem_u32(&sm.afull), 1);
    for (int s = 0; s < kR0BStages; ++s) {
      mbar_init(smem_u32(&sm.bfull[s]), 1);
      mbar_init(smem_u32(&sm.bempty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&sm.dfull[s]), 1);
      mbar_init(smem_u32(&sm.dfree[s]), 2 * kR0EpiWarps);   // both CTAs' epilogue warps, on the leader's
    }
    mbar_init(smem_u32(&sm.drain), 1);
    sm.abort = 0;
    fence_mbar_init();
    prefetch_tensormap(&cmap);
    prefetch_tensormap(&wmap);
  }
  grid_dependency_wait();
  if (warp == 0) find_tile(p, sm, lane);
  __syncthreads();
  if (!sm.pair_live) return;   // past the last page (uniform in both CTAs of the pair)
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&sm.tmem_base), kR0TmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync();   // both CTAs' barriers are ready before either signals them
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;

  bool epi_ok = false;
  if (warp == 0) {
    // ---- TMA: the tile's two pages (all K chunks), then this CTA's half of
    // W^UKV_h chunk by chunk; both CTAs' copies complete on the leader's
    // barriers, which its producer arms for both
    if (elect_one()) {
      const uint64_t pol_stream = policy_evict_first(), pol_keep = policy_evict_last();
      const uint32_t afull = map_to_rank(smem_u32(&sm.afull), 0);
      if (rank == 0) mbar_arrive_expect_tx(smem_u32(&sm.afull), 2 * static_cast<uint32_t>(p.nkc) * kR0AChunkBytes);
      for (int kc = 0; kc < p.nkc; ++kc)
#pragma unroll
        for (int k = 0; k < 2; ++k)
          tma_load_2d_pair(sbase + kc * kR0AChunkBytes + k * kR0APageBytes, &cmap, kc * kR0Chunk,
                           sm.tile_page[k] * kPage, afull, pol_stream);
      int issued = 0, s = 0;
      uint32_t ph = 0;   // phase of stage s
      bool ok = true;
      for (int h = 0; ok && h < kR0Heads; ++h) {
        for (int kc = 0; kc < p.nkc; ++kc) {
          if (issued >= kR0BStages) ok = mbar_wait(smem_u32(&sm.bempty[s]), ph ^ 1, abort_flag, p.wait_ns);
          if (!ok) break;
          if (rank == 0) mbar_arrive_expect_tx(smem_u32(&sm.bfull[s]), 2 * kR0BChunkBytes);
          tma_load_2d_pair(sbase + b_off + s * kR0BChunkBytes, &wmap, kc * kR0Chunk,
                           h * kR0Feat + static_cast<int>(rank) * kR0Half,
                           map_to_rank(smem_u32(&sm.bfull[s]), 0), pol_keep);
          ++issued;
          if (++s == kR0BStages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      // every copy issued lands before either CTA can leave (own flag: bounded,
      // not cut short; the other CTA waits at the cluster barrier at the end)
      if (rank == 0) {
        volatile int own = 0;
        if (!mbar_wait(smem_u32(&sm.afull), 0, &own, p.wait_ns)) *abort_flag = 1;
        for (int i = issued > kR0BStages ? issued - kR0BStages : 0; i < issued; ++i)
          if (!mbar_wait(smem_u32(&sm.bfull[i % kR0BStages]), (i / kR0BStages) & 1, &own, p.wait_ns))
            *abort_flag = 1;
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA (one thread of the leader): head h into accumulator h % 2 once both
    // CTAs' epilogues have read it out; M = 256 (both tiles' rows), N = 256
    if (rank == 0 && elect_one()) {
      constexpr uint32_t idesc = idesc_bf16(2 * kR0Rows, kR0Feat, 0, 0);
      bool ok = mbar_wait(smem_u32(&sm.afull), 0, abort_flag, p.wait_ns), issued = false;
      int s = 0;
      uint32_t ph = 0;
      for (int h = 0; ok && h < kR0Heads; ++h) {
        const int db = h & 1;
        if (h >= 2) ok = mbar_wait_cluster(smem_u32(&sm.dfree[db]), ((h - 2) >> 1) & 1, abort_flag, p.wait_ns);
        for (int kc = 0; ok && kc < p.nkc; ++kc) {
          ok = mbar_wait(smem_u32(&sm.bfull[s]), ph, abort_flag, p.wait_ns);
          if (!ok) break;
          tc_fence_after();
          const uint64_t ad = smem_desc(sbase + kc * kR0AChunkBytes, 16, 1024, kSwizzle128B);
          const uint64_t bd = smem_desc(sbase + b_off + s * kR0BChunkBytes, 16, 1024, kSwizzle128B);
#pragma unroll
          for (int kk = 0; kk < kR0Chunk / 16; ++kk)
            mma_bf16_ss_pair(tmem + db * kR0Feat, ad + ((kk * 32) >> 4), bd + ((kk * 32) >> 4), idesc,
                             (kc > 0 || kk > 0) ? 1u : 0u);
          issued = true;
          mma_commit_pair(smem_u32(&sm.bempty[s]));
          if (++s == kR0BStages) {
            s = 0;
            ph ^= 1;
          }
        }
        if (ok) mma_commit_pair(smem_u32(&sm.dfull[db]));
      }
      // every MMA issued completes before TMEM is released
      if (issued) {
        mma_commit_pair(smem_u32(&sm.drain));
        volatile int own = 0;
        if (!mbar_wait(smem_u32(&sm.drain), 0, &own, p.wait_ns)) *abort_flag = 1;
      }
    }
    __syncwarp();
  } else {
    // ---- epilogue: tile row r is TMEM lane r (warp w reads lane quadrant
    // w % 4); rows 0-63 are the first page, 64-127 the second.  Group g takes
    // columns 64 g .. 64 g + 63 of every head: g < 2 key, g >= 2 value features.
    const uint32_t dfree = map_to_rank(smem_u32(&sm.dfree[0]), 0);
    const int quad = warp & 3, grp = (warp - 2) / 4;
    const bool key = grp < 2;
    const int r = 32 * quad + lane, k = r >> 6, jrow = r & (kPage - 1);
    const int n = sm.tile_n[k], page = sm.tile_page[k];
    const bool valid = jrow < n;
    const size_t prow = static_cast<size_t>(page) * kPage + jrow;
    int id = p.id_pool[prow];
    if (static_cast<unsigned>(id) >= static_cast<unsigned>(p.vocab)) {
      if (valid && grp == 0) report_status(p.status, kStatusOutOfRange);   // the gate uses row 0
      id = 0;
    }
    // the query terms of the tile's two sequences: q gamma (key features),
    // q^R, sum q gamma and q . beta per head
    const int et = tid - 64;
    for (int i = et; i < 2 * kR0Heads * kR0Half; i += 32 * kR0EpiWarps) {
      const int s = i / (kR0Heads * kR0Half), h = (i / kR0Half) % kR0Heads, f = i % kR0Half;
      const float qf = bf(p.q[(static_cast<size_t>(sm.tile_b[s]) * kR0Heads + h) * (kR0Half + kR0Rope) + f]);
      sm.qg[s][h][f] = qf * (p.gamma ? p.gamma[h * kR0Feat + f] : 1.f);
    }
    for (int i = et; i < 2 * kR0Heads * kR0Rope; i += 32 * kR0EpiWarps) {
      const int s = i / (kR0Heads * kR0Rope), h = (i / kR0Rope) % kR0Heads, d = i % kR0Rope;
      sm.qr[s][h][d] = p.q[(static_cast<size_t>(sm.tile_b[s]) * kR0Heads + h) * (kR0Half + kR0Rope) + kR0Half + d];
    }
    for (int pidx = warp - 2; pidx < 2 * kR0Heads; pidx += kR0EpiWarps) {
      const int s = pidx / kR0Heads, h = pidx % kR0Heads;
      const __nv_bfloat16* qh = p.q + (static_cast<size_t>(sm.tile_b[s]) * kR0Heads + h) * (kR0Half + kR0Rope);
      float w = 0.f, bq = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int f = 4 * lane + i;
        const float qf = bf(qh[f]);
        w += qf * (p.gamma ? p.gamma[h * kR0Feat + f] : 1.f);
        bq = fmaf(qf, p.beta ? p.beta[h * kR0Feat + f] : 0.f, bq);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        w += __shfl_xor_sync(0xffffffffu, w, o);
        bq += __shfl_xor_sync(0xffffffffu, bq, o);
      }
      if (lane == 0) sm.wb[s][h] = make_float2(w, bq);
    }
    epi_sync();

    const __nv_bfloat16* grow = p.gate + static_cast<size_t>(id) * kR0Width + grp * kR0GroupFeat;
    const uint64_t pol_gate = policy_evict_last();
    uint8_t* vst = sm.vstage[(warp - 2) & 7];
    const bool store_v = !key && n > 0;   // uniform in the warp
    float2 s1 = make_float2(0.f, 0.f), s2 = make_float2(0.f, 0.f);
    bool ok = true;
    // this group's part of the row's gate values of a head (64 bf16): each
    // quarter of them is requested for head h + 1 as soon as head h has used
    // it, so that the loads run while the rest of head h is processed
    uint4 g[kR0GroupFeat / 8];
    auto load_g = [&](int hh, int i) {
      const __nv_bfloat16* src = grow + hh * kR0Feat + 16 * i;
      if constexpr (WIDE) {
        ldg_32_na_hint(src, pol_gate, g[2 * i], g[2 * i + 1]);
      } else {
        g[2 * i] = ldg_16_na_hint(src, pol_gate);
        g[2 * i + 1] = ldg_16_na_hint(src + 8, pol_gate);
      }
    };
#pragma unroll
    for (int i = 0; i < kR0GroupFeat / 16; ++i) load_g(0, i);
    for (int h = 0; h < kR0Heads; ++h) {
      const int db = h & 1;
      if (h + 2 < kR0Heads) prefetch_l2(grow + (h + 2) * kR0Feat);   // two heads ahead into L2
      ok = ok && warp_all_wait(smem_u32(&sm.dfull[db]), (h >> 1) & 1, abort_flag, p.wait_ns);
      if (!ok) break;
      tc_fence_after();
      const float* qgh = &sm.qg[k][h][(grp & 1) * kR0GroupFeat];
      float2 dot2 = make_float2(0.f, 0.f);
#pragma unroll
      for (int c0 = 0; c0 < kR0GroupFeat; c0 += 32) {
        float v[32];
        const uint32_t ta = tmem + (static_cast<uint32_t>(32 * quad) << 16) + db * kR0Feat + grp * kR0GroupFeat + c0;
        tmem_ld16(ta, *reinterpret_cast<float(*)[16]>(&v[0]));
        tmem_ld16(ta + 16, *reinterpret_cast<float(*)[16]>(&v[16]));
        tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < 4; ++u) {   // 8 columns: one 16-byte unit
          const uint32_t* gw = reinterpret_cast<const uint32_t*>(&g[c0 / 8 + u]);
          uint32_t packed[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 z = __fmul2_rn(make_float2(v[8 * u + 2 * i], v[8 * u + 2 * i + 1]), widen2(gw[i]));
            const __nv_bfloat162 zb = __floats2bfloat162_rn(z.x, z.y);
            packed[i] = *reinterpret_cast<const uint32_t*>(&zb);
            const float2 zr = widen2(packed[i]);   // statistics and dots of the rounded values
            s1 = __fadd2_rn(s1, zr);
            s2 = __ffma2_rn(zr, zr, s2);
            if (key) {
              const float2 qv = *reinterpret_cast<const float2*>(qgh + c0 + 8 * u + 2 * i);
              dot2 = __ffma2_rn(qv, zr, dot2);
            }
          }
          if (!key)   // this unit of the row, at (unit ^ (row % 8)) in its 128-byte row
            *reinterpret_cast<uint4*>(vst + lane * kR0GroupBytes + (((c0 / 8 + u) ^ (lane & 7)) << 4)) =
                make_uint4(packed[0], packed[1], packed[2], packed[3]);
          if ((u & 1) && h + 1 < kR0Heads) load_g(h + 1, c0 / 16 + u / 2);   // these 16 columns done
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(dfree + db * 8);
      if (key) {
        sm.s1[grp][r][h] = dot2.x + dot2.y;
      } else if (store_v) {
        // the warp's 32 rows of head h (head-major), its 128 bytes of each:
        // four rows per store instruction
        uint8_t* dst = reinterpret_cast<uint8_t*>(
                           p.zv + (static_cast<size_t>(h) * p.pool_rows + static_cast<size_t>(page) * kPage +
                                   32 * (quad & 1)) * kR0Half) + (grp & 1) * kR0GroupBytes;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int rr = 4 * i + (lane >> 3), c = lane & 7;
          *reinterpret_cast<uint4*>(dst + rr * kR0RowBytes + c * 16) =
              *reinterpret_cast<const uint4*>(vst + rr * kR0GroupBytes + ((c ^ (rr & 7)) << 4));
        }
        __syncwarp();   // the tile is read before the next head rewrites it
      }
    }
    sm.sums[grp][r] = make_float2(s1.x + s1.y, s2.x + s2.y);
    epi_ok = ok;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (epi_ok && !sm.abort) {
    // the row's statistics over all 4096 features, then its logits: four heads
    // per group
    const int grp = (warp - 2) / 4, r = 32 * (warp & 3) + lane, k = r >> 6, jrow = r & (kPage - 1);
    const size_t prow = static_cast<size_t>(sm.tile_page[k]) * kPage + jrow;
    float t1 = 0.f, t2 = 0.f;
#pragma unroll
    for (int g = 0; g < kR0Groups; ++g) {
      t1 += sm.sums[g][r].x;
      t2 += sm.sums[g][r].y;
    }
    const float mu = t1 / kR0Width;
    const float var = fmaxf(t2 / kR0Width - mu * mu, 0.f);
    const float rinv = rsqrtf(var + p.eps);
    if (grp == 0 && sm.tile_n[k] > 0) p.stats[prow] = make_float2(mu, rinv);
    if (jrow < sm.tile_n[k]) {
      const uint4* kr4 = reinterpret_cast<const uint4*>(p.kr_pool + prow * kR0Rope);
      uint4 kr[kR0Rope / 8];
#pragma unroll
      for (int i = 0; i < kR0Rope / 8; ++i) kr[i] = kr4[i];
      float lg[kR0Heads / kR0Groups];
#pragma unroll
      for (int e = 0; e < kR0Heads / kR0Groups; ++e) {
        const int h = 4 * grp + e;
        const __nv_bfloat162* qr2 = reinterpret_cast<const __nv_bfloat162*>(&sm.qr[k][h][0]);
        float sr = 0.f;
#pragma unroll
        for (int d = 0; d < kR0Rope / 2; ++d) {
          const float2 qf = __bfloat1622float2(qr2[d]);
          const float2 kf = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(kr)[d]);
          sr = fmaf(qf.x, kf.x, fmaf(qf.y, kf.y, sr));
        }
        const float2 wb = sm.wb[k][h];
        lg[e] = p.scale_log2 * (rinv * (sm.s1[0][r][h] + sm.s1[1][r][h] - mu * wb.x) + wb.y + sr);
      }
      const size_t pos = static_cast<size_t>(sm.tile_b[k]) * p.max_pages * kPage +
                         static_cast<size_t>(sm.tile_lp[k]) * kPage + jrow;
      reinterpret_cast<float4*>(p.logit + pos * kR0Heads)[grp] = make_float4(lg[0], lg[1], lg[2], lg[3]);
    }
  }
  // neither CTA leaves (or frees its tensor memory) while the other's copies,
  // MMAs or arrivals may still reach it
  __syncwarp();
  tc_fence_before();
  cluster_sync();
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem, kR0TmemCols);
  if (tid == 0 && sm.abort) report_status(p.status, kStatusTimeout);
}

struct R0AttnParams {
  const int32_t* block_table;
  const int32_t* seq_lens;
  const __nv_bfloat16* zv;      // [16][pool rows][d_v]
  const float2* stats;          // [pool rows]
  const float* logit;           // [B][max_pages * 64][16]
  const float* gamma;           // [4096] or null
  const float* beta;
  __nv_bfloat16* out;           // [B, H, d_v]
  int max_pages, num_pages, pool_rows;
  int32_t* status;
};

constexpr int kR0AttnWarps = 16;
constexpr int kR0AttnThreads = 32 * kR0AttnWarps;
constexpr int kR0AttnPairs = 12;   // row pairs a warp has in flight at once (24 rows, 6 KB)

// One block per (sequence, head).  Warp w takes the sequence's pages w, w +
// 16, ...: a page's 64 rows of the head's gated values are 16 KB in one piece
// (head-major), read as two rows per load instruction (lane l: row 2i + l/16,
// features 8 (l % 16) .. + 7), 24 rows in flight.  Each half-warp keeps its
// own online softmax over its rows (m, l = sum p, the sums of P' z and P' mu
// with P' = p r); the 32 half-warps are merged at the end.
__global__ void __launch_bounds__(kR0AttnThreads) r0_attend_kernel(const R0AttnParams p) {
  __shared__ float part[2 * kR0AttnWarps][3 + kR0Half];
  const int b = blockIdx.x / kR0Heads, h = blockIdx.x % kR0Heads;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int hw = lane >> 4, c8 = 8 * (lane & 15);   // half-warp, first feature of the lane
  const int max_len = p.max_pages * kPage;
  grid_dependency_wait();
  const int L = min(p.seq_lens[b], max_len);
  if (threadIdx.x == 0 && h == 0 && p.seq_lens[b] > max_len) report_status(p.status, kStatusOutOfRange);
  const float* lgb = p.logit + static_cast<size_t>(b) * max_len * kR0Heads + h;
  const __nv_bfloat16* zh = p.zv + static_cast<size_t>(h) * p.pool_rows * kR0Half + c8;
  const int npages = L > 0 ? (L + kPage - 1) / kPage : 0;
  float m = -INFINITY, l = 0.f, bm = 0.f, acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
  bool bad = false;
  int lp = warp;
  int page = lp < npages ? p.block_table[static_cast<size_t>(b) * p.max_pages + lp] : -1;
  while (lp < npages) {
    // the next page of this warp, requested before this one's rows
    const int lp_next = lp + kR0AttnWarps;
    const int page_next = lp_next < npages ? p.block_table[static_cast<size_t>(b) * p.max_pages + lp_next] : -1;
    if (page < 0 || page >= p.num_pages) {
      bad = true;
    } else {
      const int nrow = min(kPage, L - lp * kPage);
      const size_t row0 = static_cast<size_t>(page) * kPage;
#pragma unroll 1
      for (int r0 = 0; r0 < nrow; r0 += 2 * kR0AttnPairs) {
        uint4 zv[kR0AttnPairs];
        float s[kR0AttnPairs];
        float2 st[kR0AttnPairs];
#pragma unroll
        for (int i = 0; i < kR0AttnPairs; ++i) {
          const int r = r0 + 2 * i + hw;
          if (r < nrow) {
            zv[i] = *reinterpret_cast<const uint4*>(zh + (row0 + r) * kR0Half);
            s[i] = lgb[static_cast<size_t>(lp * kPage + r) * kR0Heads];
            st[i] = p.stats[row0 + r];
          }
        }
#pragma unroll
        for (int i = 0; i < kR0AttnPairs; ++i) {
          if (r0 + 2 * i + hw >= nrow) continue;   // uniform in the half-warp
          const float mn = fmaxf(m, s[i]);
          const float alpha = exp2f(m - mn), pj = exp2f(s[i] - mn);
          const float w = pj * st[i].y;
          l = fmaf(l, alpha, pj);
          bm = fmaf(bm, alpha, w * st[i].x);
          const __nv_bfloat162* z2 = reinterpret_cast<const __nv_bfloat162*>(&zv[i]);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 zf = __bfloat1622float2(z2[j]);
            acc[2 * j] = fmaf(acc[2 * j], alpha, w * zf.x);
            acc[2 * j + 1] = fmaf(acc[2 * j + 1], alpha, w * zf.y);
          }
          m = mn;
        }
      }
    }
    lp = lp_next;
    page = page_next;
  }
  if (bad) report_status(p.status, kStatusOutOfRange);
  const int slot = 2 * warp + hw;
  if ((lane & 15) == 0) {
    part[slot][0] = m;
    part[slot][1] = l;
    part[slot][2] = bm;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) part[slot][3 + c8 + i] = acc[i];
  __syncthreads();
  if (warp == 0) {
    // lane l: value features 4l .. 4l + 3
    const int fv = h * kR0Feat + kR0Half + 4 * lane;
    float M = -INFINITY;
    for (int w = 0; w < 2 * kR0AttnWarps; ++w) M = fmaxf(M, part[w][0]);
    float Ls = 0.f, Bs = 0.f, a[4] = {0.f, 0.f, 0.f, 0.f};
    for (int w = 0; w < 2 * kR0AttnWarps; ++w) {
      const float sc = part[w][0] == -INFINITY ? 0.f : exp2f(part[w][0] - M);
      Ls = fmaf(part[w][1], sc, Ls);
      Bs = fmaf(part[w][2], sc, Bs);
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = fmaf(part[w][3 + 4 * lane + i], sc, a[i]);
    }
    __nv_bfloat16* ob = p.out + (static_cast<size_t>(b) * kR0Heads + h) * kR0Half + 4 * lane;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float gv = p.gamma ? p.gamma[fv + i] : 1.f, bv = p.beta ? p.beta[fv + i] : 0.f;
      ob[i] = __float2bfloat16_rn(L > 0 && Ls > 0.f ? fmaf(gv, (a[i] - Bs) / Ls, bv) : 0.f);
    }
  }
}

// row-major bf16 [rows, cols], boxes of 64 columns x box_rows rows, 128-byte swizzle
bool r0_encode(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  std::memset(map, 0, sizeof(*map));
  return encode_map(map, base, {cols, rows}, {cols}, {kR0Chunk, box_rows});
}

}  // namespace

size_t r0_workspace_bytes(int batch, int max_pages, int num_pages) {
  const size_t rows = static_cast<size_t>(num_pages) * kPage;
  const size_t positions = static_cast<size_t>(batch) * max_pages * kPage;
  return align_up(rows * kR0Heads * kR0Half * 2, 256) + align_up(rows * sizeof(float2), 256) +
         align_up(positions * kR0Heads * sizeof(float), 256);
}

cudaError_t launch_decode_r0(const R0Args& a, cudaStream_t st) {
  const size_t rows = static_cast<size_t>(a.num_pages) * kPage;
  uint8_t* ws = static_cast<uint8_t*>(a.workspace);
  __nv_bfloat16* zv = reinterpret_cast<__nv_bfloat16*>(ws);
  size_t off = align_up(rows * kR0Heads * kR0Half * 2, 256);
  float2* stats = reinterpret_cast<float2*>(ws + off);
  off += align_up(rows * sizeof(float2), 256);
  float* logit = reinterpret_cast<float*>(ws + off);
  CUtensorMap cmap, wmap;
  if (!r0_encode(&cmap, a.c_pool, rows, static_cast<uint64_t>(a.d_c), kPage)) return cudaErrorInvalidValue;
  if (!r0_encode(&wmap, a.w_ukv, kR0Width, static_cast<uint64_t>(a.d_c), kR0Half)) return cudaErrorInvalidValue;
  const int nkc = a.d_c / kR0Chunk;
  const size_t smem = r0_smem(nkc);
  const auto project = (reinterpret_cast<uintptr_t>(a.gate_r0) & 31) == 0 ? r0_project_kernel<true> : r0_project_kernel<false>;
  cudaError_t e = allow_smem(project, r0_smem(kR0MaxChunks));
  if (e != cudaSuccess) return e;
  R0ProjParams pp;
  pp.q = static_cast<const __nv_bfloat16*>(a.q);
  pp.kr_pool = static_cast<const __nv_bfloat16*>(a.kr_pool);
  pp.id_pool = a.id_pool;
  pp.block_table = a.block_table;
  pp.seq_lens = a.seq_lens;
  pp.gate = static_cast<const __nv_bfloat16*>(a.gate_r0);
  pp.gamma = a.ln_gamma;
  pp.beta = a.ln_beta;
  pp.zv = zv;
  pp.stats = stats;
  pp.logit = logit;
  pp.batch = a.batch;
  pp.max_pages = a.max_pages;
  pp.pool_rows = static_cast<int>(rows);
  pp.num_pages = a.num_pages;
  pp.vocab = a.vocab;
  pp.nkc = nkc;
  pp.eps = a.eps;
  pp.scale_log2 = a.scale_log2;
  pp.wait_ns = kWaitLimitNs;
  pp.status = a.status;
  // one CTA per two pages of the walk: the block table bounds the pages in use
  // (an even number: the CTAs work in pairs)
  const int tiles = static_cast<int>((static_cast<int64_t>(a.batch) * a.max_pages + 3) / 4 * 2);
  e = launch_chained(project, dim3(tiles), dim3(kR0Threads), smem, st, cmap, wmap, pp);
  if (e != cudaSuccess) return e;
  R0AttnParams ap;
  ap.block_table = a.block_table;
  ap.seq_lens = a.seq_lens;
  ap.zv = zv;
  ap.stats = stats;
  ap.logit = logit;
  ap.gamma = a.ln_gamma;
  ap.beta = a.ln_beta;
  ap.out = static_cast<__nv_bfloat16*>(a.out);
  ap.max_pages = a.max_pages;
  ap.num_pages = a.num_pages;
  ap.pool_rows = static_cast<int>(rows);
  ap.status = a.status;
  return launch_chained(r0_attend_kernel, dim3(a.batch * kR0Heads), dim3(kR0AttnThreads), 0, st, ap);
}

}  // namespace egmla
