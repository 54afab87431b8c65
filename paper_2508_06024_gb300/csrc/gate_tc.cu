// Gate of the layer path on the sm_103a tensor cores (Eq. 4-7 gate, Top-k
// and the fused routing reservations); the SIMT gates and the dispatch are in
// gate.cu.
#include <stdlib.h>

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include "common.cuh"
#include "gate_common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace ec2moe {

__device__ unsigned int g_gate_error;  // bit 0: a bounded wait of the tensor-core gate timed out

namespace gatek {
namespace {

// ---------------------------------------------------------------------------
// Gate on the tensor cores (bf16 activations, O = E + K <= 80 gate rows).
//
// The logits are the contraction X_tile W^T with W the fp32 gate rows.  Each
// fp32 weight is split exactly into three bf16 terms, w = w0 + w1 + w2 (w0 =
// bf16(w), w1 = bf16(w - w0), w2 = bf16(w - w0 - w1); every difference is
// exact in fp32, and the remainder is below 2^-24 |w|).  A bf16 activation
// times a bf16 term is exact in fp32, so X W^T = X w0^T + X w1^T + X w2^T keeps
// the fp32 weights to fp32 accuracy.  The three terms are stacked as the rows
// of one B operand [w0; w1; w2] (N = 3 * O_pad, O_pad = O rounded up to 16),
// so one tcgen05.mma per 16 columns of d_model produces all three partial
// products side by side in TMEM; the epilogue adds them in fp32.
//
// One CTA owns 128-token tiles; d_model streams through shared memory 64
// columns per stage:
//   warp 0       TMA: the X box (128 x 64 bf16, 128-byte swizzle) and the
//                stacked split rows of the stage -- either straight from a
//                prepared [3 * O_pad, d] bf16 matrix (PREP: made by
//                gate_split_kernel); without one, warps 6..13 take the fp32
//                rows (staged by TMA or loaded to registers, gc_raw) and write
//                their split into the swizzled layout;
//   warp 1       4 MMAs (M = 128, N = 3 O_pad, K = 16) per stage into one of
//                two TMEM accumulators; every GC_SEG stages (256 columns of
//                d_model) the accumulator is handed over and the next segment
//                starts from zero in the other one;
//   warps 2..5   add each segment into fp32 registers (one token row per
//                thread; warp w reads TMEM lanes 32 (w % 4) .. +31), so every
//                dot product is a sum of short partial sums; at the end of the
//                tile they add the bias and write the logits rows;
//   warps 2..13  take the softmax / Top-k decisions (lse_rows, pick_row) and, on
//                the layer path, reserve the tile's rows per expert.
// With d_model of 2048 or more (32 or more stages per tile) a tile belongs to
// a cluster of GC_CS CTAs on as many SMs instead: CTA c of the cluster runs
// the stages [c nk / GC_CS, (c + 1) nk / GC_CS) and owns the decisions of
// rows [c 128 / GC_CS, (c + 1) 128 / GC_CS).  Each drain thread sends its
// row's partial logits to the row's owner (st.async into the owner's shared
// memory, counted on the owner's receive barrier), and the owner adds the
// cluster's partials in CTA order before the bias and the decision; every CTA
// reserves the rows it decided.  One tile per cluster: such grids are one
// cluster per tile, run in waves when they exceed the SMs.  A tile's stages
// (the stream of X, the MMAs and the accumulator drains) are then spread over
// twice the SMs.
// Every mbarrier wait is bounded; on a timeout the error word is set, copies
// and MMAs in flight are drained and the CTA finishes its tiles without
// waiting (the decisions then see garbage logits but still name valid experts).
constexpr int GC_BM = 128;
constexpr int GC_BK = 64;
constexpr int GC_SEG = 4;
constexpr int GC_MAX_O = 80;
constexpr int GC_MAX_STAGES = 10;
constexpr int GC_THREADS = 448;
constexpr int GC_WORKERS = 384;     // warps 2..13
// Without prepared rows every worker warp is busy in the main loop, so a warp of
// its own brings the decision's code to the SM (a drain warp doing it held up
// short main loops: fine-grained steps, T = 2001, 343 -> 340 us).
constexpr int GC_WARM_WARP = 14;
constexpr int GC_ACC_STRIDE = 256;  // TMEM columns between the two accumulators (3 * O_pad <= 240 each)
constexpr int GC_CS = 2;            // CTAs per tile (cluster) when d_model is split
constexpr int GC_SPLIT_MIN_NK = 32; // stages per tile from which d_model is split

// Without prepared rows, whether the fp32 rows of a stage come by TMA (nb blocks
// of 16 gate rows) or from global memory to the converting warps' registers, one
// stage ahead.  By TMA they arrive as many stages ahead as the ring is deep, but
// take 256 bytes a row of each stage: up to 32 rows the ring stays deep and the
// loads' latency decides, beyond that the stages do (standalone gate, T = 2000,
// cold L2, launch bracket included, us, registers -> TMA: d = 768, E = 16 20.8 ->
// 17.6, E = 32 24.2 -> 20.2; d = 4096, E = 16 36.5 -> 27.9, E = 32 51.8 -> 43.7;
// E = 64, Top-1, TMA -> registers: d = 768 39 -> 30, d = 4096 74 -> 68).
__host__ __device__ constexpr bool gc_raw(int nb, bool prep) { return !prep && nb <= 2; }

struct GcLayout {
  int n_pad, O, k, E, stages, cs;
  int stage_bytes, w3_off, raw_off;
  int log_stride;  // logits row of a token: O logits + 16 group scratch words, odd (conflict-free rows)
  int rstride;     // floats per received partial-logit row: n_pad + 4 (16-byte rows, shifted banks)
  int log_off, idx_off, tab_off, base_off, bias_off, list_off, recv_off, bar_off, warm_off, total;
  __host__ __device__ GcLayout(int O_, int k_, int E_, int stages_, int cs_, bool raw)
      : O(O_), k(k_), E(E_), stages(stages_), cs(cs_) {
    n_pad = (O + 15) / 16 * 16;
    w3_off = GC_BM * GC_BK * 2;
    raw_off = w3_off + 3 * n_pad * 128;
    stage_bytes = raw_off + (raw ? n_pad * 256 : 0);  // a multiple of 1024
    log_stride = (O + 16) | 1;
    rstride = n_pad + 4;
    log_off = stages * stage_bytes;
    idx_off = log_off + GC_BM * log_stride * 4;
    tab_off = idx_off + GC_BM * k * 4;
    base_off = tab_off + (GC_BM * k / 32) * E * 4;
    bias_off = base_off + 4 * E;
    // received partials: [source CTA][owned row][rstride] (cs > 1)
    list_off = bias_off + 4 * O;  // allowed experts, then the first list place of each group
    recv_off = (list_off + 4 * (E + 17) + 15) / 16 * 16;
    bar_off = (recv_off + (cs > 1 ? GC_BM * rstride * 4 : 0) + 7) / 8 * 8;
    // a logits row of its own for the warm-up of the decision's code
    warm_off = bar_off + (3 * stages + 6) * 8 + 16;
    total = warm_off + (O + 16) * 4;
  }
};

struct GcParams {
  KParams kp;
  int n_pad;
  int stages;
  int cs;  // CTAs per tile (cluster size); 1 = one CTA per tile, persistent over tiles
  long long timeout;
};

// The decision, from a tile's logits rows in shared memory (L[0..E) local,
// L[E..E+K) global, then 16 scratch words G) and the list of allowed experts
// in ascending order, cut into groups by s_grp[0..K].  Two steps:
//   lse_rows   G[g] = log-sum-exp of group g's allowed members (Eq. 5), one
//              (row, group) per thread, all worker threads; K = 1: the whole
//              list as one group
//   pick_row   one thread per row: top-group pruning when top_groups > 0 (only
//              the top_groups live groups by m stay), log-sum-exp of the global
//              logits over the live (kept) groups (Eq. 6), key = (m_g - lse_g) +
//              l_i (K = 1: l_i), Top-k by insertion into a sorted list (larger
//              key first, ties to the lower index), weight exp((m_g - LSE_m) +
//              (l_i - lse_g)) (Eq. 7).  Slots left empty by non-finite keys take
//              the lowest allowed experts not chosen yet.
// The steps run once per tile, with code that the previous kernels' streams
// have evicted from L2, so their size counts as much as their arithmetic: they
// are rolled loops behind one call each, and an idle warp calls both on a
// scratch row during the main loop, which brings the code to the SM before it
// is needed.  (Fully unrolled per-thread decisions took 25 us of the
// fine-grained gate and ~20 us of a 64-expert Top-1 one.)
struct MaskRegs {
  uint32_t w0, w1, w2, w3;
  __device__ __forceinline__ bool has(int e) const {
    const uint32_t w = e < 64 ? (e < 32 ? w0 : w1) : (e < 96 ? w2 : w3);
    return (w >> (e & 31)) & 1u;
  }
};

// Insert (key, e, lw) into a list sorted by key (descending); e arrives in
// ascending order, so an equal key stays behind the earlier expert.
template <int KS>
__device__ __forceinline__ void topk_insert(float* tk, float* tl, int* ti, float key, int e, float lw) {
#pragma unroll
  for (int q = KS - 1; q >= 0; --q) {
    if (key > tk[q]) {
      if (q > 0 && key > tk[q - 1]) {
        tk[q] = tk[q - 1];
        tl[q] = tl[q - 1];
        ti[q] = ti[q - 1];
      } else {
        tk[q] = key;
        tl[q] = lw;
        ti[q] = e;
      }
    }
  }
}

__device__ __noinline__ void lse_rows(float* sLog, int log_stride, int O, const int* s_list, const int* s_grp, int K,
                                      int row_lo, int n_rows, int wt, int threads) {
#pragma unroll 1
  for (int i = wt; i < n_rows * K; i += threads) {
    const int r = i / K, g = i - r * K;
    float* L = sLog + (row_lo + r) * log_stride;
    const int lo = s_grp[g], hi = s_grp[g + 1];
    float mx = -CUDART_INF_F;
#pragma unroll 4
    for (int j = lo; j < hi; ++j) mx = fmaxf(mx, L[s_list[j]]);
    float sum = 0.0f;
#pragma unroll 4
    for (int j = lo; j < hi; ++j) sum += expf(L[s_list[j]] - mx);
    L[O + g] = mx > -CUDART_INF_F ? mx + logf(sum) : -CUDART_INF_F;
  }
}

// KS >= k slots are kept (KS in {1, 2, 4, 8}); `real` false: nothing is written
// outside the row's scratch words.
template <int KS>
__device__ __noinline__ void pick_row(const KParams& p, float* L, int O, const int* s_list, const int* s_grp, int tok,
                                      int* s_idx, bool real) {
  const bool grouped = p.K > 1;
  const int ng = p.K;
  const int k = p.k;
  float* G = L + O;
  float tk[KS], tl[KS];
  int ti[KS];
#pragma unroll
  for (int j = 0; j < KS; ++j) {
    tk[j] = -CUDART_INF_F;
    tl[j] = 0.0f;
    ti[j] = -1;
  }
  float lse_m = 0.0f;
  if (grouped) {
    // top-group pruning: only the top_groups live groups by m (ties to the
    // lower group index) keep their experts and their share of p_group
    if (p.top_groups > 0 && p.top_groups < ng) {
      uint32_t keep = 0;
#pragma unroll 1
      for (int g = 0; g < ng; ++g) {
        if (G[g] == -CUDART_INF_F) continue;
        const float mg = L[p.E + g];
        int rank = 0;
#pragma unroll 1
        for (int j = 0; j < ng; ++j) {
          const float mj = L[p.E + j];
          if (j != g && G[j] > -CUDART_INF_F && (mj > mg || (mj == mg && j < g))) ++rank;
        }
        if (rank < p.top_groups) keep |= 1u << g;
      }
#pragma unroll 1
      for (int g = 0; g < ng; ++g)
        if (!((keep >> g) & 1u)) G[g] = -CUDART_INF_F;
    }
    float mxm = -CUDART_INF_F;
#pragma unroll 2
    for (int g = 0; g < ng; ++g)
      if (G[g] > -CUDART_INF_F) mxm = fmaxf(mxm, L[p.E + g]);
    float summ = 0.0f;
#pragma unroll 2
    for (int g = 0; g < ng; ++g)
      if (G[g] > -CUDART_INF_F) summ += expf(L[p.E + g] - mxm);
    lse_m = mxm + logf(summ);
  }
#pragma unroll 1
  for (int g = 0; g < ng; ++g) {
    const float lg = G[g];
    if (grouped && lg == -CUDART_INF_F) continue;  // no allowed member, or pruned
    const float mk = grouped ? L[p.E + g] : 0.0f;
    const int hi = s_grp[g + 1];
#pragma unroll 2
    for (int j = s_grp[g]; j < hi; ++j) {
      const int e = s_list[j];
      const float le = L[e];
      const float key = grouped ? (mk - lg) + le : le;
      if (key > tk[KS - 1]) topk_insert<KS>(tk, tl, ti, key, e, grouped ? (mk - lse_m) + (le - lg) : le - lg);
    }
  }
  // non-finite keys: fill empty slots with the lowest allowed experts not chosen
  if (ti[KS - 1] < 0) {
    const MaskRegs m{p.mask_bits[0], p.mask_bits[1], p.mask_bits[2], p.mask_bits[3]};
    const int gsize = p.E / ng;
    int next = 0;
#pragma unroll
    for (int s = 0; s < KS; ++s) {
      if (s < k && ti[s] < 0) {
#pragma unroll 1
        for (; next < p.E; ++next) {
          if (!m.has(next)) continue;
          bool used = false;
#pragma unroll
          for (int q = 0; q < KS; ++q) used |= (ti[q] == next);
          if (!used) break;
        }
        const int e = next < p.E ? next : 0;
        ++next;
        const int g = e / gsize;
        ti[s] = e;
        tl[s] = grouped ? (L[p.E + g] - lse_m) + (L[e] - G[g]) : L[e] - G[0];
      }
    }
  }
  float gw[KS];
  float wsum = 0.0f;
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    gw[s] = s < k ? expf(tl[s]) : 0.0f;
    wsum += gw[s];
  }
  if (!real) {
    G[0] = wsum;  // keep the work
    return;
  }
#pragma unroll
  for (int s = 0; s < KS; ++s)
    if (s < k) {
      p.topk_idx[(size_t)tok * k + s] = ti[s];
      p.topk_w[(size_t)tok * k + s] = p.renorm ? gw[s] / wsum : gw[s];
      s_idx[s] = ti[s];
    }
}

// The Top-1 decision for one group of at most 16 experts from the logits in
// registers (x[e], bias included; only the standalone gate takes it), with the
// arithmetic of lse_rows and pick_row<1>: straight-line code, short enough to be
// fetched while it runs (E = 16, T = 2000, us, rolled loops -> this: d = 768 17.6
// -> 16.9, d = 4096 27.9 -> 26.2; the same for Top-2 was slower, 19.2 -> 20.1).
__device__ __forceinline__ void decide_top1(const KParams& p, const float (&x)[16], int tok) {
  const uint32_t allowed = p.mask_bits[0];
  float mx = -CUDART_INF_F, best = -CUDART_INF_F;
  int pick = -1;
#pragma unroll
  for (int e = 0; e < 16; ++e)
    if (allowed >> e & 1u) {
      mx = fmaxf(mx, x[e]);
      if (x[e] > best) {
        best = x[e];
        pick = e;
      }
    }
  float sum = 0.0f;
#pragma unroll
  for (int e = 0; e < 16; ++e)
    if (allowed >> e & 1u) sum += expf(x[e] - mx);
  const float lse = mx > -CUDART_INF_F ? mx + logf(sum) : -CUDART_INF_F;
  if (pick < 0) {  // non-finite logits: the lowest allowed expert
#pragma unroll
    for (int e = 15; e >= 0; --e)
      if (allowed >> e & 1u) {
        best = x[e];
        pick = e;
      }
  }
  const float w = expf(best - lse);
  p.topk_idx[tok] = pick;
  p.topk_w[tok] = p.renorm ? w / w : w;
}

// Rows [row_lo, row_lo + n_rows) of the tile reserved per expert (the layer
// path), with the worker warps only: entry i of the range (token row_lo + i /
// k of the tile, slot i % k) gets route_rel = the expert's reserved base + the
// number of earlier entries of the range with the same expert.  sIdx holds the
// range's decisions.  32-entry chunks are ranked with a warp match, chunk
// counts are turned into per-expert prefixes, and one atomicAdd per expert
// reserves the range's rows.
__device__ void route_tile_workers(const KParams& p, int tile, int row_lo, int n_rows, const int* sIdx, int* sTab,
                                   int* s_base, int wt) {
  const int wi = wt >> 5, lane = wt & 31;
  const int nt = n_rows * p.k;
  const long long e0 = ((long long)tile * GC_BM + row_lo) * p.k;
  const long long n = (long long)p.T * p.k;
  const long long rem = n - e0;
  const int live = rem <= 0 ? 0 : (int)(rem < nt ? rem : nt);
  const int nch = (live + 31) / 32;
  constexpr int NW = GC_WORKERS / 32;
  constexpr int MAXC = (GC_BM * MAX_TOPK / 32 + NW - 1) / NW;
  for (int i = wt; i < nch * p.E; i += GC_WORKERS) sTab[i] = 0;
  asm volatile("bar.sync 1, %0;" ::"r"(GC_WORKERS) : "memory");
  int rank[MAXC], ex[MAXC];
#pragma unroll
  for (int ci = 0; ci < MAXC; ++ci) {
    const int c = wi + ci * NW;
    const int i = c * 32 + lane;
    int e = -1;
    if (c < nch && i < live) {
      e = sIdx[i];
      if (e < 0 || e >= p.E) e = -1;
    }
    ex[ci] = e;
    rank[ci] = 0;
    if (c < nch) {
      const unsigned m = __match_any_sync(0xffffffffu, e);
      rank[ci] = __popc(m & ((1u << lane) - 1u));
      if (e >= 0 && lane == __ffs(m) - 1) sTab[c * p.E + e] = __popc(m);
    }
  }
  asm volatile("bar.sync 1, %0;" ::"r"(GC_WORKERS) : "memory");
  if (wt < p.E) {
    int run = 0;
    for (int c = 0; c < nch; ++c) {
      const int t = sTab[c * p.E + wt];
      sTab[c * p.E + wt] = run;
      run += t;
    }
    s_base[wt] = run ? atomicAdd(&p.route_counts[wt], run) : 0;
  }
  asm volatile("bar.sync 1, %0;" ::"r"(GC_WORKERS) : "memory");
#pragma unroll
  for (int ci = 0; ci < MAXC; ++ci) {
    const int c = wi + ci * NW;
    const int e = ex[ci];
    if (c < nch && e >= 0) p.route_rel[e0 + c * 32 + lane] = s_base[e] + sTab[c * p.E + e] + rank[ci];
  }
}

// The three bf16 terms of one fp32 pair, packed as bf16x2 words.
__device__ __forceinline__ void split3_pair(float lo, float hi, uint32_t& t0, uint32_t& t1, uint32_t& t2) {
  t0 = pack_bf16x2(lo, hi);
  const float lo1 = lo - bf16_lo(t0), hi1 = hi - bf16_hi(t0);
  t1 = pack_bf16x2(lo1, hi1);
  const float lo2 = lo1 - bf16_lo(t1), hi2 = hi1 - bf16_hi(t1);
  t2 = pack_bf16x2(lo2, hi2);
}

// Prepared split rows for the layer path: Wsplit[j * O_pad + o][c] = term j
// of W[o][c] (local rows, then global rows; rows O..O_pad-1 zero), bf16
// [3 * O_pad, d].  Block 0 also clears the expert row counters the gate's
// routing reserves from.  Thread = 8 consecutive columns of one gate row.
__global__ void __launch_bounds__(256) gate_split_kernel(const float* W_local, const float* W_global, int E, int K,
                                                         int d, int n_pad, __nv_bfloat16* Wsplit,
                                                         int32_t* route_counts) {
  pdl_trigger();
  const int O = E + (K == 1 ? 0 : K);
  if (blockIdx.x == 0 && route_counts)
    for (int e = threadIdx.x; e < E; e += blockDim.x) route_counts[e] = 0;
  const int per_row = d / 8;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)n_pad * per_row) return;
  const int o = (int)(i / per_row);
  const int c = (int)(i % per_row) * 8;
  float v[8];
  if (o < O) {
    const float* src = o < E ? W_local + (size_t)o * d : W_global + (size_t)(o - E) * d;
    load8(src + c, v);
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = 0.0f;
  }
  uint32_t t[3][4];
#pragma unroll
  for (int u = 0; u < 4; ++u) split3_pair(v[2 * u], v[2 * u + 1], t[0][u], t[1][u], t[2][u]);
#pragma unroll
  for (int j = 0; j < 3; ++j)
    *reinterpret_cast<U4*>(Wsplit + ((size_t)j * n_pad + o) * d + c) = U4{t[j][0], t[j][1], t[j][2], t[j][3]};
}

template <int NB, bool PREP>
__global__ void __launch_bounds__(PREP ? GC_THREADS : GC_THREADS + 32, 1)
    gate_tc_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                   const __grid_constant__ CUtensorMap tmWg, const __grid_constant__ GcParams gp) {
  using namespace tc;
  constexpr bool RAW = gc_raw(NB, PREP);
  const KParams& p = gp.kp;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int nglob = (p.K == 1) ? 0 : p.K;
  const int O = p.E + nglob;
  const int cs = gp.cs;
  const GcLayout L(O, p.k, p.E, gp.stages, cs, RAW);
  const int S = gp.stages;
  float* sLog = reinterpret_cast<float*>(smem + L.log_off);
  int* sIdx = reinterpret_cast<int*>(smem + L.idx_off);
  int* sTab = reinterpret_cast<int*>(smem + L.tab_off);
  int* s_base = reinterpret_cast<int*>(smem + L.base_off);
  float* s_bias = reinterpret_cast<float*>(smem + L.bias_off);
  int* s_list = reinterpret_cast<int*>(smem + L.list_off);
  int* s_grp = s_list + p.E;
  float* s_recv = reinterpret_cast<float*>(smem + L.recv_off);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + L.bar_off);
  uint64_t* conv = full + S;
  uint64_t* empty = conv + S;
  uint64_t* tfull = empty + S;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint64_t* recvb = drain + 1;  // partial logits from the other CTAs of the cluster (cs > 1)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(recvb + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const bool top1_regs = NB == 1 && !PREP && !nglob && p.k == 1 && !p.route_counts;  // decide_top1
  const int n_tiles = (p.T + GC_BM - 1) / GC_BM;
  const int nk = (p.d + GC_BK - 1) / GC_BK;
  const long long budget = gp.timeout;
  const int n_pad = gp.n_pad;
  // cs > 1: cluster `tile` of cs CTAs (one tile per cluster); this CTA runs
  // stages [kb_lo, kb_lo + cnt) and decides rows [rank * rows_own, ...)
  const int rank = cs > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int tile_first = cs > 1 ? static_cast<int>(cluster_id_x()) : static_cast<int>(blockIdx.x);
  const int tile_step = cs > 1 ? static_cast<int>(cluster_count_x()) : static_cast<int>(gridDim.x);
  const int kb_lo = rank * nk / cs;
  const int cnt = (rank + 1) * nk / cs - kb_lo;
  const int rows_own = GC_BM / cs;
  pdl_trigger();

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&conv[s]), 8);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tfull[a]), 1);
      mbar_init(smem_u32(&tempty[a]), 4);
    }
    mbar_init(smem_u32(drain), 1);
    mbar_init(smem_u32(recvb), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    // the owned rows' partials of the other cs - 1 CTAs (one tile per cluster)
    if (cs > 1) mbar_expect_tx(smem_u32(recvb), static_cast<uint32_t>((cs - 1) * rows_own * n_pad * 4));
  }
  for (int o = threadIdx.x - 64; o >= 0 && o < O; o += PREP ? GC_THREADS - 64 : GC_THREADS - 32)
    s_bias[o] = o < p.E ? p.b_local[o] : p.b_global[o - p.E];
  if (warp == 2 && !top1_regs) {
    // the allowed experts in ascending order, and where each group's begin
    const int gsize = p.E / p.K;
    int base = 0;
    for (int c = 0; c * 32 < p.E; ++c) {
      const uint32_t bits = p.mask_bits[c];
      const int e = c * 32 + lane;
      const int at = base + __popc(bits & ((1u << lane) - 1u));
      if (bits >> lane & 1u) s_list[at] = e;
      if (e < p.E && e % gsize == 0) s_grp[e / gsize] = at;
      base += __popc(bits);
    }
    if (lane == 0) s_grp[p.K] = base;
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmX);
    if (PREP || RAW) tma_prefetch_desc(&tmW);
    if (RAW && nglob) tma_prefetch_desc(&tmWg);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  // every receive barrier of the cluster is initialised before any partial is sent
  if (cs > 1) cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    // Activations do not depend on the previous kernel, the prepared split
    // rows (PREP) do: the X boxes of the first stages go out before the
    // dependency wait, their split rows after it.
    // The whole warp waits and counts; one elected lane issues.
    {
      const bool issue = elect_one();
      const uint32_t bytes = GC_BM * GC_BK * 2 + (PREP ? 3 * n_pad * GC_BK * 2 : RAW ? O * GC_BK * 4 : 0);
      const int my_tiles = tile_first < n_tiles ? (n_tiles - 1 - tile_first) / tile_step + 1 : 0;
      const int total = my_tiles * cnt;
      const int pre = total < S ? total : S;
      int kc = 0, x_row = tile_first * GC_BM;  // next stage's place
      auto load_x = [&](uint8_t* st, uint32_t fb) {
        if (issue) {
          mbar_expect_tx(fb, bytes);
          if (RAW) {  // first: the rows are converted before X is multiplied
            tma_load_2d(smem_u32(st + L.raw_off), &tmW, (kb_lo + kc) * GC_BK, 0, fb);
            if (nglob) tma_load_2d(smem_u32(st + L.raw_off + p.E * GC_BK * 4), &tmWg, (kb_lo + kc) * GC_BK, 0, fb);
          }
          tma_load_2d(smem_u32(st), &tmX, (kb_lo + kc) * GC_BK, x_row, fb);
        }
      };
      auto next = [&] {
        if (++kc == cnt) {
          kc = 0;
          x_row += tile_step * GC_BM;
        }
      };
      for (int c = 0; c < pre; ++c, next()) load_x(smem + c * L.stage_bytes, smem_u32(&full[c]));
      pdl_wait();
      if (PREP && issue)
        for (int c = 0, wk = 0; c < pre; ++c, wk = wk + 1 == cnt ? 0 : wk + 1)
          tma_load_2d(smem_u32(smem + c * L.stage_bytes + L.w3_off), &tmW, (kb_lo + wk) * GC_BK, 0, smem_u32(&full[c]));
      int stage = pre == S ? 0 : pre;
      uint32_t phase = (pre == S) ? 1u : 0u;
      uint32_t issued = pre ? ((1u << pre) - 1u) : 0u, issued_phase = 0;
      bool ok = true;
      for (int c = pre; c < total; ++c) {
        if (!__all_sync(0xffffffffu,
                        mbar_wait(smem_u32(&empty[stage]), phase ^ 1u, budget, abort_flag, &g_gate_error))) {
          ok = false;
          break;
        }
        uint8_t* st = smem + stage * L.stage_bytes;
        const uint32_t fb = smem_u32(&full[stage]);
        load_x(st, fb);
        if (PREP && issue) tma_load_2d(smem_u32(st + L.w3_off), &tmW, (kb_lo + kc) * GC_BK, 0, fb);
        next();
        issued |= 1u << stage;
        issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
        if (++stage == S) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!ok || *abort_flag) {
        for (int s = 0; s < S; ++s)
          if (issued & (1u << s)) mbar_drain(smem_u32(&full[s]), (issued_phase >> s) & 1u, DRAIN_CYCLES);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // the whole warp waits and counts, so that descriptors stay in uniform
    // registers; one elected lane issues
    {
      const bool issue = elect_one();
      const uint32_t idesc = idesc_bf16(GC_BM, 3 * n_pad);
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t uses0 = 0, uses1 = 0;
      bool ok = true, any = false;
      for (int tile = tile_first; tile < n_tiles && ok; tile += tile_step) {
        for (int seg = 0; seg < cnt && ok; seg += GC_SEG) {
          const uint32_t uses = acc ? uses1 : uses0;
          if (!__all_sync(0xffffffffu,
                          mbar_wait(smem_u32(&tempty[acc]), (uses & 1u) ^ 1u, budget, abort_flag, &g_gate_error))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + acc * GC_ACC_STRIDE;
          const int seg_end = seg + GC_SEG < cnt ? seg + GC_SEG : cnt;
          for (int kc = seg; kc < seg_end; ++kc) {
            const bool landed =
                (PREP || mbar_wait(smem_u32(&conv[stage]), phase, budget, abort_flag, &g_gate_error)) &&
                mbar_wait(smem_u32(&full[stage]), phase, budget, abort_flag, &g_gate_error);
            if (!__all_sync(0xffffffffu, landed)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint8_t* st = smem + stage * L.stage_bytes;
            const uint64_t da = sdesc_sw128(smem_u32(st));
            const uint64_t db = sdesc_sw128(smem_u32(st + L.w3_off));
            if (issue) {
#pragma unroll
              for (int kk = 0; kk < GC_BK / 16; ++kk)
                umma_bf16(d_tmem, da + 2 * kk, db + 2 * kk, idesc, (kc != seg || kk != 0) ? 1u : 0u);
              umma_commit(smem_u32(&empty[stage]));
            }
            any = true;
            if (++stage == S) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (!ok) break;
          if (issue) umma_commit(smem_u32(&tfull[acc]));
          if (acc) ++uses1;
          else ++uses0;
          acc ^= 1;
        }
      }
      if ((!ok || *abort_flag) && any && issue) {
        umma_commit(smem_u32(drain));
        mbar_drain(smem_u32(drain), 0, DRAIN_CYCLES);
      }
    }
  } else if (!PREP && warp == GC_WARM_WARP) {
    // the decision's code to the SM, as an idle warp does below with prepared rows
    if (!top1_regs) {
      float* warm = reinterpret_cast<float*>(smem + L.warm_off);
      lse_rows(warm, 0, O, s_list, s_grp, p.K, 0, 1, lane, 32);
      if (p.k == 1) pick_row<1>(p, warm, O, s_list, s_grp, 0, nullptr, false);
      else if (p.k == 2) pick_row<2>(p, warm, O, s_list, s_grp, 0, nullptr, false);
      else if (p.k <= 4) pick_row<4>(p, warm, O, s_list, s_grp, 0, nullptr, false);
      else pick_row<8>(p, warm, O, s_list, s_grp, 0, nullptr, false);
    }
  } else {
    // ------------------------------------------------------------ worker warps
    const int wt = threadIdx.x - 64;
    const bool is_drain = warp < 6;
    const int q = warp & 3;
    const int row = q * 32 + lane;
    const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
    auto pick = [&](float* Lr, int* sx, int tok, bool real) {
      if (p.k == 1) pick_row<1>(p, Lr, O, s_list, s_grp, tok, sx, real);
      else if (p.k == 2) pick_row<2>(p, Lr, O, s_list, s_grp, tok, sx, real);
      else if (p.k <= 4) pick_row<4>(p, Lr, O, s_list, s_grp, tok, sx, real);
      else pick_row<8>(p, Lr, O, s_list, s_grp, tok, sx, real);
    };
    if (PREP && warp == 6) {
      // an idle warp: bring the decision's code to the SM (on a row of its own,
      // whatever it holds; nothing reads the outcome)
      float* warm = reinterpret_cast<float*>(smem + L.warm_off);
      lse_rows(warm, 0, O, s_list, s_grp, p.K, 0, 1, lane, 32);
      pick(warm, nullptr, 0, false);
    }
    if (!PREP && !RAW && !is_drain) {
      // The fp32 gate rows to L2: the grid's converting threads together name
      // each 128-byte line once, so that the loads below, one stage ahead of
      // their use, wait for L2 and not for DRAM (fine-grained steps, T = 2001:
      // 346.5 -> 343 us).
      const long long row_lines = (p.d * 4LL + 127) / 128, lines = O * row_lines;
      constexpr int conv_threads = GC_THREADS - 192;
      for (long long i = static_cast<long long>(blockIdx.x) * conv_threads + (threadIdx.x - 192); i < lines;
           i += static_cast<long long>(gridDim.x) * conv_threads) {
        const int r = static_cast<int>(i / row_lines);
        const float* src = (r < p.E ? p.W_local + (size_t)r * p.d : p.W_global + (size_t)(r - p.E) * p.d) +
                           (i - r * row_lines) * 32;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(src));
      }
    }
    pdl_wait();  // the routing counters are cleared by the previous kernel (PREP)
    int stage = 0;
    uint32_t phase = 0;
    int acc_sel = 0;
    uint32_t uses0 = 0, uses1 = 0;
    bool ok = true;
    for (int tile = tile_first; tile < n_tiles; tile += tile_step) {
      if (is_drain) {
        float acc[NB][16];
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[b][j] = 0.0f;
        for (int seg = 0; seg < cnt; seg += GC_SEG) {
          const uint32_t uses = acc_sel ? uses1 : uses0;
          if (ok) ok = mbar_wait(smem_u32(&tfull[acc_sel]), uses & 1u, budget, abort_flag, &g_gate_error);
          if (ok) {
            tc_fence_after();
            const uint32_t t_acc = t_lane + acc_sel * GC_ACC_STRIDE;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
              uint32_t v0[16], v1[16], v2[16];
              tmem_ld16_nw(t_acc + b * 16, v0);
              tmem_ld16_nw(t_acc + n_pad + b * 16, v1);
              tmem_ld16_nw(t_acc + 2 * n_pad + b * 16, v2);
              tmem_wait();
#pragma unroll
              for (int j = 0; j < 16; ++j)
                acc[b][j] += (__uint_as_float(v0[j]) + __uint_as_float(v1[j])) + __uint_as_float(v2[j]);
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&tempty[acc_sel]));
          if (acc_sel) ++uses1;
          else ++uses0;
          acc_sel ^= 1;
        }
        bool decide_here = true;
        if (cs > 1) {
          // this row's partial logits go to the CTA that owns its decision;
          // the owner adds the cluster's partials in CTA order
          const int owner = row / rows_own;
          const int lrow = row - owner * rows_own;
          if (owner != rank) {
            decide_here = false;
            if (ok) {
              const uint32_t dst = map_to_rank(smem_u32(s_recv + (rank * rows_own + lrow) * L.rstride), owner);
              const uint32_t rb = map_to_rank(smem_u32(recvb), owner);
#pragma unroll
              for (int b = 0; b < NB; ++b)
                if (b * 16 < n_pad)
#pragma unroll
                  for (int j = 0; j < 16; j += 4)
                    st_async_v4(dst + (b * 16 + j) * 4, acc[b][j], acc[b][j + 1], acc[b][j + 2], acc[b][j + 3], rb);
            }
          } else {
            if (ok) ok = mbar_wait_cluster(smem_u32(recvb), 0, budget, abort_flag, &g_gate_error);
            if (ok) {
#pragma unroll
              for (int b = 0; b < NB; ++b)
                if (b * 16 < n_pad)
#pragma unroll
                  for (int j = 0; j < 16; ++j) {
                    float t = rank == 0 ? acc[b][j] : s_recv[lrow * L.rstride + b * 16 + j];
                    for (int c = 1; c < cs; ++c)
                      t += c == rank ? acc[b][j] : s_recv[(c * rows_own + lrow) * L.rstride + b * 16 + j];
                    acc[b][j] = t;
                  }
            }
          }
        }
        if (top1_regs) {
          const int tok = tile * GC_BM + row;
          if (decide_here && tok < p.T) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (j < O) acc[0][j] += s_bias[j];
            decide_top1(p, acc[0], tok);
          }
        } else if (decide_here) {
          float* Lrow = sLog + row * L.log_stride;
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int o = b * 16 + j;
              if (o < O) Lrow[o] = acc[b][j] + s_bias[o];
            }
          if (!nglob) {
            // one group: the row's own thread takes the whole decision
            const int tok = tile * GC_BM + row;
            lse_rows(sLog, L.log_stride, O, s_list, s_grp, 1, row, 1, 0, 1);
            if (tok < p.T) pick(Lrow, sIdx + row * p.k, tok, true);
          }
        }
      } else if (!PREP) {
        // split the fp32 gate rows of each stage into three bf16 terms, written
        // in the swizzled K-major layout of the B operand; without RAW the next
        // stage's pieces (8 columns of a row) are loaded while this one is written
        const int ct = threadIdx.x - 192;
        constexpr int ITEMS = ((RAW ? 16 * NB : GC_MAX_O) * 8 + 255) / 256;
        float v[ITEMS][8];
        auto load_items = [&](int kc) {
          if (RAW) return;
#pragma unroll
          for (int t = 0; t < ITEMS; ++t) {
            const int i = ct + 256 * t, r = i >> 3, c = kc * GC_BK + (i & 7) * 8;
            if (r < O && c < p.d) {
              load8((r < p.E ? p.W_local + (size_t)r * p.d : p.W_global + (size_t)(r - p.E) * p.d) + c, v[t]);
            } else {
#pragma unroll
              for (int u = 0; u < 8; ++u) v[t][u] = 0.0f;
            }
          }
        };
        load_items(kb_lo);
        for (int kc = 0; kc < cnt; ++kc) {
          // RAW: the stage's fp32 rows have landed, else: the stage is free
          if (ok)
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(RAW ? &full[stage] : &empty[stage]), RAW ? phase : phase ^ 1u,
                                                   budget, abort_flag, &g_gate_error));
          if (ok) {
            uint8_t* st = smem + stage * L.stage_bytes;
#pragma unroll
            for (int t = 0; t < ITEMS; ++t) {
              const int i = ct + 256 * t, r = i >> 3, ch = i & 7;
              if (r >= n_pad) break;
              if (RAW) {
                if (r < O) {
                  load8(reinterpret_cast<const float*>(st + L.raw_off) + r * GC_BK + ch * 8, v[t]);
                } else {
#pragma unroll
                  for (int u = 0; u < 8; ++u) v[t][u] = 0.0f;
                }
              }
              uint32_t t0[4], t1[4], t2[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) split3_pair(v[t][2 * u], v[t][2 * u + 1], t0[u], t1[u], t2[u]);
              const int off = L.w3_off + r * 128 + ((ch ^ (r & 7)) << 4);
              *reinterpret_cast<U4*>(st + off) = U4{t0[0], t0[1], t0[2], t0[3]};
              *reinterpret_cast<U4*>(st + off + n_pad * 128) = U4{t1[0], t1[1], t1[2], t1[3]};
              *reinterpret_cast<U4*>(st + off + 2 * n_pad * 128) = U4{t2[0], t2[1], t2[2], t2[3]};
            }
            // the tensor core reads these through the async proxy
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&conv[stage]));
          if (kc + 1 < cnt) load_items(kb_lo + kc + 1);
          if (++stage == S) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      // the tile's decisions over several groups: all worker warps (without
      // prepared rows the drain warps alone, while the others convert the next
      // tile's rows)
      const int n_dec = PREP ? GC_WORKERS : 128;
      const int first_row = rank * rows_own;
      if (nglob && (PREP || is_drain)) {
        asm volatile("bar.sync 2, %0;" ::"r"(n_dec) : "memory");
        lse_rows(sLog, L.log_stride, O, s_list, s_grp, p.K, first_row, rows_own, wt, n_dec);
        asm volatile("bar.sync 2, %0;" ::"r"(n_dec) : "memory");
        const int tok = tile * GC_BM + first_row + wt;
        const int r = first_row + wt;
        if (wt < rows_own && tok < p.T) pick(sLog + r * L.log_stride, sIdx + r * p.k, tok, true);
        // the rows are read before the next tile's logits replace them
        if (!p.route_counts) asm volatile("bar.sync 2, %0;" ::"r"(n_dec) : "memory");
      }
      if (p.route_counts) {
        asm volatile("bar.sync 1, %0;" ::"r"(GC_WORKERS) : "memory");
        route_tile_workers(p, tile, rank * rows_own, rows_own, sIdx + rank * rows_own * p.k, sTab, s_base, wt);
      }
    }
    tc_fence_before();
  }

  tc_fence_before();
  __syncthreads();
  // no CTA of the cluster leaves while partials to or from it are in flight
  if (cs > 1) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

// Stages that fit next to the logits, routing tables and received partials.
int gc_stages(int O, int k, int E, int cs, bool raw) {
  for (int s = GC_MAX_STAGES; s >= 2; --s)
    if (GcLayout(O, k, E, s, cs, raw).total + 1024 <= 232448) return s;
  return 0;
}

// CTAs per tile: d_model is split over a cluster of GC_CS when a tile has at
// least GC_SPLIT_MIN_NK stages and four stages with staged fp32 rows fit next to
// the received partials, which is so up to 32 gate rows (the split of more rows
// has not been measured since only up to 32 rows are staged), whatever the token
// count and whether the rows come prepared, so every call of one layer shape sums
// its logits in the same order.
// EC2MOE_GATE_SPLIT_MIN_STAGES=n in the environment moves the threshold
// (A/B comparisons; the split computes the same logits up to summation order).
int gc_cluster_size(int O, int k, int E, int d) {
  static const int min_nk = [] {
    const char* v = getenv("EC2MOE_GATE_SPLIT_MIN_STAGES");
    return v && atoi(v) > 0 ? atoi(v) : GC_SPLIT_MIN_NK;
  }();
  if ((d + GC_BK - 1) / GC_BK < min_nk) return 1;
  return GcLayout(O, k, E, 4, GC_CS, true).warm_off + 1024 <= 232448 ? GC_CS : 1;
}

// CTAs the gate kernel launches (cs > 1: a cluster per tile, run in waves
// when they exceed the SMs; cs = 1: persistent, at most one per SM).
int gc_blocks(int T, int cs) {
  const int n_tiles = (T + GC_BM - 1) / GC_BM;
  if (cs > 1) return n_tiles * cs;
  return n_tiles < sm_count() ? n_tiles : sm_count();
}

template <int NB, bool PREP>
cudaError_t launch_gate_tc_nb(const KParams& p, int stages, int cs, cudaStream_t s, const CUtensorMap& mX,
                              const CUtensorMap& mW, const CUtensorMap& mWg) {
  const int O = p.E + (p.K == 1 ? 0 : p.K);
  GcParams gp;
  gp.kp = p;
  gp.n_pad = (O + 15) / 16 * 16;
  gp.stages = stages;
  gp.cs = cs;
  gp.timeout = default_timeout_cycles();
  const int smem = GcLayout(O, p.k, p.E, stages, cs, gc_raw(NB, PREP)).total + 1024;
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(gate_tc_kernel<NB, PREP>), smem);
  if (e != cudaSuccess) return e;
  const int blocks = gc_blocks(p.T, cs);
  const int threads = PREP ? GC_THREADS : GC_THREADS + 32;
  if (cs == 1)
    return launch_kernel(gate_tc_kernel<NB, PREP>, dim3(blocks), dim3(threads), (size_t)smem, s, mX, mW, mWg, gp);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = next_launch_pdl() ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gate_tc_kernel<NB, PREP>, mX, mW, mWg, gp);
}

template <bool PREP>
cudaError_t launch_gate_tc(const KParams& p, int stages, int cs, cudaStream_t s, const CUtensorMap& mX,
                           const CUtensorMap& mW, const CUtensorMap& mWg) {
  const int O = p.E + (p.K == 1 ? 0 : p.K);
  // NB = accumulator blocks of 16 gate rows a drain thread keeps; 3 and 4
  // run as 5 (the extra blocks read allocated TMEM columns past the gate rows
  // and are never used), which keeps the number of kernel variants small.
  switch ((O + 15) / 16) {
    case 1: return launch_gate_tc_nb<1, PREP>(p, stages, cs, s, mX, mW, mWg);
    case 2: return launch_gate_tc_nb<2, PREP>(p, stages, cs, s, mX, mW, mWg);
    default: return launch_gate_tc_nb<5, PREP>(p, stages, cs, s, mX, mW, mWg);
  }
}

}  // namespace

cudaError_t launch_gate_tensor(const GateArgs& a, KParams p, int O, bool bf16, cudaStream_t s, bool* routed, int* held_sms,
                               bool* handled) {
  *handled = false;
  cudaError_t e = cudaSuccess;
  // Tensor-core gate (bf16 activations, up to 80 gate rows).  With a
  // workspace for the prepared split rows (layer path) a small kernel first
  // splits the gate rows and clears the routing counters; without one the
  // gate kernel splits them itself.
  static const bool simt_only = [] {
    const char* v = getenv("EC2MOE_GATE_SIMT");
    return v && atoi(v) > 0;
  }();
  const bool w_aligned = (reinterpret_cast<uintptr_t>(a.W_local) % 16 == 0) &&
                         (a.K == 1 || reinterpret_cast<uintptr_t>(a.W_global) % 16 == 0);
  if (bf16 && !simt_only && O <= GC_MAX_O && a.d % 8 == 0 && a.T > 0 && w_aligned) {
    const bool prep = a.w_split != nullptr;
    const int n_pad = (O + 15) / 16 * 16;
    const int cs = gc_cluster_size(O, a.k, a.E, a.d);
    const bool raw = gc_raw(n_pad / 16, prep);
    const int stages = gc_stages(O, a.k, a.E, cs, raw);
    CUtensorMap mX, mW, mWg;
    bool maps = stages >= 2 && make_tensor_map_bf16(&mX, a.X, a.T, a.d, GC_BM);
    if (prep) {
      maps = maps && make_tensor_map_bf16(&mW, a.w_split, 3LL * n_pad, a.d, 3 * n_pad);
      mWg = mW;
    } else if (raw) {
      maps = maps && make_tensor_map_f32(&mW, a.W_local, a.E, a.d, a.E);
      if (maps && a.K > 1) maps = make_tensor_map_f32(&mWg, a.W_global, a.K, a.d, a.K);
      else mWg = mW;
    } else if (maps) {
      mW = mWg = mX;  // not read: the kernel loads the gate rows to registers
    }
    if (maps) {
      *handled = true;
      const bool route = a.route_counts && a.route_rel;
      if (route) {
        p.route_counts = a.route_counts;
        p.route_rel = a.route_rel;
        if (!prep) {
          e = cudaMemsetAsync(a.route_counts, 0, sizeof(int32_t) * a.E, s);
          if (e != cudaSuccess) return e;
        }
        if (routed) *routed = true;
      }
      if (prep) {
        KernelScope ks("gate_prep", s);
        const long long items = (long long)n_pad * (a.d / 8);
        e = launch_kernel(gate_split_kernel, dim3((unsigned)((items + 255) / 256)), dim3(256), 0, s, a.W_local,
                          a.W_global, a.E, a.K, a.d, n_pad, static_cast<__nv_bfloat16*>(a.w_split),
                          route ? a.route_counts : nullptr);
        if (e != cudaSuccess) return e;
      }
      KernelScope ks("gate_topk", s);
      if (held_sms) {  // one CTA per SM (the kernel's shared memory allows no second)
        const int b = gc_blocks(a.T, cs);
        *held_sms = b < sm_count() ? b : sm_count();
      }
      e = prep ? launch_gate_tc<true>(p, stages, cs, s, mX, mW, mWg)
               : launch_gate_tc<false>(p, stages, cs, s, mX, mW, mWg);
      if (e != cudaSuccess) return e;
      return cudaGetLastError();
    }
  }
  return cudaSuccess;
}

}  // namespace gatek

using namespace gatek;

size_t gate_split_bytes(int E, int K, int d, bool bf16) {
  const int O = E + (K == 1 ? 0 : K);
  if (!bf16 || O > GC_MAX_O || d % 8 != 0) return 0;
  return (size_t)3 * ((O + 15) / 16 * 16) * d * 2;
}

cudaError_t read_gate_error(unsigned int* word) {
  unsigned int zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(word, g_gate_error, sizeof(unsigned int));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(g_gate_error, &zero, sizeof(unsigned int));
}

}  // namespace ec2moe
