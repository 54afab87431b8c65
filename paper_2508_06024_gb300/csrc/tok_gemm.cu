// Grouped bf16 GEMM with the weights on the MMA's M side and the tokens on
// its N side, on CTA pairs (tcgen05.mma.cta_group::2), for expert groups of a
// few dozen to a few hundred rows (Eq. 1, each E_i an FFN):
//
//   C_g^T = B_g A_g^T : 256 weight rows of group g fill the pair's M side
//                       (128 per CTA), the group's token rows its N side.
//
// With tokens on M a group is padded to whole 128- or 256-row tiles (259 rows
// run as 384).  N, in contrast, is any multiple of 32, so a group's rows are
// spread evenly over tiles of at most 256 and padded to the next 32 of each.
// What bounds it then: the operand bytes an SM takes from L2, 16 KB of weights
// and n / 2 token rows per 64-column block and CTA (~100 GB/s per SM
// measured), and under long runs the power cap.  Tiles of up to 512 tokens on
// one weight tile (two MMAs per step, accumulators not double-buffered) and a
// deeper ring for the weights than for the tokens were slower (Mixtral-shaped
// layer, T = 777: 533 and 517 us against 492).  Measured times against the
// tokens-on-M kernels are at the rule below (tok_gemm_preferred).
//
// A unit is (group, 256 weight rows, run of tokens).  Pairs take units
// round-robin, whole token tiles first; the tiles of the last, partial wave
// are cut along the tokens so that every pair gets a piece.  SwiGLU tiles
// stack 64 W1 rows over the same 64 W3 rows in each CTA; the epilogue warps of
// a column's two halves trade values through shared memory.
//
// Roles: warp 0 loads, warp 1 of the even CTA issues the pair's MMAs (both
// walk their loops as a whole warp, one elected lane issues: as one lane's
// divergent loop with an inner loop the issue made the kernel 20-40% slower),
// warps 2..17 read the accumulators (TMEM lane quadrant = warp % 4, lane =
// weight row, column = token), transpose 32 x 32 blocks through shared memory
// and store row segments.  Barriers, bounded waits and the end after an abort
// are those of the pair GEMM in tc_gemm.cu.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace ec2moe {

// bit 0: a bounded wait timed out; bit 1: a group range (offsets) or a
// scatter destination (perm) outside the rows of the call was skipped
__device__ unsigned int g_tok_error;

namespace {

using namespace tc;

constexpr int TG_M = 128;    // weight rows per CTA (MMA M = 256 over the pair)
constexpr int TG_BK = 64;    // K per stage: one 128-byte swizzle row of bf16
constexpr int TG_UK = 16;    // K of one tcgen05.mma kind::f16
constexpr int TG_NT = 256;    // most tokens of a tile (MMA N)
constexpr int TG_STAGES = 6;
constexpr int TG_EPI_WARPS = 16;  // four per TMEM lane quadrant
constexpr int TG_THREADS = 64 + 32 * TG_EPI_WARPS;
constexpr int TG_MAX_GROUPS = 132;
constexpr int TG_MAX_CUT = 4;     // pieces of a tile of the last wave
constexpr int TG_W_BYTES = TG_M * TG_BK * 2;       // 16 KB of weights per stage and CTA
constexpr int TG_X_BYTES = TG_NT / 2 * TG_BK * 2;  // 16 KB of tokens
constexpr int TG_STAGE_BYTES = TG_W_BYTES + TG_X_BYTES;
constexpr int TG_STG_BYTES = 32 * 64;         // per epilogue warp: 32 tokens x 32 columns bf16
constexpr int TG_OFF_STG = TG_STAGES * TG_STAGE_BYTES;
constexpr int TG_OFF_BARS = TG_OFF_STG + TG_EPI_WARPS * TG_STG_BYTES;
constexpr int TG_N_BARS = 2 * TG_STAGES + 5;  // full, empty, accumulator full / free (2 each), drain
constexpr int TG_OFF_SLOT = TG_OFF_BARS + TG_N_BARS * 8;  // TMEM address, abort flag
constexpr int TG_OFF_PREFIX = TG_OFF_SLOT + 16;
constexpr int TG_OFF_GROUPS = (TG_OFF_PREFIX + (TG_MAX_GROUPS + 1) * 4 + 15) / 16 * 16;
constexpr int TG_SMEM = 1024 + TG_OFF_GROUPS + TG_MAX_GROUPS * 8;
static_assert(TG_OFF_BARS % 8 == 0 && TG_SMEM <= 232448, "shared memory per CTA");

struct TgParams {
  const int32_t* offsets;
  int G, M, a_shared;
  long long a_row_base, out_row_base;
  int N, K, b_group_rows;
  __nv_bfloat16* out;
  long long ldo;
  const int32_t* perm;
  const float* scale;
  int n_mblk;        // weight blocks per group
  long long timeout;
  long long row_limit;  // rows of the call: group ranges and scatter destinations lie in [0, row_limit)
  // groups [G_main, G): shared experts (GemmArgs::sh_*)
  int G_main, sh_rows;
  long long sh_row0, sh_a_row;
  __nv_bfloat16* sh_out;
};

// Token boxes of 16, 32, 64 and 128 rows, weight boxes (W2: SwiGLU's W3).
struct TgMaps {
  CUtensorMap x[4];
  CUtensorMap w, w2;
  CUtensorMap ws, w2s;  // shared experts'
};

// A group's rows; its token tiles spread them evenly over the fewest tiles of
// at most TG_NT rows, rounded up to 32 (the last one holds fewer).
struct TgGroup {
  int row0, rows;
};

struct TgUnit {
  int g, mb;   // group, weight block
  int t0, tn;  // first token within the group, tokens (<= 0: nothing to do)
  int n;       // MMA N: tn rounded up to 32 (M = 256 wants a multiple of 32)
};

// The unit list of the call: `full` whole tiles, then the remaining tiles in
// `cut` pieces each.
struct TgList {
  int full, cut, units;
};
__device__ __forceinline__ TgList unit_list(int tiles, int pairs) {
  TgList l;
  l.full = tiles / pairs * pairs;
  const int tail = tiles - l.full;
  l.cut = tail > 0 ? pairs / tail : 1;
  if (l.cut > TG_MAX_CUT) l.cut = TG_MAX_CUT;
  l.units = l.full + tail * l.cut;
  return l;
}
__device__ __forceinline__ TgUnit unit_at(int u, const TgList& l, const int* tile_prefix, const TgGroup* groups,
                                          int& cursor) {
  int tile = u, piece = 0, pieces = 1;
  if (u >= l.full) {
    tile = l.full + (u - l.full) / l.cut;
    piece = (u - l.full) % l.cut;
    pieces = l.cut;
  }
  while (tile >= tile_prefix[cursor + 1]) ++cursor;
  TgUnit x;
  x.g = cursor;
  const TgGroup gr = groups[x.g];
  const int ntile = (gr.rows + TG_NT - 1) / TG_NT;
  const int size = ntile == 1 ? gr.rows : ((gr.rows + ntile - 1) / ntile + 31) / 32 * 32;
  const int rem = tile - tile_prefix[x.g];
  x.mb = ntile == 1 ? rem : rem / ntile;
  x.t0 = (rem - x.mb * ntile) * size;
  x.tn = gr.rows - x.t0 < size ? gr.rows - x.t0 : size;
  if (pieces > 1) {
    const int ps = ((x.tn + pieces - 1) / pieces + 31) / 32 * 32;
    x.t0 += piece * ps;
    x.tn -= piece * ps;
    if (x.tn > ps) x.tn = ps;
  }
  x.n = (x.tn + 31) / 32 * 32;
  return x;
}

template <int EPI>
__global__ void __launch_bounds__(TG_THREADS, 1)
    tok_gemm_kernel(const __grid_constant__ TgMaps tm, const TgParams p) {
  constexpr bool GLU = EPI == EPI_SWIGLU;
  constexpr int COLS = GLU ? TG_M / 2 : TG_M;  // output columns per CTA and weight block
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + TG_OFF_BARS);
  uint64_t* empty = full + TG_STAGES;
  uint64_t* tfull = empty + TG_STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + TG_OFF_SLOT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* tile_prefix = reinterpret_cast<int*>(smem + TG_OFF_PREFIX);
  TgGroup* groups = reinterpret_cast<TgGroup*>(smem + TG_OFF_GROUPS);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair_id = static_cast<int>(cluster_id_x());
  const int pairs = static_cast<int>(cluster_count_x());
  // Barrier set-up, TMEM allocation and descriptor prefetch overlap the
  // previous kernel; everything that reads its results comes after pdl_wait.
  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < TG_STAGES; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tfull[a]), 1);
      mbar_init(smem_u32(&tempty[a]), 2 * TG_EPI_WARPS);
    }
    mbar_init(smem_u32(drain), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    pdl_wait();
    warp_exclusive_scan<(TG_MAX_GROUPS + 31) / 32>(
        p.G, lane,
        [&](int g) {
          int r0 = g * p.M, mg = p.M;
          if (g >= p.G_main) {
            r0 = static_cast<int>(p.sh_row0) + (g - p.G_main) * p.sh_rows;
            mg = p.sh_rows;
          } else if (p.offsets) {
            r0 = p.offsets[g];
            mg = p.offsets[g + 1] - r0;
            if (r0 < 0 || mg < 0 || static_cast<long long>(r0) + mg > p.row_limit) {
              // not a range of this call's rows: the group is skipped
              atomicOr(&g_tok_error, 2u);
              r0 = 0;
              mg = 0;
            }
          }
          groups[g] = TgGroup{r0, mg};
          return (mg + TG_NT - 1) / TG_NT * p.n_mblk;
        },
        tile_prefix);
  }
  if (warp == 0 && lane == 0) {
    for (int i = 0; i < 4; ++i) tma_prefetch_desc(&tm.x[i]);
    tma_prefetch_desc(&tm.w);
    if (GLU) tma_prefetch_desc(&tm.w2);
  }
  if (warp == 1) {
    // the pair's columns, allocated by one warp of each CTA together
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  // both CTAs' barriers are initialised before either arrives remotely
  cluster_sync_all();
  tc_fence_after();
  pdl_wait();
  const uint32_t tmem_base = *tmem_slot;
  const TgList list = unit_list(tile_prefix[p.G], pairs);
  const int num_kb = (p.K + TG_BK - 1) / TG_BK;
  const long long budget = p.timeout;

  if (warp == 0) {
    // ---------------------------------------------------------------- producer
    {
      const bool leader = elect_one();
      int stage = 0, cursor = 0;
      uint32_t phase = 0;
      uint32_t issued = 0;  // bit s: stage s holds a copy the consumer has not released
      uint32_t issued_phase = 0;
      bool ok = true;
      for (int u = pair_id; u < list.units && ok; u += pairs) {
        const TgUnit x = unit_at(u, list, tile_prefix, groups, cursor);
        if (x.tn <= 0) continue;
        // this CTA's tokens: one run of n / 2 rows, as two boxes at most (a box
        // costs the copy engine tens of clocks whatever its height)
        const int run = x.n / 2;
        const int b1 = 31 - __clz(run);
        const int rest = run - (1 << b1);
        const int b2 = rest > 0 ? (rest <= 16 ? 4 : 32 - __clz(rest - 1)) : -1;
        const uint32_t bytes = TG_W_BYTES + ((1 << b1) + (b2 >= 0 ? 1 << b2 : 0)) * (TG_BK * 2);
        const CUtensorMap* x1 = &tm.x[b1 - 4];
        const CUtensorMap* x2 = &tm.x[b2 >= 0 ? b2 - 4 : 0];
        const bool sh = x.g >= p.G_main;
        const int x_row = (sh && p.sh_a_row >= 0
                               ? static_cast<int>(p.sh_a_row)
                               : static_cast<int>(p.a_row_base) + (p.offsets || sh || !p.a_shared ? groups[x.g].row0 : 0)) +
                          x.t0 + static_cast<int>(rank) * run;
        const int w_row = (sh ? x.g - p.G_main : x.g) * p.b_group_rows + (x.mb * 2 + static_cast<int>(rank)) * COLS;
        const CUtensorMap* mw = sh ? &tm.ws : &tm.w;
        const CUtensorMap* mw2 = sh ? &tm.w2s : &tm.w2;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!__all_sync(0xffffffffu,
                          mbar_wait(smem_u32(&empty[stage]), phase ^ 1u, budget, abort_flag, &g_tok_error))) {
            ok = false;
            break;
          }
          // both CTAs' copies complete on the even CTA's full barrier
          const uint32_t fb = smem_u32(&full[stage]);
          if (leader && rank == 0) mbar_expect_tx(fb, 2 * bytes);
          const uint32_t fb0 = rank == 0 ? fb : map_to_rank(fb, 0);
          const uint32_t sw = smem_u32(smem) + stage * TG_STAGE_BYTES;
          if (leader) {
            tma_load_2d_to_pair_bar(sw, mw, kb * TG_BK, w_row, fb0);
            if (GLU) tma_load_2d_to_pair_bar(sw + TG_W_BYTES / 2, mw2, kb * TG_BK, w_row, fb0);
            tma_load_2d_to_pair_bar(sw + TG_W_BYTES, x1, kb * TG_BK, x_row, fb0);
            if (b2 >= 0)
              tma_load_2d_to_pair_bar(sw + TG_W_BYTES + ((TG_BK * 2) << b1), x2, kb * TG_BK, x_row + (1 << b1), fb0);
          }
          issued |= 1u << stage;
          issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
          if (++stage == TG_STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok || *abort_flag) {
        // Let every copy this CTA started land before shared memory is released.
        if (rank != 0) {
          // its copies complete on the even CTA's barriers: wait a fixed time
          if (issued) {
            const unsigned long long t0 = globaltimer_ns();
            while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
          }
        } else {
          for (int s = 0; s < TG_STAGES; ++s)
            if (issued & (1u << s)) mbar_drain(smem_u32(&full[s]), (issued_phase >> s) & 1u, DRAIN_CYCLES);
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---------------------------------------------------------------- MMA issuer
      const bool leader = elect_one();
      const uint64_t d0 = sdesc_sw128(smem_u32(smem));
      const uint32_t full0 = smem_u32(&full[0]), empty0 = smem_u32(&empty[0]);
      int stage = 0, cursor = 0;
      uint32_t phase = 0;
      uint32_t used = 0;  // accumulators handed out so far: accumulator used & 1
      bool ok = true, any = false;
      for (int u = pair_id; u < list.units && ok; u += pairs) {
        const TgUnit x = unit_at(u, list, tile_prefix, groups, cursor);
        if (x.tn <= 0) continue;
        const uint32_t n = __shfl_sync(0xffffffffu, x.n, 0);
        const uint32_t idesc = idesc_bf16(2 * TG_M, n);
        const uint32_t acc = tmem_base + (used & 1) * TG_NT;
        // both CTAs' epilogue warps release an accumulator on this barrier
        ok = __all_sync(0xffffffffu, mbar_wait_cluster(smem_u32(&tempty[used & 1]), ((used >> 1) & 1u) ^ 1u, budget,
                                                       abort_flag, &g_tok_error));
        for (int kb = 0; kb < num_kb && ok; ++kb) {
          if (!__all_sync(0xffffffffu, mbar_wait(full0 + 8u * stage, phase, budget, abort_flag, &g_tok_error))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t dw = d0 + static_cast<uint64_t>(stage) * (TG_STAGE_BYTES >> 4);
          const uint64_t dx = dw + (TG_W_BYTES >> 4);
          if (leader) {
            umma_bf16_pair(acc, dw, dx, idesc, kb ? 1u : 0u);
#pragma unroll
            for (int kk = 1; kk < TG_BK / TG_UK; ++kk) umma_bf16_pair(acc, dw + 2 * kk, dx + 2 * kk, idesc, 1u);
            umma_commit_pair_mc(empty0 + 8u * stage);
          }
          any = true;
          if (++stage == TG_STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        if (leader) umma_commit_pair_mc(smem_u32(&tfull[used & 1]));
        ++used;
      }
      if ((!ok || *abort_flag) && any && leader) {
        // All MMAs issued so far must finish before TMEM is freed.
        umma_commit_pair(smem_u32(drain));
        mbar_drain(smem_u32(drain), 0, DRAIN_CYCLES);
      }
    }
  } else {
    // ---------------------------------------------------------------- epilogue
    const int q = warp & 3;            // TMEM lane quadrant this warp may access
    const int part = (warp - 2) >> 2;  // which 32-token blocks of an accumulator
    const uint32_t t_row = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
    uint8_t* stg = smem + TG_OFF_STG + (warp - 2) * TG_STG_BYTES;
    // SwiGLU: lanes 0-63 hold W1's values of 64 columns, lanes 64-127 W3's of
    // the same; the warps of quadrants q and q + 2 trade halves of a block, and
    // each finishes 16 of its 32 tokens.
    constexpr int TOK = GLU ? 16 : 32;     // tokens of a block this warp finishes
    const int hi = GLU ? q >> 1 : 0;       // SwiGLU: which half of the block
    uint8_t* stg_other = smem + TG_OFF_STG + ((warp - 2) ^ 2) * TG_STG_BYTES;
    const int bar_id = 1 + part * 2 + (q & 1);
    (void)stg_other;
    uint32_t used = 0;
    int cursor = 0;
    bool ok = true;
    for (int u = pair_id; u < list.units && ok; u += pairs) {
      const TgUnit x = unit_at(u, list, tile_prefix, groups, cursor);
      if (x.tn <= 0) continue;
      const int col0 = (x.mb * 2 + static_cast<int>(rank)) * COLS + (GLU ? q & 1 : q) * 32;
      const bool sh = EPI == EPI_SCATTER && x.g >= p.G_main;  // stored to sh_out, unscaled
      const long long base = (sh ? -p.sh_row0 : p.out_row_base) + groups[x.g].row0 + x.t0;
      __nv_bfloat16* out = sh ? p.sh_out : p.out;
      {
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&tfull[used & 1]), (used >> 1) & 1u, budget, abort_flag,
                                               &g_tok_error));
        if (GLU) {
          // the two warps meet at named barriers below: agree on the outcome
          uint32_t both;
          asm volatile(
              "{\n .reg .pred p, r;\n setp.ne.u32 p, %1, 0;\n"
              " bar.red.and.pred r, %2, 64, p;\n selp.u32 %0, 1, 0, r;\n}"
              : "=r"(both)
              : "r"(ok ? 1u : 0u), "r"(bar_id)
              : "memory");
          ok = both != 0;
        }
        if (!ok) break;
        tc_fence_after();
        const uint32_t t_acc = t_row + (used & 1) * TG_NT;
        for (int b = part * 32; b < x.n; b += 32 * (TG_EPI_WARPS / 4)) {
          // lane t's token of the block
          bool valid = b + lane < x.tn;
          long long dest = base + b + lane;
          float sc = 1.0f;
          if (EPI == EPI_SCATTER && !sh && valid) {
            const long long o = dest;
            dest = p.perm ? p.perm[o] : o;
            if (dest < 0 || dest >= p.row_limit) {
              atomicOr(&g_tok_error, 2u);
              valid = false;
              dest = 0;
            } else if (p.scale) {
              sc = p.scale[dest];
            }
          }
          const unsigned vmask = __ballot_sync(0xffffffffu, valid);
          if (vmask == 0) continue;  // the same for both warps of a SwiGLU pair
          uint32_t r[32];
          tmem_ld32_nw(t_acc + b, r);
          tmem_wait();
          if (GLU) {
            float* xs = reinterpret_cast<float*>(stg) + lane;
            const float* xo = reinterpret_cast<const float*>(stg_other) + lane;
#pragma unroll
            for (int j = 0; j < 16; ++j) xs[j * 32] = __uint_as_float(hi ? r[j] : r[16 + j]);
            asm volatile("bar.sync %0, 64;" ::"r"(bar_id) : "memory");
            float o[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) o[j] = xo[j * 32];
            asm volatile("bar.sync %0, 64;" ::"r"(bar_id) : "memory");
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float a = hi ? o[j] : __uint_as_float(r[j]);
              const float g = hi ? __uint_as_float(r[16 + j]) : o[j];
              *reinterpret_cast<__nv_bfloat16*>(stg + j * 64 + lane * 2) = __float2bfloat16_rn(silu_bf16out(a) * g);
            }
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              float v = __uint_as_float(r[j]);
              if (EPI == EPI_GELU) v = gelu_bf16out(v);
              if (EPI == EPI_SCATTER) v *= __shfl_sync(0xffffffffu, sc, j);
              *reinterpret_cast<__nv_bfloat16*>(stg + j * 64 + lane * 2) = __float2bfloat16_rn(v);
            }
          }
          __syncwarp();
          // four lanes per token, 16 bytes each
#pragma unroll
          for (int i = 0; i < TOK / 8; ++i) {
            const int ts = i * 8 + (lane >> 2), seg = lane & 3;
            const int t = hi * 16 + ts;
            const U4 v = *reinterpret_cast<const U4*>(stg + ts * 64 + seg * 16);
            const long long drow = __shfl_sync(0xffffffffu, dest, t);
            const int col = col0 + seg * 8;
            if ((vmask >> t & 1u) && col < p.N) *reinterpret_cast<U4*>(out + drow * p.ldo + col) = v;
          }
          __syncwarp();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(map_to_rank(smem_u32(&tempty[used & 1]), 0));
        ++used;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  // the even CTA's MMAs write both CTAs' TMEM; neither releases its columns
  // before both are done with them
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

template <int EPI>
cudaError_t launch_epi(const GemmArgs& a, TgParams p, cudaStream_t s) {
  constexpr bool GLU = EPI == EPI_SWIGLU;
  auto* kernel = tok_gemm_kernel<EPI>;
  const void* kfn = reinterpret_cast<const void*>(kernel);
  cudaError_t e = ensure_smem_attr(kfn, TG_SMEM);
  if (e != cudaSuccess) return e;
  TgMaps tm;
  for (int i = 0; i < 4; ++i)
    if (!make_tensor_map_bf16(&tm.x[i], a.A, a.a_rows, a.K, 16 << i)) return cudaErrorInvalidValue;
  if (!make_tensor_map_bf16(&tm.w, a.B, a.b_rows, a.K, GLU ? TG_M / 2 : TG_M)) return cudaErrorInvalidValue;
  tm.w2 = tm.w;
  if (GLU && !make_tensor_map_bf16(&tm.w2, a.B2, a.b_rows, a.K, TG_M / 2)) return cudaErrorInvalidValue;
  tm.ws = tm.w;
  tm.w2s = tm.w2;
  if (a.sh_groups > 0) {
    const long long rows = (long long)a.sh_groups * a.b_group_rows;
    if (!make_tensor_map_bf16(&tm.ws, a.sh_B, rows, a.K, GLU ? TG_M / 2 : TG_M)) return cudaErrorInvalidValue;
    if (GLU && !make_tensor_map_bf16(&tm.w2s, a.sh_B2, rows, a.K, TG_M / 2)) return cudaErrorInvalidValue;
  }
  const int cols = GLU ? TG_M : 2 * TG_M;  // output columns of a pair's weight block
  p.n_mblk = (a.N + cols - 1) / cols;
  int clusters = max_clusters(kfn, TG_THREADS, TG_SMEM, 2);
  if (clusters < 1) return cudaErrorInvalidConfiguration;
  const long long units = (a.max_rows / 32 + p.G) * p.n_mblk;  // pieces hold 32 rows or more, but for each group's last
  if (units < clusters) clusters = static_cast<int>(units < 1 ? 1 : units);
  KernelScope ks(a.name ? a.name : "gemm_tok", s);
  return launch_cluster(kernel, clusters, 2, TG_THREADS, (size_t)TG_SMEM, s, tm, p);
}

}  // namespace

bool gemm_tok_supported(const GemmArgs& a, int epi) {
  if (epi != EPI_STORE && epi != EPI_GELU && epi != EPI_SWIGLU && epi != EPI_SCATTER) return false;
  if (a.G < 1 || a.G + a.sh_groups > TG_MAX_GROUPS || a.N % 32 != 0 || a.K % 8 != 0) return false;
  return true;
}

// Where this orientation is the faster one (both sides measured on one GPU,
// us; Mixtral-shaped d = 4096, d_ff = 14336, 6 experts, and fine-grained d =
// 2048, d_ff = 1408, 32 experts; rows per expert in brackets):
//   up    Mixtral [85] 213 -> 219, [128] 229 -> 223, [171] 259 -> 229, [259] 298 -> 271, [512] 513 -> 450,
//         [1024] 825 -> 798; fine [75] 72 -> 74, [187] 88 -> 86, [375] 119 -> 112, [1500] 323 -> 317, [3072] 596 -> 637
//   down  Mixtral [128] 122 -> 143, [213] 145 -> 149, [259] 184 -> 150, [512] 323 -> 260, [1024] 439 -> 419;
//         fine (K = 1408) [375] 67 -> 65, [750] 98 -> 99
//   Switch-shaped up, K = 768 [341] 27 -> 31
// So: a K of 2048 or more (shorter main loops do not cover a tile's start), up
// projections from 128 expected rows per group, down projections, whose N
// leaves few weight blocks, from 240, up to 1536 rows (beyond, the padding no
// longer matters and the pair GEMM overlaps its epilogue better), and at least
// one tile for every pair.
bool tok_gemm_preferred(const GemmArgs& a, int epi) {
  if (!gemm_tok_supported(a, epi) || a.K < 2048) return false;
  const bool up = epi == EPI_GELU || epi == EPI_SWIGLU;
  const long long groups = a.g_active > 0 ? a.g_active : a.G;
  const long long rows = a.max_rows / groups;
  if (rows < (up ? 128 : 240) || rows > 1536) return false;
  const int cols = epi == EPI_SWIGLU ? TG_M : 2 * TG_M;
  return (rows + TG_NT - 1) / TG_NT * groups * ((a.N + cols - 1) / cols) >= sm_count() / 2;
}

cudaError_t launch_gemm_tok(const GemmArgs& a, int epi, cudaStream_t s) {
  if (!gemm_tok_supported(a, epi)) return cudaErrorInvalidValue;
  TgParams p{};
  p.offsets = a.offsets;
  p.G = a.G + a.sh_groups;
  p.G_main = a.G;
  p.sh_rows = a.sh_rows;
  p.sh_row0 = a.sh_row0;
  p.sh_a_row = a.sh_groups > 0 ? a.sh_a_row : -1;
  p.sh_out = static_cast<__nv_bfloat16*>(a.sh_out);
  p.M = a.M;
  p.a_shared = a.a_shared;
  p.a_row_base = a.a_row_base;
  p.out_row_base = a.out_row_base;
  p.N = a.N;
  p.K = a.K;
  p.b_group_rows = a.b_group_rows;
  p.out = static_cast<__nv_bfloat16*>(a.out);
  p.ldo = a.ldo;
  p.perm = a.perm;
  p.scale = a.scale;
  p.timeout = a.timeout_cycles;
  p.row_limit = a.row_limit > 0 ? a.row_limit : a.max_rows > 0 ? a.max_rows : (1LL << 62);
  cudaError_t e;
  switch (epi) {
    case EPI_GELU: e = launch_epi<EPI_GELU>(a, p, s); break;
    case EPI_SWIGLU: e = launch_epi<EPI_SWIGLU>(a, p, s); break;
    case EPI_SCATTER: e = launch_epi<EPI_SCATTER>(a, p, s); break;
    default: e = launch_epi<EPI_STORE>(a, p, s); break;
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

cudaError_t read_tok_error(unsigned int* word) {
  unsigned int zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(word, g_tok_error, sizeof(unsigned int));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(g_tok_error, &zero, sizeof(unsigned int));
}

}  // namespace ec2moe
