// Grouped fp32 GEMM on the sm_103a tensor cores, for layers stored in fp32:
// C_g = A_g B_g^T with A_g [M_g, K] and B_g [N, K] (rows of a weight stored
// [out, in]), the same groups and epilogues as the bf16 path.
//
// The tensor cores have no mode that keeps full fp32 products (kind::tf32
// rounds the operands to 10 mantissa bits), so every fp32 operand is split
// into three bf16 terms, x = x0 + x1 + x2 (x0 = bf16(x), x1 = bf16(x - x0),
// x2 = bf16(x - x0 - x1); both differences are exact in fp32 and the rest is
// below 2^-26 |x|).  A product of two bf16 terms is exact in fp32, and
//   x w = x0 w0 + (x0 w1 + x1 w0) + (x0 w2 + x1 w1 + x2 w0) + rest,
// with a rest of at most about 2^-25 |x w|, under one fp32 rounding of the
// product.  bf16 ends 16 binary places before fp32, and the tensor core reads
// subnormal operands as 0, so operands are scaled by 2^24 first (exact), which
// keeps that true down to fp32's smallest numbers.  What the scaling makes
// overflow (operands above 2^104, sums above 2^80) is computed again, see below.
//
// The tensor core adds into its fp32 accumulator without rounding to
// nearest, so sums are kept short: x0 w0 accumulates in one TMEM accumulator
// and the five smaller products in another, both only over a segment of 128
// columns of K; the warps then add the two and the segment's sum to fp32
// registers.  Against 64-bit results this is closer than the sequential fp32
// FMA sums of a CUDA-core kernel: relative error of a layer's Y 5.0e-7
// against 1.3e-6 (d = 768, d_ff = 3072), 4.4e-7 against 8.7e-7 (512, 1024).
//
// What bounds it: a chain of nearly equal parts per 64-column block.  A pass of
// a layer (12 experts, 1024 rows, 768 x 3072; the two expert GEMMs are 4/5 of
// it) takes 149 us.  When it took 155, copies of the kernel without the MMAs took
// 128, with half of them 133, without B's split and stores 142, without the loads
// 142, without A's stores 150, and with A's terms in shared memory as well, where
// the MMAs then read twice as much, 162.  CUDA-core tiles took 426 us for
// expert_up alone and 758 for expert_down.
//
// One persistent CTA of 16 warps per SM (a 17th warp for the MMAs alone would
// cut the registers per thread from 128 to 96).  Every warp loads A and B blocks
// as fp32, one block ahead in registers, and writes the three terms: of A into
// tensor memory (a thread's row is its TMEM lane; a warp takes a quarter of the
// block's columns), of B into the swizzled K-major stage (16 bytes per lane,
// whole 256-byte row pieces).  It drains the finished segment's accumulators
// (TMEM lanes 32 (w % 4) .. +31, a quarter of the columns) and at the end of the
// tile applies the epilogue.  Warp 0 also issues the MMAs.
// Two stages, so a block is loaded and split while the previous one multiplies;
// two pairs of accumulators for 64-wide tiles, one for 128-wide ones (the A
// stages take the other pair's columns).  Every wait is bounded; a timeout sets
// the error word and the CTA ends after its MMAs in flight.  A comes by plain
// loads: the kernel before may still write it when this one starts, which the
// read-only path does not allow.  The waits are too short to outlast a first try,
// so with a budget of 0 those for the accumulators look once (looking everywhere
// cost 3%, this 0.4%).
//
// A result that is not finite (an infinite or NaN operand, an overflow of a
// scaled operand or sum) is computed again as the sequential fp32 FMA sum: the
// split of an infinity has no exact terms.  That is slow (the
// layer above, 164 us eager: 202 with one infinite value in one row, 1015 with one
// in every row; with one sum after the other 274 and 2119).
#include <cuda_runtime.h>

#include <atomic>

#include "common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace ec2moe {
// bit 0: a bounded wait timed out; bit 1: a group range (offsets) or a scatter
// destination (perm) outside the rows of the call was skipped
__device__ unsigned int g_f32_error;

namespace {

using namespace tc;

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int UK = 16;
constexpr int WARPS = 16;
constexpr int NUM_THREADS = 32 * WARPS;
constexpr int STAGES = 2;
constexpr int SEG = 2;         // blocks summed in TMEM before they are added to registers
constexpr int MAX_SPLIT = 4;   // CTAs of a cluster that share a tile's K range
constexpr int MAX_GROUPS = 136;

struct FParams {
  const float* A;
  const float* B;
  const float* B2;
  const int32_t* offsets;
  int G, M, a_shared;
  long long a_row_base, out_row_base;
  int N, K, b_group_rows;
  float* out;
  long long ldo;
  const int32_t* perm;
  const float* scale;
  int rep_k;
  long long self_row_base;
  int n_tiles_n;
  int split;          // CTAs of a cluster sharing a tile's K range (1: no cluster)
  int kb_per_split;
  int wide_a;         // A is 32-byte aligned: 256-bit loads
  long long a_rows;
  long long timeout;
  long long row_limit;  // rows of the call: group ranges and scatter destinations lie in [0, row_limit)
};

template <int BN>
struct FCfg {
  static constexpr int B_BYTES = BN * BK * 2;  // one term of the B block
  static constexpr int STAGE_BYTES = 3 * B_BYTES;
  static constexpr int NC = BN / 4;            // accumulator columns of a thread
  static constexpr int PITCH = BN + 4;         // floats per row of the result tile (conflict-free 16-byte columns)
  // the stages; the other CTAs' sums and the result tile use the space between tiles
  static constexpr int SUM_BYTES = (MAX_SPLIT - 1) * NUM_THREADS * NC * 4;
  static constexpr int DATA_BYTES = (SUM_BYTES > 120 * 1024 ? SUM_BYTES : 120 * 1024);  // one CTA per SM in any case
  static constexpr int OFF_BARS = DATA_BYTES;
  static constexpr int N_BARS = 2 * STAGES + 5;
  static constexpr int OFF_SLOT = OFF_BARS + N_BARS * 8;  // TMEM address, abort flag
  static constexpr int OFF_PREFIX = OFF_SLOT + 16;
  static constexpr int OFF_ROW0 = OFF_PREFIX + (MAX_GROUPS + 1) * 4;
  static constexpr int SMEM = 1024 + OFF_ROW0 + MAX_GROUPS * 4;
  // Tensor memory: N_ACC pairs of accumulators, then two stages of A terms (a
  // term is 32 columns: 64 bf16 per lane, two to a column).
  static constexpr int N_ACC = BN == 64 ? 2 : 1;
  static constexpr int A_COL = N_ACC * 2 * BN;
  static constexpr int A_TERM = BK / 2;
  static constexpr int TMEM_COLS = 512;
  static constexpr int B_CHUNKS = BN * BK / 4 / NUM_THREADS;  // 16-byte pieces of B per thread and block
  static_assert(STAGES * STAGE_BYTES <= DATA_BYTES && A_COL + STAGES * 3 * A_TERM <= TMEM_COLS, "on-chip memory");
  static_assert(SMEM <= 232448 && OFF_BARS % 1024 == 0, "shared memory per CTA");
  static_assert(BM * PITCH * 4 <= DATA_BYTES, "the result tile fits");
};

// Packed pairs of fp32 (one instruction for two additions).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// Every operand is multiplied by SCALE before it is split, every sum by UNSCALE
// after: with the last bit of an fp32 number at 2^-149 or above, all its terms
// are then normal bf16 numbers.
constexpr float SCALE = 0x1p24f;
constexpr float UNSCALE = 0x1p-48f;

// The three bf16 terms of two fp32 values, scaled.
__device__ __forceinline__ void split3(float x, float y, uint32_t& t0, uint32_t& t1, uint32_t& t2) {
  unpack2(mul2(pack2(x, y), pack2(SCALE, SCALE)), x, y);
  t0 = pack_bf16x2(x, y);
  const uint64_t r1 = sub2(pack2(x, y), pack2(bf16_lo(t0), bf16_hi(t0)));
  float a, b;
  unpack2(r1, a, b);
  t1 = pack_bf16x2(a, b);
  const uint64_t r2 = sub2(r1, pack2(bf16_lo(t1), bf16_hi(t1)));
  unpack2(r2, a, b);
  t2 = pack_bf16x2(a, b);
}
__device__ __forceinline__ void split3(const float4& v, uint2& t0, uint2& t1, uint2& t2) {
  split3(v.x, v.y, t0.x, t1.x, t2.x);
  split3(v.z, v.w, t0.y, t1.y, t2.y);
}

__device__ __forceinline__ bool finite(float v) { return fabsf(v) < __int_as_float(0x7f800000); }

// Four neighbouring results (rows b, b + K, ... of the weights) from their scaled
// sums: those that are not finite as sequential fp32 FMA sums, side by side, so that a row of
// infinities waits for the loads of eight columns once and not once per result.
// A sum that has become NaN stays NaN, so rows of NaNs end at once.
__device__ __noinline__ float4 fma_redo(float4 v, const float* a, const float* b, int K) {
  float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  const bool redo[4] = {!finite(v.x), !finite(v.y), !finite(v.z), !finite(v.w)};
#pragma unroll 2
  for (int k = 0; k < K; k += 8) {  // K is a multiple of 8
    float x[8], w[4][8];
    load8(a + k, x);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int u = 0; u < 8; ++u) w[j][u] = 0.0f;
      if (redo[j]) load8(b + (long long)j * K + k, w[j]);
    }
    bool open = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int u = 0; u < 8; ++u) s[j] = fmaf(x[u], w[j][u], s[j]);
      open |= redo[j] && s[j] == s[j];
    }
    if (!open) break;
  }
  return make_float4(redo[0] ? s[0] : v.x * UNSCALE, redo[1] ? s[1] : v.y * UNSCALE, redo[2] ? s[2] : v.z * UNSCALE,
                     redo[3] ? s[3] : v.w * UNSCALE);
}
__device__ __forceinline__ void finish(float (&v)[4], const float* a, const float* b, int K) {
  if (finite(v[0]) && finite(v[1]) && finite(v[2]) && finite(v[3])) {
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] *= UNSCALE;
    return;
  }
  const float4 r = fma_redo(make_float4(v[0], v[1], v[2], v[3]), a, b, K);
  v[0] = r.x;
  v[1] = r.y;
  v[2] = r.z;
  v[3] = r.w;
}

// A tile's place: group, valid rows and output columns, first rows of A and B.
struct FTile {
  int g, m_blk, n_blk, m_left, n_left;
  long long a_row, b_row;
};
__device__ __forceinline__ FTile tile_at(const FParams& p, int tile, const int* tile_prefix, const int* row0, int& cursor,
                                         int bn_out) {
  while (tile >= tile_prefix[cursor + 1] * p.n_tiles_n) ++cursor;
  FTile t;
  t.g = cursor;
  const int mt = tile_prefix[t.g + 1] - tile_prefix[t.g];
  const int rem = tile - tile_prefix[t.g] * p.n_tiles_n;
  t.m_blk = rem % mt;
  t.n_blk = rem / mt;
  const int mg = p.offsets ? (p.offsets[t.g + 1] - p.offsets[t.g]) : p.M;
  t.m_left = mg - t.m_blk * BM;
  t.n_left = p.N - t.n_blk * bn_out;
  t.a_row = p.a_row_base + ((p.offsets || !p.a_shared) ? row0[t.g] : 0) + (long long)t.m_blk * BM;
  t.b_row = (long long)t.g * p.b_group_rows + (long long)t.n_blk * bn_out;
  return t;
}

// NC accumulator columns: two runs of NC / 2 (SwiGLU: W1 columns, W3 columns).
template <int NC>
__device__ __forceinline__ void drain_add(uint32_t t_main, uint32_t t_minor, int c0, int c1, float (&acc)[NC]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = h ? c1 : c0;
    uint32_t a[NC / 2], b[NC / 2];
    if constexpr (NC / 2 == 16) {
      tmem_ld16_nw(t_main + c, a);
      tmem_ld16_nw(t_minor + c, b);
    } else {
      tmem_ld8_nw(t_main + c, a);
      tmem_ld8_nw(t_minor + c, b);
    }
    tmem_wait();
#pragma unroll
    for (int j = 0; j < NC / 2; j += 2) {
      float& lo = acc[h * (NC / 2) + j];
      float& hi = acc[h * (NC / 2) + j + 1];
      const uint64_t m = pack2(__uint_as_float(a[j]), __uint_as_float(a[j + 1]));
      const uint64_t n = pack2(__uint_as_float(b[j]), __uint_as_float(b[j + 1]));
      unpack2(add2(pack2(lo, hi), add2(m, n)), lo, hi);
    }
  }
}

template <int BN, int EPI>
__global__ void __launch_bounds__(NUM_THREADS, 1) f32_gemm_kernel(const FParams p) {
  using C = FCfg<BN>;
  constexpr bool GLU = EPI == EPI_SWIGLU;
  constexpr int BN_OUT = GLU ? BN / 2 : BN;
  constexpr int NC = C::NC;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::OFF_BARS);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_SLOT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* tile_prefix = reinterpret_cast<int*>(smem + C::OFF_PREFIX);
  int* row0 = reinterpret_cast<int*>(smem + C::OFF_ROW0);
  float* tile_out = reinterpret_cast<float*>(smem);  // the result tile, over the stages
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);  // warp-uniform for the compiler
  const int lane = threadIdx.x & 31;
  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full[s]), WARPS);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tfull[a]), 1);
      mbar_init(smem_u32(&tempty[a]), WARPS);
    }
    mbar_init(smem_u32(drain), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(C::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (warp == 0) {
    pdl_wait();
    warp_exclusive_scan<(MAX_GROUPS + 31) / 32>(
        p.G, lane,
        [&](int g) {
          int r0 = g * p.M, mg = p.M;
          if (p.offsets) {
            r0 = p.offsets[g];
            mg = p.offsets[g + 1] - r0;
            if (r0 < 0 || mg < 0 || static_cast<long long>(r0) + mg > p.row_limit) {
              // not a range of this call's rows: the group is skipped
              atomicOr(&g_f32_error, 2u);
              r0 = 0;
              mg = 0;
            }
          }
          row0[g] = r0;
          return (mg + BM - 1) / BM;
        },
        tile_prefix);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();
  const uint32_t tmem_base = *tmem_slot;
  const int n_tiles = tile_prefix[p.G] * p.n_tiles_n;
  const int num_kb = (p.K + BK - 1) / BK;
  const long long budget = p.timeout;
  const int rank = p.split > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int tile_first = p.split > 1 ? static_cast<int>(cluster_id_x()) : static_cast<int>(blockIdx.x);
  const int tile_step = p.split > 1 ? static_cast<int>(cluster_count_x()) : static_cast<int>(gridDim.x);

  {
    const int q = warp & 3;      // TMEM lane quadrant
    const int part = warp >> 2;  // which quarter of the columns
    const uint32_t t_row = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
    // accumulator columns [c0, c0 + NC / 2) and [c1, c1 + NC / 2) (SwiGLU: the
    // same output columns of W1 and of W3)
    const int c0 = GLU ? part * (NC / 2) : part * NC;
    const int c1 = GLU ? BN / 2 + part * (NC / 2) : part * NC + NC / 2;
    // A: this thread's row is its TMEM lane, 16 columns of a block (its warp's
    // quarter).  B: 16-byte pieces, rows lr + 32 i, columns lc .. lc + 3.
    const int ac0 = part * 16;
    const bool wide_a = p.wide_a != 0;
    const int lr = threadIdx.x >> 4;
    const int lc = (threadIdx.x & 15) * 4;
    const int soff = lr * 128 + (((lc >> 3) ^ (lr & 7)) << 4) + ((lc >> 2) & 1) * 8;
    int cursor = 0;
    int it = 0;   // blocks so far: stage it & 1
    int seg = 0;  // segments so far: accumulator pair seg & 1
    bool ok = true, any = false;
    // The MMAs of block i of segment sg, by warp 0 once every warp has written
    // its part.  The warp index, the stage and the accumulator go through a
    // shuffle, which tells the compiler that they are warp-uniform, so that the
    // operands of the 24 MMAs stay in uniform registers; one elected lane issues.
    auto multiply = [&](int i, int sg, bool first, bool last) {
      constexpr uint32_t IDESC = idesc_bf16(BM, BN);
      constexpr uint64_t DB = C::B_BYTES >> 4;  // next term of B
      const int st = __shfl_sync(0xffffffffu, i & 1, 0), ac = __shfl_sync(0xffffffffu, sg % C::N_ACC, 0);
      const uint32_t tb = __shfl_sync(0xffffffffu, tmem_base, 0);
      const bool issue = elect_one();
      if ((first && !__all_sync(0xffffffffu, mbar_wait(smem_u32(&tempty[ac]), (static_cast<uint32_t>(sg / C::N_ACC) & 1u) ^ 1u,
                                                       budget, abort_flag, &g_f32_error))) ||
          !__all_sync(0xffffffffu, mbar_wait(smem_u32(&full[st]), static_cast<uint32_t>(i >> 1) & 1u, budget, abort_flag,
                                             &g_f32_error)))
        return;  // the abort flag is up: every later wait of the CTA fails too
      tc_fence_after();
      const uint32_t a0 = tb + C::A_COL + st * 3 * C::A_TERM;
      const uint64_t db = sdesc_sw128(smem_u32(smem + st * C::STAGE_BYTES));
      const uint32_t d_main = tb + static_cast<uint32_t>(ac * 2 * BN);
      const uint32_t d_minor = d_main + BN;
      if (issue) {
#pragma unroll
        for (int kk = 0; kk < BK / UK; ++kk) {
          const uint32_t a = a0 + kk * (UK / 2);
          const uint64_t b = db + 2 * kk;
          const uint32_t more = kk || !first ? 1u : 0u;
          umma_bf16_ts(d_minor, a, b + 2 * DB, IDESC, more);        // x0 w2
          umma_bf16_ts(d_minor, a + C::A_TERM, b + DB, IDESC, 1u);  // x1 w1
          umma_bf16_ts(d_minor, a + 2 * C::A_TERM, b, IDESC, 1u);   // x2 w0
          umma_bf16_ts(d_minor, a, b + DB, IDESC, 1u);              // x0 w1
          umma_bf16_ts(d_minor, a + C::A_TERM, b, IDESC, 1u);       // x1 w0
          umma_bf16_ts(d_main, a, b, IDESC, more);                  // x0 w0
        }
        umma_commit(smem_u32(&empty[st]));
        if (last) umma_commit(smem_u32(&tfull[ac]));
      }
      any = true;
    };
    const int kb_lo = rank * p.kb_per_split;
    const int kb_hi = kb_lo + p.kb_per_split < num_kb ? kb_lo + p.kb_per_split : num_kb;
    for (int tile = tile_first; tile < n_tiles; tile += tile_step) {
      const FTile tc = tile_at(p, tile, tile_prefix, row0, cursor, BN_OUT);
      const int m_left = tc.m_left, n_left = tc.n_left;
      // Rows that are never stored read the tile's first row instead; of B they
      // are neither split nor written.
      const int arow_l = q * 32 + lane;
      const float* src_a =
          p.A + (tc.a_row + (arow_l < m_left && tc.a_row + arow_l < p.a_rows ? arow_l : 0)) * p.K + ac0;
      uint32_t live = 0;  // bit i: B piece i
      // rows 0 .. BN_OUT - 1 of the block from B, the rest (SwiGLU) from B2; 32-bit
      // offsets, as registers are short
      const float* src_b = p.B + tc.b_row * p.K + lc;
      const float* src_b2 = GLU ? p.B2 + tc.b_row * p.K + lc : src_b;
      int off_b[C::B_CHUNKS];
#pragma unroll
      for (int i = 0; i < C::B_CHUNKS; ++i) {
        const int r = (lr + 32 * i) % BN_OUT;
        const bool in = r < n_left;
        live |= in ? 1u << i : 0u;
        off_b[i] = (in ? r : 0) * p.K;
      }
      float ra[16];
      float4 rb[C::B_CHUNKS];
      const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      auto load_a = [&](int kb) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k = kb * BK + ac0 + h * 8;  // K is a multiple of 8: eight columns are inside or outside
          float* r = ra + h * 8;
          if (k >= p.K) {
#pragma unroll
            for (int u = 0; u < 8; ++u) r[u] = 0.0f;
          } else if (wide_a) {
            asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
                         : "l"(src_a + kb * BK + h * 8));
          } else {
            const float4 x = *reinterpret_cast<const float4*>(src_a + kb * BK + h * 8);
            const float4 y = *reinterpret_cast<const float4*>(src_a + kb * BK + h * 8 + 4);
            r[0] = x.x; r[1] = x.y; r[2] = x.z; r[3] = x.w; r[4] = y.x; r[5] = y.y; r[6] = y.z; r[7] = y.w;
          }
        }
      };
      auto load_b = [&](int kb) {
        const bool in_k = kb * BK + lc < p.K;
#pragma unroll
        for (int i = 0; i < C::B_CHUNKS; ++i) {
          const float* src = (GLU && 32 * i >= BN_OUT ? src_b2 : src_b) + off_b[i] + kb * BK;
          rb[i] = in_k ? __ldg(reinterpret_cast<const float4*>(src)) : zero;
        }
      };
      float acc[NC];
#pragma unroll
      for (int j = 0; j < NC; ++j) acc[j] = 0.0f;
      auto drain_segment = [&](int i) {  // segment i of this CTA
        const int ac = i % C::N_ACC;
        if (!__all_sync(0xffffffffu, mbar_wait_strict(smem_u32(&tfull[ac]), static_cast<uint32_t>(i / C::N_ACC) & 1u, budget,
                                               abort_flag, &g_f32_error)))
          return false;
        tc_fence_after();
        const uint32_t t = t_row + static_cast<uint32_t>(ac * 2 * BN);
        drain_add<NC>(t, t + BN, c0, c1, acc);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tempty[ac]));
        return true;
      };
      if (ok) {
        load_a(kb_lo);
        load_b(kb_lo);
      }
      for (int kb = kb_lo; kb < kb_hi && ok; ++kb, ++it) {
        const int st = it & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&empty[st]), (static_cast<uint32_t>(it >> 1) & 1u) ^ 1u, budget,
                                               abort_flag, &g_f32_error))) {
          ok = false;
          break;
        }
        tc_fence_after();
        {
          uint32_t t0[8], t1[8], t2[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) split3(ra[2 * j], ra[2 * j + 1], t0[j], t1[j], t2[j]);
          const uint32_t ta = t_row + C::A_COL + st * 3 * C::A_TERM + part * 8;
          tmem_st8(ta, t0);
          tmem_st8(ta + C::A_TERM, t1);
          tmem_st8(ta + 2 * C::A_TERM, t2);
        }
        uint8_t* sb = smem + st * C::STAGE_BYTES + soff;
#pragma unroll
        for (int i = 0; i < C::B_CHUNKS; ++i) {
          if (!(live >> i & 1u)) continue;
          uint2 t0, t1, t2;
          split3(rb[i], t0, t1, t2);
          *reinterpret_cast<uint2*>(sb + i * 4096) = t0;
          *reinterpret_cast<uint2*>(sb + i * 4096 + C::B_BYTES) = t1;
          *reinterpret_cast<uint2*>(sb + i * 4096 + 2 * C::B_BYTES) = t2;
        }
        // the tensor core reads the B terms through the async proxy, the A terms
        // once the stores to tensor memory have completed
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&full[st]));
        if (kb + 1 < kb_hi) {
          load_a(kb + 1);
          load_b(kb + 1);
        }
        const bool first = (kb - kb_lo) % SEG == 0;
        const bool last = (kb - kb_lo) % SEG == SEG - 1 || kb + 1 == kb_hi;
        // The segment before this one is drained while this one multiplies, or,
        // with one pair of accumulators, before it may.
        if (C::N_ACC == 1 && first && kb > kb_lo && !drain_segment(seg - 1)) ok = false;
        if (warp == 0 && ok) multiply(it, seg, first, last);
        __syncwarp();
        if (C::N_ACC == 2 && first && kb > kb_lo && !drain_segment(seg - 1)) ok = false;
        if (last) ++seg;
      }
      if (ok && !drain_segment(seg - 1)) ok = false;
      if (p.split > 1) {
        // The other CTAs' sums go to the first one's shared memory (its stages
        // are idle: its MMAs of the tile have been drained), which adds them in
        // CTA order.  Every CTA passes both barriers of every tile, also after
        // a wait gave up.
        cluster_sync_all();
        if (rank > 0) {
          const uint32_t dst = map_to_rank(smem_u32(smem) + (rank - 1) * (NUM_THREADS * NC * 4) + threadIdx.x * 16, 0);
#pragma unroll
          for (int j = 0; j < NC; j += 4)
            st_cluster_v4(dst + j * (NUM_THREADS * 4), acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
        }
        cluster_sync_all();
        if (rank > 0) continue;
        for (int r = 1; r < p.split; ++r) {
          const uint8_t* src = smem + (r - 1) * (NUM_THREADS * NC * 4) + threadIdx.x * 16;
#pragma unroll
          for (int j = 0; j < NC; j += 4) {
            const float4 o = *reinterpret_cast<const float4*>(src + j * (NUM_THREADS * 4));
            acc[j] += o.x;
            acc[j + 1] += o.y;
            acc[j + 2] += o.z;
            acc[j + 3] += o.w;
          }
        }
        // every read is done before the result tile below overwrites the sums
        asm volatile("bar.sync 1, %0;" ::"r"(NUM_THREADS) : "memory");
      }

      // Epilogue through shared memory (the stages are idle until the next
      // tile): rows of BN + 4 floats, then whole rows back, 16 bytes per thread
      // in a rolled loop.  Straight from the accumulator registers it was 4-6 KB
      // of code per variant, run once per tile, and 16-byte pieces of 32 rows
      // per store.
      {
        float* row = tile_out + (q * 32 + lane) * C::PITCH;
#pragma unroll
        for (int j = 0; j < NC; j += 4)
          *reinterpret_cast<float4*>(row + (j < NC / 2 ? c0 + j : c1 + j - NC / 2)) =
              make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
      }
      asm volatile("bar.sync 1, %0;" ::"r"(NUM_THREADS) : "memory");
      constexpr int V = BN_OUT / 4;  // float4 per row of the output tile
#pragma unroll 1
      for (int i = threadIdx.x; i < BM * V; i += NUM_THREADS) {
        const int local = i / V, c = i % V * 4;
        if (!ok || local >= m_left || c >= n_left) continue;  // N is a multiple of 8
        const long long out_row = p.out_row_base + row0[tc.g] + (long long)tc.m_blk * BM + local;
        long long dest = out_row;
        float sc = 1.0f;
        if (EPI == EPI_SCATTER) {
          dest = p.perm ? p.perm[out_row] : out_row;
          if (dest < 0 || dest >= p.row_limit) {
            atomicOr(&g_f32_error, 2u);
            continue;
          }
          if (p.scale) sc = p.scale[dest];
        }
        float v[4], w[4];
        *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(tile_out + local * C::PITCH + c);
        if (GLU) *reinterpret_cast<float4*>(w) = *reinterpret_cast<const float4*>(tile_out + local * C::PITCH + BN / 2 + c);
        const float* arow = p.A + (tc.a_row + local) * p.K;
        const long long brow = (tc.b_row + c) * p.K;
        finish(v, arow, p.B + brow, p.K);
        if (GLU) finish(w, arow, p.B2 + brow, p.K);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (EPI == EPI_GELU) v[u] = gelu_erf(v[u]);
          if (GLU) v[u] = silu(v[u]) * w[u];
          if (EPI == EPI_SCATTER) v[u] *= sc;
        }
        const float4 o = make_float4(v[0], v[1], v[2], v[3]);
        const long long col = (long long)tc.n_blk * BN_OUT + c;
        if (EPI == EPI_REPLICATE) {
          for (int r = 0; r < p.rep_k; ++r)
            *reinterpret_cast<float4*>(p.out + (long long)p.perm[out_row * p.rep_k + r] * p.ldo + col) = o;
          if (p.self_row_base >= 0) *reinterpret_cast<float4*>(p.out + (p.self_row_base + out_row) * p.ldo + col) = o;
        } else {
          *reinterpret_cast<float4*>(p.out + dest * p.ldo + col) = o;
        }
      }
      // the tile is read before the next one's blocks overwrite it
      asm volatile("bar.sync 1, %0;" ::"r"(NUM_THREADS) : "memory");
    }
    if (warp == 0 && any && __any_sync(0xffffffffu, !ok || *abort_flag) && elect_one()) {
      // All MMAs issued so far must finish before TMEM is freed.
      umma_commit(smem_u32(drain));
      mbar_drain(smem_u32(drain), 0, DRAIN_CYCLES);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::TMEM_COLS)
                 : "memory");
  }
}

// CTAs (split 1 of `sms` SMs) or clusters of `split` CTAs that run at once; 0
// when such clusters cannot be placed.  Kept here per device beside max_clusters'
// own table, as a launch asks up to five times.
template <int BN, int EPI>
int slots(int split, int sms) {
  if (split == 1) return sms;
  constexpr int DEVICES = 16;
  static std::atomic<int> known[DEVICES][MAX_SPLIT + 1];  // one more than the answer; 0: not asked yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (dev < DEVICES)
    if (const int n = known[dev][split].load(std::memory_order_relaxed)) return n - 1;
  const void* kernel = reinterpret_cast<const void*>(f32_gemm_kernel<BN, EPI>);
  if (ensure_smem_attr(kernel, FCfg<BN>::SMEM) != cudaSuccess) return 0;
  const int n = max_clusters(kernel, NUM_THREADS, FCfg<BN>::SMEM, split);
  if (dev < DEVICES && n > 0) known[dev][split].store(n + 1, std::memory_order_relaxed);
  return n;
}

template <int BN, int EPI>
cudaError_t launch_bn(const GemmArgs& a, const FParams& p, long long tiles, bool one_wave, cudaStream_t s) {
  using C = FCfg<BN>;
  auto* kernel = f32_gemm_kernel<BN, EPI>;
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(kernel), C::SMEM);
  if (e != cudaSuccess) return e;
  const int sms = sm_count();
  const long long cap = one_wave ? sms / p.split : slots<BN, EPI>(p.split, sms);
  const int clusters = static_cast<int>(tiles < cap ? (tiles > 0 ? tiles : 1) : cap);
  KernelScope ks(a.name ? a.name : "gemm_f32", s);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(clusters * p.split);
  cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (p.split > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = p.split;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  if (next_launch_pdl()) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, p);
}

// Tile width and K split by the expected time in units of one 128-wide block:
// a 64-wide block takes about 3/4 of it (A is loaded, split and read by the
// MMAs either way), a tile about 2 more for its first loads and its epilogue,
// a split one 1 more for handing the sums over; waves of the expected tiles
// (one per group of at most 0.8 x 128 rows, else half a partial tile per
// group) times that decide.  So large calls take
// 128-wide tiles, and calls with fewer tiles than SMs split K over a cluster.
// A wave is what runs at once: 152 CTAs, 76 clusters of two, 36 of four (not 38:
// a cluster's SMs lie in one GPC).  Taken as 38, 111 expected tiles were three
// waves on paper and four on the GPU (layer with E = 8, d = 768, d_ff = 3072, T =
// 994: 260 us against 221; T = 1057, 4 allowed 326 against 231; d = 512, d_ff =
// 2048, T = 1585 239 against 175).  37 and 38 tiles still count as one wave: the
// number is an expectation, and the next best choice is the slower one (d = 768,
// T = 260: 143 us against 155; d = 512, d_ff = 2048, T = 400 129 against 134).
// Such a launch has 38 clusters, of which those without a tile end at once.
template <int EPI>
cudaError_t launch_epi(const GemmArgs& a, FParams p, cudaStream_t s) {
  constexpr int DIV = EPI == EPI_SWIGLU ? 2 : 1;
  const int num_kb = (a.K + BK - 1) / BK;
  const int sms = sm_count();
  const int ga = a.g_active > 0 ? a.g_active : a.G;
  const double rows = (double)a.max_rows / ga;  // expected rows per group
  const double m_tiles = a.G == 1 ? (double)((a.max_rows + BM - 1) / BM) : ga * (rows <= 0.8 * BM ? 1.0 : rows / BM + 0.5);
  double best = 0.0;
  int best_bn = 0;
  bool best_one = false;
  for (int bn = 128; bn >= 64; bn /= 2) {
    const int nt = (a.N + bn / DIV - 1) / (bn / DIV);
    for (int sp = 1; sp <= MAX_SPLIT && sp <= num_kb; sp *= 2) {
      const int per = (num_kb + sp - 1) / sp;
      if ((num_kb + per - 1) / per != sp) continue;  // an empty K range
      const int at_once = bn == 128 ? slots<128, EPI>(sp, sms) : slots<64, EPI>(sp, sms);
      if (at_once < 1) continue;
      const double tiles = m_tiles * nt;
      const bool one_wave = tiles <= 1.001 * (sms / sp);
      const double waves = one_wave ? 1.0 : static_cast<double>(static_cast<long long>(tiles / at_once + 0.999));
      const double t = waves * (per * (bn == 128 ? 1.0 : 0.75) + 2.0 + (sp > 1 ? 1.0 : 0.0));
      if (!best_bn || t < best) {
        best = t;
        best_bn = bn;
        best_one = one_wave;
        p.split = sp;
        p.kb_per_split = per;
        p.n_tiles_n = nt;
      }
    }
  }
  const long long tiles = (a.max_rows / BM + a.G) * p.n_tiles_n;
  return best_bn == 64 ? launch_bn<64, EPI>(a, p, tiles, best_one, s) : launch_bn<128, EPI>(a, p, tiles, best_one, s);
}

}  // namespace

cudaError_t launch_gemm_f32(const GemmArgs& a, int epi, cudaStream_t s) {
  if (a.G < 1 || a.G > MAX_GROUPS || a.N % 8 != 0 || a.K % 8 != 0) return cudaErrorInvalidValue;
  FParams p;
  p.A = static_cast<const float*>(a.A);
  p.B = static_cast<const float*>(a.B);
  p.B2 = static_cast<const float*>(a.B2);
  p.offsets = a.offsets;
  p.G = a.G;
  p.M = a.M;
  p.a_shared = a.a_shared;
  p.a_row_base = a.a_row_base;
  p.out_row_base = a.out_row_base;
  p.N = a.N;
  p.K = a.K;
  p.b_group_rows = a.b_group_rows;
  p.out = static_cast<float*>(a.out);
  p.ldo = a.ldo;
  p.perm = a.perm;
  p.scale = a.scale;
  p.rep_k = a.rep_k;
  p.self_row_base = a.self_row_base;
  p.n_tiles_n = p.split = p.kb_per_split = 0;  // launch_epi
  p.a_rows = a.a_rows;
  p.timeout = a.timeout_cycles;
  p.wide_a = reinterpret_cast<uintptr_t>(a.A) % 32 == 0;
  p.row_limit = a.max_rows > 0 ? a.max_rows : (1LL << 62);
  cudaError_t e;
  switch (epi) {
    case EPI_STORE: e = launch_epi<EPI_STORE>(a, p, s); break;
    case EPI_GELU: e = launch_epi<EPI_GELU>(a, p, s); break;
    case EPI_SWIGLU: e = launch_epi<EPI_SWIGLU>(a, p, s); break;
    case EPI_SCATTER: e = launch_epi<EPI_SCATTER>(a, p, s); break;
    case EPI_REPLICATE: e = launch_epi<EPI_REPLICATE>(a, p, s); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

cudaError_t read_f32_error(unsigned int* word) {
  unsigned int zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(word, g_f32_error, sizeof(unsigned int));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(g_f32_error, &zero, sizeof(unsigned int));
}

}  // namespace ec2moe
