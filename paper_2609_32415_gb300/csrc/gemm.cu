// refadapt_gemm: the linear layers of the DiT block around the attention
// (QKV projection, output projection, MLP), bf16 in, fp32 accumulate in TMEM,
// with the elementwise work that follows each layer fused into the epilogue.
//
//   D[r, n] = sum_k A[r, k] W[n, k]        (A rows of one segment and sample,
//                                           W in nn.Linear layout [N][K])
//
// Two kernels: CTA pairs on 256-row output tiles (gemm_pair_kernel, below) and
// one CTA per SM on 128-row tiles (gemm_kernel), both persistent, tiles up to
// 256 columns wide. Calls of few tiles and a long K go to a third form, where
// the CTAs of a cluster share a 128-row tile's K (gemm_kernel, SPLIT). make_plan()
// picks the form and the width. Live tiles
// (those the modes do not skip) are numbered segment-major, then sample, then
// in bands of GROUP_M row tiles, rows fastest inside a band (so the CTAs that
// run at once share a few A row blocks and a few W column blocks, both held in
// L2); CTA c takes tiles c, c + G, c + 2G, ...
//   warp 0      TMA producer: per K step one 128 x 64 A box and one W box of the
//               tile's width x 64 (128-byte swizzle, rows past a segment's end read as
//               zeros) into a 4-stage ring.
//   warp 1      TMEM allocator (512 columns: two 256-column accumulators) and
//               MMA issuer: tcgen05.mma kind::f16, M = 128, N = the tile's
//               width, K = 16, four per stage; commits free the stage and, after a tile's
//               last step, hand the accumulator to the epilogue.
//   warps 2..9  epilogue: two warps per TMEM lane quarter (quarter = warp % 4,
//               thread = output row = TMEM lane), which take the tile's 32-column
//               chunks (QKV: heads) in turn; the next tile's MMAs run into the
//               other accumulator meanwhile.
// Epilogues (fp32 until the final bf16 rounding):
//   STORE  out = acc + bias
//   GELU   out = gelu_tanh(acc + bias)
//   RESID  out = resid + gate[sample] * (acc + bias)        (gated residual)
//   QKV    columns [q | k | v] of H heads of width d: q and k RMS-normalised
//          per head with a [d] weight, then rotated by RoPE on interleaved
//          pairs at the row's joint position; written head-major.
// A tile whose MMAs take 4 us (K = 1024) left the epilogue of four warps, with
// 16-byte accesses 32 rows apart and a global-load latency per 32 columns, as
// the longer part (11 us a tile with GELU). So the per-column vectors of a tile
// go to shared memory and the first residuals to registers before its
// accumulator is ready, and global rows are read and written through a 2 KB
// staging buffer per warp, 64 contiguous bytes of eight rows per instruction.
// Reference segments may be gated on the per-sample mode: their tiles are
// skipped when the mode is REUSE (Algorithm 1 skips reference rows) and, for
// QKV, the K and V column tiles also when it is BOUNDARY (the block keeps its
// cached reference K/V). Every mbarrier wait is bounded; on a timeout the CTA
// drains its own TMA and MMA work, frees TMEM, flags the error word and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>

#include "api_common.h"
#include "tc_ptx.cuh"

namespace ra {
namespace gemm {

constexpr int BM = 128, BN = 256, BK = 64;
constexpr int STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;
constexpr int B_BYTES = BN * BK * 2;
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int OFF_BAR = STAGES * STAGE_BYTES;
constexpr int NUM_BARS = 2 * STAGES + 2 + 2 + 1 + 1;  // full, empty, tfull[2], tempty[2], drain, parts_full
constexpr int OFF_MISC = OFF_BAR + NUM_BARS * 8;
constexpr int EPI_WARPS = 8;
constexpr int EPI_STAGE_BYTES = 32 * 64;                  // 32 rows x 32 bf16 (or 16 fp32) of one warp
constexpr int EPI_WARP_BYTES = EPI_STAGE_BYTES + 2 * 512;  // and two per-column vectors of its 128 columns
constexpr int OFF_EPI = (OFF_MISC + 16 + 127) / 128 * 128;
constexpr int SMEM_BYTES = OFF_EPI + EPI_WARPS * EPI_WARP_BYTES;
constexpr int SMEM_ALLOC = SMEM_BYTES + 1024;
constexpr int THREADS = 64 + 32 * EPI_WARPS;
constexpr int TMEM_COLS = 512;
constexpr int MAX_SPLIT = 4;  // CTAs of a cluster that share one tile's K
static_assert(SMEM_ALLOC <= 232448, "shared memory budget");
// split tiles: the parts to send and those received take the place of the stages
static_assert(2 * (MAX_SPLIT - 1) * (BM * BN * 4 / MAX_SPLIT) <= OFF_BAR, "parts fit the stages");

// CTA-pair kernel: 256-row output tiles; each CTA stages its 128 rows of A
// and its half of the W tile (up to 128 columns), 128 of K per stage (two 128-byte
// swizzle chunks per operand, 64 KB per stage, 3 stages): half the stage
// hand-offs of 64-wide stages, which the fused epilogues gained from (GELU
// +3 %); a K % 128 == 64 tail is a half stage.
constexpr int P_TM = 256;
constexpr int P_STAGES = 3;
constexpr int P_BK = 128;              // K per stage: two 64-column chunks per operand
constexpr int P_CHUNK = 128 * 64 * 2;  // 128 rows x 64 K of one operand (one 128-byte swizzle span)
constexpr int P_A_BYTES = 128 * P_BK * 2;
constexpr int P_B_BYTES = 128 * P_BK * 2;
constexpr int P_STAGE_BYTES = P_A_BYTES + P_B_BYTES;
constexpr int P_OFF_BAR = P_STAGES * P_STAGE_BYTES;
constexpr int P_NUM_BARS = 2 * P_STAGES + 2 + 2 + 1;
constexpr int P_OFF_MISC = P_OFF_BAR + P_NUM_BARS * 8;
constexpr int P_OFF_EPI = (P_OFF_MISC + 16 + 127) / 128 * 128;
constexpr int P_SMEM_BYTES = P_OFF_EPI + EPI_WARPS * EPI_WARP_BYTES;
constexpr int P_SMEM_ALLOC = P_SMEM_BYTES + 1024;
static_assert(P_SMEM_ALLOC <= 232448, "shared memory budget");

struct Seg {
  int32_t pos_offset, reserved;
  const float* bias;
  __nv_bfloat16* out;
  int64_t out_ss, out_sr;
  const __nv_bfloat16* resid;
  int64_t res_ss, res_sr;
  const float* gate;
  int64_t gate_ss;
  __nv_bfloat16* dst[3];  // QKV: q, k, v, head-major
  int64_t dst_sb[3], dst_sh[3], dst_sn[3];
  const float* norm_w[2];  // QKV: q, k
};

// What every role reads before its first tile comes first: a kernel starts with
// a cold constant cache, and each line it touches costs hundreds of cycles.
struct Params {
  int32_t n_seg, B, N, C, kblocks;
  int32_t bn;                // columns of a tile
  int32_t slots, rest_max;   // rest_max > 0: whole rounds of `slots` pair tiles, a rest of up to rest_max split
  int32_t cols, cols_q;      // column tiles of N; of the query part (QKV)
  int32_t rows[3], m_tiles[3], gated[3];
  int32_t K;
  const int32_t* mode;
  int32_t* err_word;
  uint64_t budget_ns;
  const float4* rope;  // [pos][d/4]: (cos, sin) of two consecutive pairs
  int32_t rope_len;
  float norm_eps;
  Seg seg[3];
  CUtensorMap tm_a[3], tm_w[3];
};

struct Tile {
  int seg, s, m0, n0;
};

constexpr int GROUP_M = 16;  // tile rows per band of the tile order

// Walks the live tiles in order; tile indices only grow. A piece is the tiles
// of one (segment, sample): all column tiles, or none when the segment is gated
// and the sample reuses, or only the query's (QKV at the boundary, which keeps
// its cached K and V).
template <int TM, int EPI>  // TM: output rows per tile, 128 (one CTA) or 256 (a CTA pair)
struct Walk {
  int g = 0, s = 0, cols = -1;  // cols: column tiles of the piece
  int64_t begin = 0;            // first tile of the piece

  __device__ __forceinline__ int piece_cols(const Params& p) const {
    if (p.gated[g]) {
      const int m = p.mode[s];
      if (m == RA_MODE_REUSE) return 0;
      if (EPI == RA_EPI_QKV && m == RA_MODE_BOUNDARY) return p.cols_q;
    }
    return p.cols;
  }
  // Tile t, or false past the last one.
  __device__ __forceinline__ bool at(const Params& p, int64_t t, Tile& r) {
    if (cols < 0) cols = piece_cols(p);
    while (t - begin >= int64_t(p.m_tiles[g]) * cols) {
      begin += int64_t(p.m_tiles[g]) * cols;
      ++s;
      if (p.m_tiles[g] == 0) {
        s = p.B;
      } else if (p.B > 4 && !p.gated[g] && t - begin <= 0xffffffff) {
        // the samples' pieces are alike: count them off at once
        const uint32_t n = uint32_t(p.m_tiles[g]) * uint32_t(cols), k = uint32_t(t - begin) / n;
        const int pass = int(min(k, uint32_t(p.B - s)));
        begin += int64_t(n) * pass;
        s += pass;
      }
      if (s == p.B) {
        s = 0;
        if (++g == p.n_seg) return false;
      }
      cols = piece_cols(p);
    }
    r.seg = g;
    r.s = s;
    const uint32_t rem = uint32_t(t - begin);
    // Grouped order: bands of GROUP_M tile rows, rows fastest inside a band, so
    // the tiles in flight at once (one per CTA pair) share a few A row blocks
    // and a few W column blocks that stay in L2, and W streams from HBM once per
    // band instead of once per wave.
    const uint32_t band_tiles = uint32_t(GROUP_M) * uint32_t(cols);
    const uint32_t band = rem / band_tiles, idx = rem - band * band_tiles;
    const int m_first = int(band) * GROUP_M;
    const uint32_t rows = uint32_t(min(GROUP_M, p.m_tiles[g] - m_first));
    r.m0 = (m_first + int(idx % rows)) * TM;
    r.n0 = int(idx / rows) * p.bn;
    return true;
  }
};

// The tiles of a call's whole rounds; those past them, if at most p.rest_max, are
// its rest. Every tile where the call has no rest.
template <int TM, int EPI>
__device__ __forceinline__ int64_t round_tiles(const Params& p) {
  if (p.rest_max == 0) return INT64_MAX;
  Walk<TM, EPI> w;
  int64_t live = 0;
  for (w.g = 0; w.g < p.n_seg; ++w.g)
    for (w.s = 0; w.s < p.B; ++w.s) live += int64_t(p.m_tiles[w.g]) * w.piece_cols(p);
  const int64_t rest = live % p.slots;
  return rest <= p.rest_max ? live - rest : live;
}

// The tile of item t of a launch. SPLIT: where the call has a rest, a quarter
// (128 rows by REST_BN columns) of a pair tile of it; p.m_tiles and p.bn are the
// pair kernel's then.
constexpr int REST_BN = 128;
template <int EPI, bool SPLIT>
__device__ __forceinline__ bool tile_at(const Params& p, Walk<BM, EPI>& walk, int64_t t, Tile& tl) {
  if (!SPLIT || p.rest_max == 0) return walk.at(p, t, tl);
  if (!walk.at(p, round_tiles<P_TM, EPI>(p) + (t >> 2), tl)) return false;
  tl.m0 = 2 * tl.m0 + (t & 1 ? BM : 0);
  tl.n0 += t & 2 ? REST_BN : 0;
  return tl.m0 < p.rows[tl.seg];
}

// GELU, tanh form, of two values through the identity
// 0.5 x (1 + tanh(u)) = x / (1 + e^(-2u)), u = sqrt(2/pi) (x + 0.044715 x^3),
// with e^(-2u) = 2^(x (c + 0.044715 c x^2)), c = -2 sqrt(2/pi) log2(e): one
// exponential and one reciprocal (an exponential that overflows to +inf for
// very negative x gives -0).
__device__ __forceinline__ void gelu_tanh2(float& x0, float& x1) {
  constexpr float c = -2.f * 0.7978845608028654f * 1.4426950408889634f;
  const uint64_t x = f2_pack(x0, x1);
  float z0, z1;
  f2_unpack(f2_mul(x, f2_fma(f2_mul(x, x), f2_pack(0.044715f * c, 0.044715f * c), f2_pack(c, c))), z0, z1);
  float d0, d1;
  f2_unpack(f2_add(f2_pack(ex2_approx(z0), ex2_approx(z1)), f2_pack(1.f, 1.f)), d0, d1);
  f2_unpack(f2_mul(x, f2_pack(rcp_approx(d0), rcp_approx(d1))), x0, x1);
}

// The 64-byte row slots of a warp's staging buffer: 16-byte piece q of row r.
// The permutation keeps both access patterns free of bank conflicts (every
// lane its own row; eight rows, four lanes a row).
__device__ __forceinline__ uint4* stage_slot(uint8_t* stage, int r, int q) {
  return reinterpret_cast<uint4*>(stage + r * 64 + ((q ^ ((r >> 1) & 3)) << 4));
}
// Four 16-byte loads per lane of up to 32 rows of 64 bytes at `src` (row
// stride in bytes): load i is piece lane % 4 of row 8 i + lane / 4.
__device__ __forceinline__ void rows_fetch(const char* src, int64_t stride, int nrow, uint4 (&v)[4]) {
  const int lane = threadIdx.x & 31, r0 = lane >> 2;
  const char* ptr = src + r0 * stride + (lane & 3) * 16;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    v[i] = (r0 + 8 * i < nrow) ? *reinterpret_cast<const uint4*>(ptr + 8 * i * stride) : make_uint4(0, 0, 0, 0);
}
// rows_fetch's registers -> the lane's own row (64 bytes), through the staging buffer.
__device__ __forceinline__ void rows_turn(uint8_t* stage, const uint4 (&v)[4], uint4 (&own)[4]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 4; ++i) *stage_slot(stage, 8 * i + (lane >> 2), lane & 3) = v[i];
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 4; ++q) own[q] = *stage_slot(stage, lane, q);
  __syncwarp();
}
// 32 fp32 of every lane's row -> bf16 -> up to 32 rows of 64 bytes at `dst`.
__device__ __forceinline__ void rows_store(uint8_t* stage, const float (&x)[32], char* dst, int64_t stride, int nrow) {
  const int lane = threadIdx.x & 31, r0 = lane >> 2;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    *stage_slot(stage, lane, q) =
        make_uint4(pack_bf16x2(x[8 * q], x[8 * q + 1]), pack_bf16x2(x[8 * q + 2], x[8 * q + 3]),
                   pack_bf16x2(x[8 * q + 4], x[8 * q + 5]), pack_bf16x2(x[8 * q + 6], x[8 * q + 7]));
  __syncwarp();
  char* ptr = dst + r0 * stride + (lane & 3) * 16;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint4 v = *stage_slot(stage, r0 + 8 * i, lane & 3);
    if (r0 + 8 * i < nrow) *reinterpret_cast<uint4*>(ptr + 8 * i * stride) = v;
  }
  __syncwarp();
}

// What an epilogue warp works on: its 32 rows (row0 + lane, nrow of them in
// the segment), its share of the tile's columns (half 0 or 1), its shared
// memory (staging buffer, two vectors of 128 per-column values) and the TMEM
// address of its lanes in the tile's accumulator; cols: columns of the tile.
struct EpiWarp {
  int row0, nrow, half, cols;
  uint8_t* stage;
  float* vec0;
  float* vec1;
  uint32_t acc;
};

// 32 accumulators plus 32 per-column values from shared memory.
__device__ __forceinline__ void add_cols(const uint32_t (&v)[32], const float* cols, float (&x)[32]) {
  const float4* c4 = reinterpret_cast<const float4*>(cols);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 c = c4[i];
    x[4 * i] = __uint_as_float(v[4 * i]) + c.x;
    x[4 * i + 1] = __uint_as_float(v[4 * i + 1]) + c.y;
    x[4 * i + 2] = __uint_as_float(v[4 * i + 2]) + c.z;
    x[4 * i + 3] = __uint_as_float(v[4 * i + 3]) + c.w;
  }
}

// STORE, GELU, RESID: chunk j of the warp is tile columns 32 (half + 2 j) ...
template <int EPI, class Ready>
__device__ __forceinline__ bool epilogue_linear(const Params& p, const Tile& tl, const EpiWarp& w, Ready ready) {
  const Seg& sg = p.seg[tl.seg];
  const int lane = threadIdx.x & 31, n0 = tl.n0 + 32 * w.half;
  // this warp's; the last tile of a row may reach past N (a multiple of 32)
  const int chunks = (min(w.cols, p.N - tl.n0) / 32 + 1 - w.half) >> 1;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (j >= chunks) break;
    w.vec0[32 * j + lane] = sg.bias ? sg.bias[n0 + 64 * j + lane] : 0.f;
    if (EPI == RA_EPI_RESID) w.vec1[32 * j + lane] = sg.gate[int64_t(tl.s) * sg.gate_ss + n0 + 64 * j + lane];
  }
  const char* res = nullptr;
  uint4 ra[4], rb[4];  // residuals of the next even and odd chunk
  if (EPI == RA_EPI_RESID && chunks > 0) {
    res = reinterpret_cast<const char*>(sg.resid + int64_t(tl.s) * sg.res_ss + int64_t(w.row0) * sg.res_sr + n0);
    rows_fetch(res, 2 * sg.res_sr, w.nrow, ra);
    if (chunks > 1) rows_fetch(res + 128, 2 * sg.res_sr, w.nrow, rb);
  }
  char* out = reinterpret_cast<char*>(sg.out + int64_t(tl.s) * sg.out_ss + int64_t(w.row0) * sg.out_sr + n0);
  __syncwarp();
  if (!ready()) return false;
  if (w.nrow <= 0 || chunks <= 0) return true;
  uint32_t v[32];
  if (EPI != RA_EPI_RESID) tmem_ld32(w.acc + 32 * w.half, v);
  auto chunk = [&](int j, uint4 (&rc)[4]) {
    float x[32];
    uint4 r[4];
    if (EPI == RA_EPI_RESID) {
      // Residuals two chunks ahead (one ahead left about 1000 cycles of global
      // latency in every chunk); the accumulators are not loaded ahead in
      // exchange, the registers allow one of the two without spills.
      tmem_ld32(w.acc + 32 * w.half + 64 * j, v);
      rows_turn(w.stage, rc, r);
      if (j + 2 < chunks) rows_fetch(res + 128 * (j + 2), 2 * sg.res_sr, w.nrow, rc);
    }
    tmem_ld_wait_for(v);
    add_cols(v, w.vec0 + 32 * j, x);
    if (EPI != RA_EPI_RESID && j + 1 < chunks) tmem_ld32(w.acc + 32 * w.half + 64 * (j + 1), v);
    if (EPI == RA_EPI_GELU) {
#pragma unroll
      for (int i = 0; i < 32; i += 2) gelu_tanh2(x[i], x[i + 1]);
    } else if (EPI == RA_EPI_RESID) {
      const float4* g4 = reinterpret_cast<const float4*>(w.vec1 + 32 * j);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t rw[4] = {r[q].x, r[q].y, r[q].z, r[q].w};
        const float4 g0 = g4[2 * q], g1 = g4[2 * q + 1];
        const float gv[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          x[8 * q + 2 * e] = fmaf(gv[2 * e], x[8 * q + 2 * e], __uint_as_float(rw[e] << 16));
          x[8 * q + 2 * e + 1] = fmaf(gv[2 * e + 1], x[8 * q + 2 * e + 1], __uint_as_float(rw[e] & 0xFFFF0000u));
        }
      }
    }
    rows_store(w.stage, x, out + 128 * j, 2 * sg.out_sr, w.nrow);
  };
#pragma unroll 1
  for (int j = 0; j < chunks; j += 2) {
    chunk(j, ra);
    if (j + 1 < chunks) chunk(j + 1, rb);
  }
  return true;
}

// QKV: heads half, half + 2, ... of the tile.
template <int D, class Ready>
__device__ __forceinline__ bool epilogue_qkv(const Params& p, const Tile& tl, const EpiWarp& w, Ready ready) {
  constexpr int CH = D / 32;
  const int heads = (p.bn / D + 1 - w.half) >> 1;  // this warp's
  const Seg& sg = p.seg[tl.seg];
  const int lane = threadIdx.x & 31;
  const int part = tl.n0 / p.C;  // 0 q, 1 k, 2 v
  const int h0 = (tl.n0 - part * p.C) / D + w.half;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (j / CH >= heads) break;
    const int c = 32 * (j % CH) + lane;  // column within head h0 + 2 (j / CH)
    w.vec0[32 * j + lane] = sg.bias ? sg.bias[part * p.C + (h0 + 2 * (j / CH)) * D + c] : 0.f;
    if (part < 2) w.vec1[32 * j + lane] = sg.norm_w[part][c];
  }
  __syncwarp();
  // RoPE rows of the warp's positions: (cos, sin) of D / 2 pairs, 64 bytes = 16 columns at a time
  const char* rope = reinterpret_cast<const char*>(p.rope + int64_t(sg.pos_offset + w.row0) * (D / 4));
  uint4 cnext[4];
  if (part < 2) rows_fetch(rope, 4 * D, w.nrow, cnext);
  if (!ready()) return false;
  if (w.nrow <= 0 || heads <= 0) return true;
  char* dst0 = reinterpret_cast<char*>(sg.dst[part] + tl.s * sg.dst_sb[part] + int64_t(w.row0) * sg.dst_sn[part]);
#pragma unroll 1
  for (int hh = 0; hh < heads; ++hh) {
    const uint32_t acc = w.acc + (w.half + 2 * hh) * D;
    const float* bias = w.vec0 + 32 * CH * hh;
    const float* nw = w.vec1 + 32 * CH * hh;
    uint32_t v[32];
    float rstd = 0.f;
    tmem_ld32(acc, v);
    if (part < 2) {
      // a first pass over the head's accumulators for the mean square
      float s0 = 0.f, s1 = 0.f;
#pragma unroll 1
      for (int c = 0; c < CH; ++c) {
        float x[32];
        tmem_ld_wait_for(v);
        add_cols(v, bias + 32 * c, x);
        tmem_ld32(acc + 32 * ((c + 1) % CH), v);
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          s0 = fmaf(x[i], x[i], s0);
          s1 = fmaf(x[i + 1], x[i + 1], s1);
        }
      }
      rstd = rsqrtf((s0 + s1) / float(D) + p.norm_eps);
    }
    char* dst = dst0 + 2 * int64_t(h0 + 2 * hh) * sg.dst_sh[part];
#pragma unroll 1
    for (int c = 0; c < CH; ++c) {
      float x[32];
      tmem_ld_wait_for(v);
      add_cols(v, bias + 32 * c, x);
      if (c + 1 < CH) tmem_ld32(acc + 32 * (c + 1), v);
      if (part < 2) {
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint4 own[4];
          rows_turn(w.stage, cnext, own);
          // the next 16 columns' table entries (the next head starts over)
          const int nx = (2 * c + hf + 1) % (2 * CH);
          if (nx != 0 || hh + 1 < heads) rows_fetch(rope + 64 * nx, 4 * D, w.nrow, cnext);
          const float4* w4 = reinterpret_cast<const float4*>(nw + 32 * c + 16 * hf);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float4 wv = w4[q];
            const float cs[4] = {__uint_as_float(own[q].x), __uint_as_float(own[q].y), __uint_as_float(own[q].z),
                                 __uint_as_float(own[q].w)};
            float* xe = &x[16 * hf + 4 * q];
            const float a0 = xe[0] * rstd * wv.x, a1 = xe[1] * rstd * wv.y;
            const float b0 = xe[2] * rstd * wv.z, b1 = xe[3] * rstd * wv.w;
            xe[0] = a0 * cs[0] - a1 * cs[1];
            xe[1] = a0 * cs[1] + a1 * cs[0];
            xe[2] = b0 * cs[2] - b1 * cs[3];
            xe[3] = b0 * cs[3] + b1 * cs[2];
          }
        }
      }
      rows_store(w.stage, x, dst + 64 * c, 2 * sg.dst_sn[part], w.nrow);
    }
  }
  return true;
}

// Epilogue of one warp's share of an output tile; ready() waits for the
// accumulator (false: the wait was given up). D: head dim (QKV).
template <int EPI, int D, class Ready>
__device__ __forceinline__ bool epilogue_tile(const Params& p, const Tile& tl, const EpiWarp& w, Ready ready) {
  if constexpr (EPI == RA_EPI_QKV)
    return epilogue_qkv<D>(p, tl, w, ready);
  else
    return epilogue_linear<EPI>(p, tl, w, ready);
}

// A split tile: each CTA of the cluster has the sums over its part of K in its
// own TMEM; afterwards rank r has columns [r, r + 1) * bn / cs of the whole sums
// there. Each rank hands every other rank that one's columns, in fp32, by a bulk
// copy between the CTAs' shared memory (the stages are idle by then), and adds
// its own columns up in rank order. Every thread of the cluster takes part in
// the cluster barrier: before it every rank's barriers exist, its stages are idle
// and its parts are written, after it they are copied (a cluster barrier of its
// own in the set-up cost 0.2 us). ok: this warp's accumulator is complete. Every
// rank sends and waits for what it receives, also after a wait of this CTA was
// given up: no CTA exits with a copy into it, or out of it, in flight.
// The merge of a 128 x 256 tile between two CTAs (64 KB each way) takes 2.6 us.
__device__ __forceinline__ bool merge_parts(const WaitCtl& ctl, uint8_t* smem, uint64_t* parts_full, uint32_t acc,
                                            bool ok, int bn, int half, int quarter, int rank, int cs) {
  const int lane = threadIdx.x & 31, row = quarter * 32 + lane;
  const int cw = bn / cs;                            // columns per rank
  const uint32_t part_bytes = uint32_t(BM) * cw * 4;  // [column / 4][row] of 16 bytes
  uint8_t* send = smem;                              // parts for the other ranks, in rank order
  uint8_t* recv = smem + (cs - 1) * part_bytes;      // parts from the other ranks, in rank order
  const bool leader = quarter == 0 && half == 0 && lane == 0;
  if (leader) mbar_arrive_expect_tx(parts_full, (cs - 1) * part_bytes);
#pragma unroll 1
  for (int c0 = 32 * half; c0 < bn; c0 += 64) {
    const int q = c0 / cw;
    if (q == rank) continue;
    uint32_t v[32];
    tmem_ld32(acc + c0, v);
    tmem_ld_wait_for(v);
    if (!ok) {  // what was given up is NaN on every rank
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = 0x7fffffffu;
    }
    uint4* dst = reinterpret_cast<uint4*>(send + (q - (q > rank ? 1 : 0)) * part_bytes) +
                 ((c0 - q * cw) >> 2) * BM + row;
#pragma unroll
    for (int i = 0; i < 32; i += 4) dst[(i >> 2) * BM] = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
  }
  fence_proxy_async_smem();  // the parts are next read by bulk copies
  cluster_sync_all();
  if (leader)
    for (int q = 0; q < cs; ++q)
      if (q != rank)
        bulk_copy_to_cta(mapa_shared(smem_u32(recv + (rank - (rank > q ? 1 : 0)) * part_bytes), q),
                         send + (q - (q > rank ? 1 : 0)) * part_bytes, part_bytes,
                         mapa_shared(smem_u32(parts_full), q));
  const bool got = __all_sync(0xffffffffu, mbar_wait(parts_full, 0, ctl) ||
                                               mbar_wait_drain(parts_full, 0, ctl.budget_ns));
  if (!got || !ok) return false;
#pragma unroll 1
  for (int c0 = 32 * half; c0 < cw; c0 += 64) {
    uint32_t v[32];
    float x[32];
    tmem_ld32(acc + rank * cw + c0, v);
    tmem_ld_wait_for(v);
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = 0.f;
#pragma unroll 1
    for (int r = 0; r < cs; ++r) {
      const float4* src = reinterpret_cast<const float4*>(recv + (r - (r > rank ? 1 : 0)) * part_bytes) +
                          (c0 >> 2) * BM + row;
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        const float4 y = r == rank ? make_float4(__uint_as_float(v[i]), __uint_as_float(v[i + 1]),
                                                 __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]))
                                   : src[(i >> 2) * BM];
        x[i] += y.x;
        x[i + 1] += y.y;
        x[i + 2] += y.z;
        x[i + 3] += y.w;
      }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(x[i]);
    tmem_st32(acc + rank * cw + c0, v);
  }
  tmem_st_wait();
  return true;
}

// SPLIT: a cluster takes one tile, each rank a contiguous part of its K
// (merge_parts adds them up), then its share of the columns in the epilogue.
template <int EPI, int D, bool SPLIT = false>
__global__ void __launch_bounds__(THREADS, 1) gemm_kernel(const __grid_constant__ Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + OFF_BAR);
  uint64_t* full = bars;
  uint64_t* empty = bars + STAGES;
  uint64_t* tfull = bars + 2 * STAGES;
  uint64_t* tempty = bars + 2 * STAGES + 2;
  uint64_t* drain = bars + 2 * STAGES + 4;
  uint64_t* parts_full = bars + 2 * STAGES + 5;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + OFF_MISC + 4);
  volatile int* live = reinterpret_cast<volatile int*>(smem + OFF_MISC + 8);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = SPLIT ? int(cluster_rank()) : 0, cs = SPLIT ? int(cluster_size()) : 1;
  const int64_t t0 = SPLIT ? blockIdx.x / cs : blockIdx.x, step = SPLIT ? gridDim.x / cs : gridDim.x;
  const int kb0 = SPLIT ? p.kblocks * rank / cs : 0;  // this CTA's K steps
  const int kb1 = SPLIT ? p.kblocks * (rank + 1) / cs : p.kblocks;
  const int bn = SPLIT && p.rest_max > 0 ? REST_BN : p.bn;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull + b, 1);
      mbar_init(tempty + b, EPI_WARPS);
    }
    mbar_init(drain, 1);
    mbar_init(parts_full, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, TMEM_COLS);
  if (SPLIT && warp == 2) {
    // The modes may leave this cluster no tile: it goes now, before the barriers
    // of the merge (reuse rows of a call planned with a rest 75.8 -> 72.2 us).
    pdl_wait();
    Walk<BM, EPI> walk;
    Tile tl;
    *live = tile_at<EPI, SPLIT>(p, walk, t0, tl);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem0 = SPLIT ? 0 : *tmem_slot;  // SPLIT reads it per role: 0.3 us less there, 0.1 more without
  if (SPLIT && !*live) {  // uniform over the cluster
    if (warp == 1) tmem_dealloc(*tmem_slot, TMEM_COLS);
    return;
  }
  const WaitCtl ctl{abort_flag, p.err_word, p.budget_ns};
  pdl_launch();
  if (warp != 0) pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      // -------------------------------------------------------------- producer
      for (int g = 0; g < p.n_seg; ++g)
        if (p.rows[g] > 0) {
          tma_prefetch_desc(&p.tm_a[g]);
          tma_prefetch_desc(&p.tm_w[g]);
        }
      pdl_wait();
      int64_t it = 0;  // K steps issued
      bool ok = true;
      Walk<BM, EPI> walk;
      Tile tl;
      for (int64_t t = t0; ok && tile_at<EPI, SPLIT>(p, walk, t, tl); t += step) {
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
          const int st = int(it % STAGES);
          if (it >= STAGES && !(ok = mbar_wait(empty + st, uint32_t((it / STAGES - 1) & 1), ctl))) break;
          uint8_t* sa = smem + st * STAGE_BYTES;
          mbar_arrive_expect_tx(full + st, A_BYTES + bn * BK * 2);
          tma_load_4d(sa, &p.tm_a[tl.seg], full + st, kb * BK, tl.m0, 0, tl.s);
          tma_load_4d(sa + A_BYTES, &p.tm_w[tl.seg], full + st, kb * BK, tl.n0, 0, 0);
        }
      }
      if (*abort_flag) {
        for (int st = 0; st < STAGES; ++st) {
          const int64_t n_s = (it > st) ? (it - st + STAGES - 1) / STAGES : 0;
          if (n_s > 0) mbar_wait_drain(full + st, uint32_t((n_s - 1) & 1), p.budget_ns);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // -------------------------------------------------------------- MMA issuer
      const uint32_t idesc = idesc_bf16_f32(BM, bn, 0, 0);
      const uint32_t s0 = smem_u32(smem), tmem = SPLIT ? *tmem_slot : tmem0;
      int64_t it = 0;
      int i = 0;
      bool ok = true, issued = false;
      Walk<BM, EPI> walk;
      Tile tl;
      for (int64_t t = t0; ok && tile_at<EPI, SPLIT>(p, walk, t, tl); t += step) {
        const int buf = i & 1, use = i >> 1;
        if (use > 0 && !(ok = mbar_wait(tempty + buf, uint32_t((use - 1) & 1), ctl))) break;
        tc_fence_after();
        const uint32_t d_t = tmem + uint32_t(buf * BN);
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
          const int st = int(it % STAGES);
          if (!(ok = mbar_wait(full + st, uint32_t((it / STAGES) & 1), ctl))) break;
          tc_fence_after();
          const uint32_t sa = s0 + st * STAGE_BYTES, sb = sa + A_BYTES;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            umma_ss(d_t, sdesc_sw128(sa + kk * 32, 16, 1024), sdesc_sw128(sb + kk * 32, 16, 1024), idesc,
                    (kb > kb0 || kk > 0) ? 1u : 0u);
          umma_commit(empty + st);
          issued = true;
        }
        if (!ok) break;
        umma_commit(tfull + buf);
        ++i;
      }
      if (!ok && issued) {
        umma_commit(drain);
        mbar_wait_drain(drain, 0, p.budget_ns);
      }
    }
  } else {
    // ---------------------------------------------------------------- epilogue
    const int quarter = warp & 3;
    const uint32_t tmem = SPLIT ? *tmem_slot : tmem0;
    EpiWarp w;
    w.half = (warp - 2) >> 2;
    w.stage = smem + OFF_EPI + (warp - 2) * EPI_WARP_BYTES;
    w.vec0 = reinterpret_cast<float*>(w.stage + EPI_STAGE_BYTES);
    w.vec1 = w.vec0 + 128;
    int i = 0;
    Walk<BM, EPI> walk;
    Tile tl;
    for (int64_t t = t0; tile_at<EPI, SPLIT>(p, walk, t, tl); t += step) {
      const int buf = i & 1, use = i >> 1;
      w.row0 = tl.m0 + quarter * 32;
      w.nrow = min(32, p.rows[tl.seg] - w.row0);
      w.acc = tmem + (uint32_t(quarter * 32) << 16) + uint32_t(buf * BN);
      w.cols = bn;
      const uint32_t acc = w.acc;
      if (SPLIT) {
        w.cols /= cs;
        w.acc += uint32_t(rank * w.cols);
        tl.n0 += rank * w.cols;
      }
      if (!epilogue_tile<EPI, D>(p, tl, w, [&] {
            bool ok = __all_sync(0xffffffffu, mbar_wait(tfull + buf, uint32_t(use & 1), ctl));
            tc_fence_after();
            if (SPLIT) ok = merge_parts(ctl, smem, parts_full, acc, ok, bn, w.half, quarter, rank, cs);
            return ok;
          }))
        break;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty + buf);
      ++i;
    }
  }
  if (SPLIT) {
    // Warps 0 and 1 meet the epilogue's cluster barrier here. No CTA exits before
    // every part has been read from it and received.
    __syncwarp();
    if (warp < 2) cluster_sync_all();
    cluster_sync_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(SPLIT ? *tmem_slot : tmem0, TMEM_COLS);
  }
}


// CTA-pair variant (cluster of two, cta_group::2). Both CTAs walk the same
// tile sequence (cluster c takes tiles c, c + G/2, ...); per K step each CTA's
// producer loads its own 128 A rows and its half of the W tile, and both
// loads complete on rank 0's full barrier (rank 0 arms it for both CTAs'
// bytes). Rank 0's MMA thread issues M = 256 MMAs of the tile's width; commits are
// multicast to both CTAs (stage free, accumulator ready). Each CTA's epilogue
// reads its own TMEM rows and arrives on rank 0's accumulator-free barrier
// (count 16). The two CTAs meet at a cluster barrier before TMEM is freed and
// before either exits, so no remote arrive or MMA outlives its target.
template <int EPI, int D>
__global__ void __launch_bounds__(THREADS, 1) gemm_pair_kernel(const __grid_constant__ Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + P_OFF_BAR);
  uint64_t* full = bars;
  uint64_t* empty = bars + P_STAGES;
  uint64_t* tfull = bars + 2 * P_STAGES;
  uint64_t* tempty = bars + 2 * P_STAGES + 2;
  uint64_t* drain = bars + 2 * P_STAGES + 4;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + P_OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + P_OFF_MISC + 4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int64_t cid = blockIdx.x >> 1, ncl = gridDim.x >> 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < P_STAGES; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull + b, 1);
      mbar_init(tempty + b, 2 * EPI_WARPS);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers and TMEM exist before any cross-CTA use
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const WaitCtl ctl{abort_flag, p.err_word, p.budget_ns};
  pdl_launch();
  if (warp != 0) pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      // -------------------------------------------------------------- producer (both CTAs)
      for (int g = 0; g < p.n_seg; ++g)
        if (p.rows[g] > 0) {
          tma_prefetch_desc(&p.tm_a[g]);
          tma_prefetch_desc(&p.tm_w[g]);
        }
      pdl_wait();
      const uint32_t full0 = mapa_shared(smem_u32(full), 0);  // rank 0's full barriers
      int64_t it = 0;
      bool ok = true;
      Walk<P_TM, EPI> walk;
      Tile tl;
      const int64_t end = round_tiles<P_TM, EPI>(p);
      for (int64_t t = cid; ok && t < end && walk.at(p, t, tl); t += ncl) {
        for (int kb = 0; kb < (p.kblocks + 1) / 2; ++kb, ++it) {
          const int st = int(it % P_STAGES);
          if (it >= P_STAGES && !(ok = mbar_wait(empty + st, uint32_t((it / P_STAGES - 1) & 1), ctl))) break;
          uint8_t* sa = smem + st * P_STAGE_BYTES;
          const int chunks = (2 * kb + 1 < p.kblocks) ? 2 : 1;  // K % 128 == 64: the last stage is half
          if (rank == 0) mbar_arrive_expect_tx(full + st, chunks * (2 * P_CHUNK + p.bn * 128));
          for (int c = 0; c < chunks; ++c) {
            tma_load_4d_pair(sa + c * P_CHUNK, &p.tm_a[tl.seg], full0 + 8u * st, kb * P_BK + c * 64,
                             tl.m0 + int(rank) * 128, 0, tl.s);
            tma_load_4d_pair(sa + P_A_BYTES + c * P_CHUNK, &p.tm_w[tl.seg], full0 + 8u * st, kb * P_BK + c * 64,
                             tl.n0 + int(rank) * (p.bn / 2), 0, 0);
          }
        }
      }
      if (*abort_flag) {
        if (rank == 0) {
          // rank 0's full barriers count both CTAs' bytes of every phase it armed
          for (int st = 0; st < P_STAGES; ++st) {
            const int64_t n_s = (it > st) ? (it - st + P_STAGES - 1) / P_STAGES : 0;
            if (n_s > 0) mbar_wait_drain(full + st, uint32_t((n_s - 1) & 1), p.budget_ns);
          }
        } else {
          // this CTA cannot observe its own loads' completion: give them time to land
          const uint64_t t0 = globaltimer_ns();
          while (globaltimer_ns() - t0 < 200000ull) {
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      // -------------------------------------------------------------- MMA issuer (rank 0)
      const uint32_t idesc = idesc_bf16_f32(P_TM, p.bn, 0, 0);
      const uint32_t s0 = smem_u32(smem);
      int64_t it = 0;
      int i = 0;
      bool ok = true, issued = false;
      Walk<P_TM, EPI> walk;
      Tile tl;
      const int64_t end = round_tiles<P_TM, EPI>(p);
      for (int64_t t = cid; ok && t < end && walk.at(p, t, tl); t += ncl) {
        const int buf = i & 1, use = i >> 1;
        if (use > 0 && !(ok = mbar_wait_cluster(tempty + buf, uint32_t((use - 1) & 1), ctl))) break;
        tc_fence_after();
        const uint32_t d_t = tmem + uint32_t(buf * BN);
        for (int kb = 0; kb < (p.kblocks + 1) / 2; ++kb, ++it) {
          const int st = int(it % P_STAGES);
          if (!(ok = mbar_wait(full + st, uint32_t((it / P_STAGES) & 1), ctl))) break;
          tc_fence_after();
          const uint32_t sa = s0 + st * P_STAGE_BYTES, sb = sa + P_A_BYTES;
          const int ksteps = (2 * kb + 1 < p.kblocks) ? P_BK / 16 : 64 / 16;
#pragma unroll
          for (int kk = 0; kk < P_BK / 16; ++kk) {
            if (kk >= ksteps) break;
            const uint32_t o = uint32_t((kk >> 2) * P_CHUNK + (kk & 3) * 32);
            umma_ss_pair(d_t, sdesc_sw128(sa + o, 16, 1024), sdesc_sw128(sb + o, 16, 1024), idesc,
                         (kb > 0 || kk > 0) ? 1u : 0u);
          }
          umma_commit_pair(empty + st, 0x3);
          issued = true;
        }
        if (!ok) break;
        umma_commit_pair(tfull + buf, 0x3);
        ++i;
      }
      if (!ok && issued) {
        umma_commit_pair(drain, 0x1);
        mbar_wait_drain(drain, 0, p.budget_ns);
      }
    }
  } else {
    // ---------------------------------------------------------------- epilogue (both CTAs)
    const int quarter = warp & 3;
    EpiWarp w;
    w.half = (warp - 2) >> 2;
    w.stage = smem + P_OFF_EPI + (warp - 2) * EPI_WARP_BYTES;
    w.vec0 = reinterpret_cast<float*>(w.stage + EPI_STAGE_BYTES);
    w.vec1 = w.vec0 + 128;
    const uint32_t tempty0 = mapa_shared(smem_u32(tempty), 0);
    int i = 0;
    Walk<P_TM, EPI> walk;
    Tile tl;
    const int64_t end = round_tiles<P_TM, EPI>(p);
    for (int64_t t = cid; t < end && walk.at(p, t, tl); t += ncl) {
      const int buf = i & 1, use = i >> 1;
      w.row0 = tl.m0 + int(rank) * 128 + quarter * 32;
      w.cols = p.bn;
      w.nrow = min(32, p.rows[tl.seg] - w.row0);
      w.acc = tmem + (uint32_t(quarter * 32) << 16) + uint32_t(buf * BN);
      if (!epilogue_tile<EPI, D>(p, tl, w, [&] {
            const bool ok = __all_sync(0xffffffffu, mbar_wait(tfull + buf, uint32_t(use & 1), ctl));
            tc_fence_after();
            return ok;
          }))
        break;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0)
          mbar_arrive(tempty + buf);
        else
          mbar_arrive_remote(tempty0 + 8u * buf);
      }
      ++i;
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem, TMEM_COLS);
}

__global__ void rope_table_kernel(float* table, int32_t n_pos, int32_t d, double base) {
  const int64_t n = int64_t(n_pos) * (d / 2);
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t pos = i / (d / 2);
    const int pair = int(i % (d / 2));
    const double ang = double(pos) * pow(base, -2.0 * pair / double(d));
    double s, c;
    sincos(ang, &s, &c);
    table[2 * i] = float(c);
    table[2 * i + 1] = float(s);
  }
}

// The kernels by epilogue (QKV: by head dim too), one CTA per tile and CTA pairs.
using Kernel = void (*)(Params);
struct Kernels {
  Kernel single, pair, split;  // split: STORE, GELU and RESID
};
Kernels pick(int epi, int d) {
  switch (epi) {
    case RA_EPI_STORE: return {gemm_kernel<RA_EPI_STORE, 0>, gemm_pair_kernel<RA_EPI_STORE, 0>, gemm_kernel<RA_EPI_STORE, 0, true>};
    case RA_EPI_GELU: return {gemm_kernel<RA_EPI_GELU, 0>, gemm_pair_kernel<RA_EPI_GELU, 0>, gemm_kernel<RA_EPI_GELU, 0, true>};
    case RA_EPI_RESID: return {gemm_kernel<RA_EPI_RESID, 0>, gemm_pair_kernel<RA_EPI_RESID, 0>, gemm_kernel<RA_EPI_RESID, 0, true>};
    default:
      return d == 128 ? Kernels{gemm_kernel<RA_EPI_QKV, 128>, gemm_pair_kernel<RA_EPI_QKV, 128>, nullptr}
                      : Kernels{gemm_kernel<RA_EPI_QKV, 64>, gemm_pair_kernel<RA_EPI_QKV, 64>, nullptr};
  }
}

bool aligned16(const void* ptr) { return (reinterpret_cast<uintptr_t>(ptr) & 15u) == 0; }

// Launches `ctas` CTAs in clusters of cs.
ra_status launch(const Params& p, Kernel fn, int smem, int64_t ctas, int cs, cudaStream_t st) {
  const ra_status as = ensure_dynamic_smem(reinterpret_cast<const void*>(fn), smem, "refadapt_gemm");
  if (as != RA_OK) return as;
  cudaLaunchAttribute attr[2];
  attr[0] = pdl_attribute();
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cs;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(unsigned(ctas), 1, 1);
  cfg.blockDim = dim3(THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = cs > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, fn, p);
  if (e != cudaSuccess) {
    set_error("refadapt_gemm: launch failed: %s", cudaGetErrorString(e));
    cudaGetLastError();
    return RA_ECUDA;
  }
  return launch_status("refadapt_gemm");
}

// How a call is cut into tiles: CTA pairs or single CTAs, tile columns, and the
// CTAs of a cluster that share a tile's K (1: a CTA has a tile of its own).
// rest_max > 0: pair tiles of 256 columns in whole rounds, and a rest of at most
// this many split, each into four tiles of clusters of cs CTAs, by a second launch.
struct Plan {
  bool pair;
  int bn, cs, rest_max;
};

// Clusters of cs CTAs of a split kernel that can run at once on the current
// device (they live inside one GPC, so the floorplan decides; every split kernel
// has the same launch shape); cached per device. 0: none, or the query failed,
// and nothing is split.
int max_clusters(Kernel fn, int cs) {
  static std::mutex mu;
  static int cache[64][MAX_SPLIT + 1];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return 0;
  }
  std::lock_guard<std::mutex> lk(mu);
  int& n = cache[dev][cs];
  if (n > 0) return n;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(cs, 1, 1);
  cfg.blockDim = dim3(THREADS, 1, 1);
  cfg.dynamicSmemBytes = SMEM_ALLOC;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int found = 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_ALLOC) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&found, fn, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n = found;
}

// The cheapest cut by a model of the two kernels' time (microseconds), fitted to
// single waves of 256 to 64 columns at K = 1024 and 4096 on a GB300 (each within
// 6 %): what one round of tiles takes grows with the operand bytes a CTA stages
// per K step (each is written to shared memory once and read once, which fills
// its port before the tensor core is full), so a narrower tile costs nearly as
// much as a wide one (256 columns 5.1 us per 1024 of K, 128 columns 4.0) and
// pays only where it saves a round: 13 row tiles of 256 by N = 3072 make 156
// tiles of 256 columns (three rounds of 76 pairs, the last one nearly empty;
// 188 us at K = 12288) or 208 of 192 columns (three shorter rounds, 164 us).
// Few tiles of a long K leave SMs idle (a small model's MLP output, 377 rows by
// N = 1024, K = 4096, is 64 narrow tiles, 19.2 us): there two or four CTAs of a
// cluster share a tile's K, which costs a merge and pays from about K = 3072 up
// while the clusters fit the GPU at once (12.1 us in clusters of four on tiles of
// 128 columns; 516 rows, K = 12288, N = 3072 58.9 -> 50.3 in clusters of two;
// at K = 1024 it loses, 7.3 -> 8.2). Not for QKV, whose epilogue needs whole heads,
// nor where the caller chose the tiles.
// Whole rounds of pair tiles and a small rest: the rest's tiles are cut into
// quarters and split in the same way by a second launch, which costs 13 us and
// its share of K, so only a long K gains (K = 12288, N = 3072: 13 row tiles, two
// rounds and 4 tiles, 162 -> 157 us; 1572 rows, one round and 8, 105 -> 95). Its
// 256-column tiles also suit what the modes leave better than narrow ones.
// Calls with gated segments are weighed with and without them.
Plan make_plan(const ra_gemm_args& a, int sms) {
  Plan best{false, 256, 1, 0};
  double best_us = 1e30;
  auto tiles_of = [&](int tm, int bn, int64_t* all, int64_t* open) {
    const int64_t cols = (a.N + bn - 1) / bn;
    *all = *open = 0;  // tiles, and those of segments that are not gated
    for (int g = 0; g < a.n_seg; ++g) {
      const int64_t t = a.seg[g].rows > 0 ? int64_t(a.B) * ((a.seg[g].rows + tm - 1) / tm) * cols : 0;
      *all += t;
      if (!a.seg[g].gated) *open += t;
    }
  };
  // Many column tiles that all read the same few rows of A contend for the L2
  // lines these lie in (4 rows, K = 2048, N = 8192: 21.7 us in 128 tiles of 64
  // columns, 11.8 in 32 of 256; from 32 rows on 10.3 and 11.9).
  bool few_rows = false;
  for (int g = 0; g < a.n_seg; ++g) few_rows |= a.seg[g].rows > 0 && a.seg[g].rows < 32;
  for (int pair = 0; pair < 2; ++pair) {
    if ((a.tile_mode == 1 && pair) || (a.tile_mode == 2 && !pair) || (pair && sms < 2)) continue;
    const int tm = pair ? P_TM : BM, slots = pair ? sms / 2 : sms;
    for (int bn = 256; bn >= 64; bn -= 32) {
      if (a.epilogue == RA_EPI_QKV && (bn % a.d != 0 || (a.H * a.d) % bn != 0)) continue;
      if (few_rows && bn < 256 && a.N / bn > 40) continue;
      int64_t all, open;
      tiles_of(tm, bn, &all, &open);
      const double epilogue = 0.0085 * bn;  // of a tile, hidden behind the next one's MMAs
      double round = a.K / 1024.0 * (pair ? 3.11 + 0.00766 * bn : 3.4 + 0.0127 * bn);
      round = round > epilogue ? round : epilogue;
      const double fixed = pair ? 4.4 + 0.0088 * bn : 3.6;
      double us = fixed + round * double((all + slots - 1) / slots);
      if (open > 0 && open < all) us += fixed + round * double((open + slots - 1) / slots);
      if (us < best_us) {
        best_us = us;
        best = Plan{pair != 0, bn, 1, 0};
      }
    }
  }
  if (a.epilogue == RA_EPI_QKV || a.tile_mode != 0) return best;
  const double merge = 4.0;
  for (int cs = 2; cs <= MAX_SPLIT; cs *= 2) {
    if (a.K / BK < 4 * cs) break;
    const int clusters = max_clusters(pick(a.epilogue, a.d).split, cs);
    if (clusters == 0) continue;
    for (int bn = 256; bn >= 32 * cs; bn /= 2) {
      int64_t all, open;
      tiles_of(BM, bn, &all, &open);
      const double wave = 3.6 + merge + a.K / 1024.0 / cs * (3.4 + 0.0127 * bn);
      double us = wave * double((all + clusters - 1) / clusters);
      if (open > 0 && open < all) us += wave * double((open + clusters - 1) / clusters);
      if (us < 0.97 * best_us) {
        best_us = us;
        best = Plan{false, bn, cs, 0};
      }
    }
    const int slots = sms / 2;
    const double round = a.K / 1024.0 * (3.11 + 0.00766 * BN), fixed = 4.4 + 0.0088 * BN;
    const double wave = 13.3 + a.K / 1024.0 / cs * (3.4 + 0.0127 * REST_BN);
    int64_t all, open;
    tiles_of(P_TM, BN, &all, &open);
    int64_t rest_max = int64_t(round / wave) * clusters / 4;
    if (rest_max > slots - 1) rest_max = slots - 1;
    if (slots < 1 || rest_max < 1 || all < slots) continue;
    auto time = [&](int64_t tiles) {
      const int64_t rest = tiles % slots;
      const bool split = rest <= rest_max;
      return fixed + round * double(split ? tiles / slots : tiles / slots + 1) +
             wave * double(split ? (4 * rest + clusters - 1) / clusters : 0);
    };
    const double us = time(all) + (open > 0 && open < all ? time(open) : 0.0);
    if (us < 0.97 * best_us) {
      best_us = us;
      best = Plan{true, BN, cs, int(rest_max)};
    }
  }
  return best;
}

}  // namespace gemm
}  // namespace ra

extern "C" ra_status refadapt_rope_table(float* table, int32_t n_pos, int32_t d, double base, void* stream) {
  using namespace ra;
  clear_error();
  if (!table || n_pos < 1 || d < 2 || d % 4 != 0 || !(base > 1.0)) {
    set_error("refadapt_rope_table: table NULL, n_pos < 1, d not a multiple of 4 or base <= 1");
    return RA_EINVAL;
  }
  const int64_t n = int64_t(n_pos) * (d / 2);
  const int blocks = int((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  gemm::rope_table_kernel<<<blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(table, n_pos, d, base);
  return launch_status("refadapt_rope_table");
}

extern "C" ra_status refadapt_gemm(const ra_gemm_args* a, void* stream) {
  using namespace ra;
  using namespace ra::gemm;
  clear_error();
  if (!a) {
    set_error("refadapt_gemm: args is NULL");
    return RA_EINVAL;
  }
  if (a->B < 1 || a->n_seg < 1 || a->n_seg > 3 || a->K < BK || a->K % BK != 0 || a->N < BN || a->N % BN != 0) {
    set_error("refadapt_gemm: need B >= 1, 1 <= n_seg <= 3, K a positive multiple of 64, N of 256 "
              "(B=%d n_seg=%d N=%d K=%d)", a->B, a->n_seg, a->N, a->K);
    return RA_EINVAL;
  }
  if (a->epilogue < RA_EPI_STORE || a->epilogue > RA_EPI_QKV) {
    set_error("refadapt_gemm: unknown epilogue %d", a->epilogue);
    return RA_EINVAL;
  }
  Params p;
  std::memset(&p, 0, sizeof(p));
  p.n_seg = a->n_seg;
  p.B = a->B;
  p.N = a->N;
  p.K = a->K;
  p.kblocks = a->K / BK;
  p.mode = a->mode;
  p.err_word = a->err_word;
  p.budget_ns = wait_budget_ns();
  p.norm_eps = a->norm_eps;
  if (a->epilogue == RA_EPI_QKV) {
    if ((a->d != 64 && a->d != 128) || a->H < 1 || int64_t(3) * a->H * a->d != a->N || (a->H * a->d) % BN != 0) {
      set_error("refadapt_gemm: QKV needs d in {64, 128}, N = 3 H d and H d a multiple of 256");
      return RA_EINVAL;
    }
    if (!a->rope || !aligned16(a->rope) || a->rope_len < 1 || !(a->norm_eps >= 0.f)) {
      set_error("refadapt_gemm: QKV needs a 16-byte aligned rope table, rope_len >= 1 and norm_eps >= 0");
      return RA_EINVAL;
    }
    p.C = a->H * a->d;
    p.rope = reinterpret_cast<const float4*>(a->rope);
    p.rope_len = a->rope_len;
  }
  if (a->tile_mode < 0 || a->tile_mode > 2) {
    set_error("refadapt_gemm: tile_mode %d (0 auto, 1 one CTA per tile, 2 CTA pairs)", a->tile_mode);
    return RA_EINVAL;
  }
  const int sms = num_sms();
  const Plan plan = make_plan(*a, sms);
  const bool pair = plan.pair;
  const int tm = pair ? P_TM : BM;
  p.bn = plan.bn;
  const int64_t cols = (a->N + plan.bn - 1) / plan.bn;
  p.cols = int32_t(cols);
  p.cols_q = p.C / plan.bn;
  int64_t tiles = 0;
  for (int g = 0; g < a->n_seg; ++g) {
    const ra_gemm_seg& s = a->seg[g];
    Seg& d = p.seg[g];
    if (s.rows < 0) {
      set_error("refadapt_gemm: seg %d rows < 0", g);
      return RA_EINVAL;
    }
    p.rows[g] = s.rows;
    p.m_tiles[g] = (s.rows + tm - 1) / tm;
    p.gated[g] = s.gated ? 1 : 0;
    d.pos_offset = s.pos_offset;
    d.bias = s.bias;
    if (s.gated && !a->mode) {
      set_error("refadapt_gemm: seg %d is gated but mode is NULL", g);
      return RA_EINVAL;
    }
    if (s.rows == 0) continue;
    if (!s.a || !s.w || !aligned16(s.a) || !aligned16(s.w) || s.a_stride_r % 8 != 0 || s.a_stride_s % 8 != 0 ||
        s.a_stride_r < a->K || s.a_stride_s < 0) {
      set_error("refadapt_gemm: seg %d: A and W must be 16-byte aligned, strides multiples of 8 elements, "
                "a_stride_r >= K", g);
      return RA_EINVAL;
    }
    if (s.bias && !aligned16(s.bias)) {
      set_error("refadapt_gemm: seg %d: bias must be 16-byte aligned", g);
      return RA_EINVAL;
    }
    if (a->epilogue == RA_EPI_QKV) {
      const ra_seg* dst[3] = {&s.q_out, &s.k_out, &s.v_out};
      const char* nm[3] = {"q_out", "k_out", "v_out"};
      for (int z = 0; z < 3; ++z) {
        if (dst[z]->n != s.rows || !check_seg(*dst[z], nm[z], false)) {
          if (dst[z]->n != s.rows) set_error("refadapt_gemm: seg %d: %s.n must equal rows", g, nm[z]);
          return RA_EINVAL;
        }
        d.dst[z] = static_cast<__nv_bfloat16*>(dst[z]->ptr);
        d.dst_sb[z] = dst[z]->stride_b;
        d.dst_sh[z] = dst[z]->stride_h;
        d.dst_sn[z] = dst[z]->stride_n;
      }
      if (!s.q_norm || !s.k_norm || !aligned16(s.q_norm) || !aligned16(s.k_norm)) {
        set_error("refadapt_gemm: seg %d: QKV needs 16-byte aligned q_norm and k_norm", g);
        return RA_EINVAL;
      }
      if (s.pos_offset < 0 || int64_t(s.pos_offset) + s.rows > a->rope_len) {
        set_error("refadapt_gemm: seg %d: positions [%d, %d) outside the rope table (%d)", g, s.pos_offset,
                  s.pos_offset + s.rows, a->rope_len);
        return RA_EINVAL;
      }
      d.norm_w[0] = s.q_norm;
      d.norm_w[1] = s.k_norm;
    } else {
      if (!s.out || !aligned16(s.out) || s.out_stride_r % 8 != 0 || s.out_stride_s % 8 != 0 ||
          s.out_stride_r < a->N) {
        set_error("refadapt_gemm: seg %d: out must be 16-byte aligned with strides multiples of 8 elements, "
                  "out_stride_r >= N", g);
        return RA_EINVAL;
      }
      d.out = static_cast<__nv_bfloat16*>(s.out);
      d.out_ss = s.out_stride_s;
      d.out_sr = s.out_stride_r;
      if (a->epilogue == RA_EPI_RESID) {
        if (!s.resid || !s.gate || !aligned16(s.resid) || !aligned16(s.gate) || s.resid_stride_r % 8 != 0 ||
            s.resid_stride_s % 8 != 0 || s.gate_stride_s % 4 != 0) {
          set_error("refadapt_gemm: seg %d: RESID needs 16-byte aligned resid and gate, resid strides "
                    "multiples of 8 elements, gate_stride_s of 4", g);
          return RA_EINVAL;
        }
        d.resid = static_cast<const __nv_bfloat16*>(s.resid);
        d.res_ss = s.resid_stride_s;
        d.res_sr = s.resid_stride_r;
        d.gate = s.gate;
        d.gate_ss = s.gate_stride_s;
      }
    }
    ra_seg as{const_cast<void*>(s.a), s.a_stride_s, 0, s.a_stride_r, s.rows, 0};
    ra_seg ws{const_cast<void*>(s.w), 0, 0, a->K, a->N, 0};
    // The pair kernel loads half a tile's rows of W per CTA.
    if (!encode_seg(&p.tm_a[g], as, a->B, 1, a->K, BK, BM, true) ||
        !encode_seg(&p.tm_w[g], ws, 1, 1, a->K, BK, pair ? plan.bn / 2 : plan.bn, true))
      return RA_EINVAL;
    if (int64_t(p.m_tiles[g]) * cols > 2147483647) {
      set_error("refadapt_gemm: seg %d: too many rows", g);
      return RA_EINVAL;
    }
    tiles += int64_t(a->B) * p.m_tiles[g] * cols;
  }
  if (tiles == 0) return RA_OK;
  const Kernels kn = pick(a->epilogue, a->d);
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t slots = pair ? (sms / 2 > 0 ? sms / 2 : 1) : sms;
  p.slots = int32_t(slots);
  p.rest_max = plan.rest_max;
  if (plan.rest_max > 0) {
    note_launch("rounds of CTA pairs, up to %d tiles in clusters of %d", plan.rest_max, plan.cs);
    // No modes leave more whole rounds than all tiles do, or a larger split rest.
    const int64_t rest = tiles % slots, whole = rest <= plan.rest_max ? tiles - rest : tiles;
    const ra_status r = launch(p, kn.pair, P_SMEM_ALLOC, 2 * (whole < slots ? whole : slots), 2, st);
    if (r != RA_OK) return r;
    return launch(p, kn.split, SMEM_ALLOC, int64_t(4) * plan.rest_max * plan.cs, plan.cs, st);
  }
  if (pair) note_launch("CTA pairs, %d columns", plan.bn);
  else if (plan.cs > 1) note_launch("clusters of %d, %d columns", plan.cs, plan.bn);
  else note_launch("single CTAs, %d columns", plan.bn);
  if (pair) return launch(p, kn.pair, P_SMEM_ALLOC, 2 * (tiles < slots ? tiles : slots), 2, st);
  if (plan.cs > 1) return launch(p, kn.split, SMEM_ALLOC, tiles * plan.cs, plan.cs, st);
  return launch(p, kn.single, SMEM_ALLOC, tiles < slots ? tiles : slots, 1, st);
}
