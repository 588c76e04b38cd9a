// refadapt_joint_attn: joint [text; reference; target] attention with the
// per-tile reference mass, on tcgen05 tensor cores (sm_103a).
//
// One CTA computes an item: a pair of 128-row Q tiles (A, B) of one role for
// one (sample, head); both tiles share every K/V tile it streams. Where items
// are too few for the SMs, or leave a small rest after whole rounds, the CTAs of
// a cluster share an item's keys (merge_split); where items fit few rounds, an
// item is one Q tile whose even and odd key tiles run as two streams (DUAL,
// merge_dual). make_plan chooses and says what each form measured.
// What bounds it: over many key tiles the shared-memory port. A key tile of a
// pair (d = 128) is 2048 cycles of MMA and as many of shared-memory reads and
// writes (Q 2 x 32 KB, K 2 x 32, V 2 x 32 read; K and V written), and takes 2712
// in all; at the largest sizes the power limit follows (joint attention of 53.5k
// keys 1650 TFLOP/s). Small launches are bound by a CTA's fixed cost (launch,
// set-up, first loads, cold code: about 5 of the 8 us of an 8-head launch of 544
// rows) and by the softmax latency of its key tiles.
// The roles of a CTA's warps, for a pair:
//   warp 0      TMA producer: Q tiles A and B once, then K and V tiles of the
//               text, reference (cache slot) and target segments in that order
//               into a STAGES-deep ring of 128-byte-swizzled shared buffers.
//   warp 1      TMEM allocator and MMA issuer (one thread). TMEM columns:
//               S_A [0,128), S_B [128,256), O_A [256,..), O_B [384,..).
//               S_t = Q_t K_j^T (kind::f16, fp32 accumulate); P_t is written
//               back over the first 64 columns of S_t as packed bf16 and read
//               from TMEM as the A operand of O_t += P_t V_j. Issue order per
//               key tile: PV_A(j), QK_A(j+1), PV_B(j), QK_B(j+1), so the tensor
//               core works on one tile while the other tile's softmax runs.
//               Each product's K steps leave one asm block (one predicate,
//               descriptors advanced by immediates): the issuing warp shares
//               its SM sub-partition with two softmax warps, and the MMA rate
//               follows the issuing thread's instruction count.
//   warps 2, 3  idle (they complete warpgroup 0, which hands registers over:
//               setmaxnreg 56 there, 224 in the softmax warpgroups; 4 x 56 +
//               8 x 224 = 12 x 168, the launch allocation).
//   warps 4..7  softmax / epilogue of tile A, warps 8..11 of tile B: thread =
//               query row = TMEM lane (lane quarter = warp % 4). Online softmax
//               in log2 units with a lazy rescale (the running max only moves
//               when a tile's max exceeds it by more than 2^8), the row sum l
//               and the reference-only row sum l_ref (paper Eq. 4's inner sum
//               is l_ref / l); then O / l -> bf16 global and the tile's sum of
//               l_ref / l over its mass rows -> mass_partial.
// Fused reference-cache update (paper Eq. 11), when the caller passes this
// step's reference projections: samples in COMPUTE or FULL read reference
// Q/K/V from them, and the producer thread copies what it streams into the
// cache slot with TMA bulk-tensor stores from the swizzled stage buffers. The
// first item of each (sample, head) stores every reference K/V tile one tile
// after its load (the stage is refilled only once the store has read it; the
// CTAs of a split item each store their own keys' tiles); each reference-row
// item stores its Q tiles. Each byte of the fresh
// reference rows is read from HBM once for both the MMAs and the copy.
// Segment tails: TMA zero-fills rows past a segment's end; tail key tiles mask
// the padded columns to -inf (probability 0) and the epilogue skips padded
// query rows; TMA stores clip rows past a segment's end. Every mbarrier wait is
// bounded (WaitCtl); on a timeout the CTA drains its own TMA and MMA work, frees
// TMEM, flags the caller's error word and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "api_common.h"
#include "tc_ptx.cuh"

namespace ra {
namespace attn {

constexpr int BM = 128;  // query rows per tile (= TMEM lanes)
constexpr int BN = 128;  // keys per tile
constexpr int NUM_THREADS = 384;
constexpr int MAX_SPLIT = 4;     // CTAs of a cluster that share one item's keys
constexpr int MAX_SAMPLES = 32;  // samples of a launch that numbers the live items (one lane each)
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLowestMax = -FLT_MAX;
constexpr float kRescaleThresh = 8.0f;  // log2 units: p <= 2^8 between rescales

// DUAL: one Q tile and a deeper ring for two streams of key tiles.
template <int D, bool DUAL = false>
struct Cfg {
  static constexpr int CHUNKS = D / 64;           // 64-element (128-byte) swizzle chunks per row
  static constexpr int CHUNK_BYTES = BM * 128;    // one chunk of a 128-row tile
  static constexpr int TILE_BYTES = BM * D * 2;   // one Q, K or V tile (BN == BM)
  static constexpr int STAGES = DUAL ? (D == 128 ? 3 : 6) : (D == 128 ? 2 : 4);
  static constexpr int OFF_Q = 0;                 // Q tiles A and B
  static constexpr int OFF_K = OFF_Q + (DUAL ? 1 : 2) * TILE_BYTES;
  static constexpr int OFF_V = OFF_K + STAGES * TILE_BYTES;
  static constexpr int OFF_BAR = OFF_V + STAGES * TILE_BYTES;
  // q_full, k_full[S], k_empty[S], v_full[S], v_empty[S], s_full[2], p_ready[2], o_done[2], drain, parts_full
  static constexpr int NUM_BARS = 1 + 4 * STAGES + 2 + 2 + 2 + 1 + 1;
  static constexpr int OFF_MISC = OFF_BAR + NUM_BARS * 8;  // tmem slot, abort flag, 8 floats
  static constexpr int OFF_ITEM = (OFF_MISC + 64 + 15) / 16 * 16;  // int4 per softmax warp
  static constexpr int SMEM_BYTES = OFF_ITEM + 8 * 16;
  static constexpr int SMEM_ALLOC = SMEM_BYTES + 1024;  // slack for 1024-byte alignment
  // Split launches (not DUAL): (m, l, l_ref) of every row from every rank of the cluster.
  // The O parts to send and those received (up to 3/4 of 256 rows x D fp32
  // each) reuse the tile buffers.
  static constexpr int OFF_STATS = (SMEM_BYTES + 15) / 16 * 16;
  static constexpr int SPLIT_BYTES = OFF_STATS + MAX_SPLIT * 2 * BM * 16;
  static constexpr int SPLIT_ALLOC = SPLIT_BYTES + 1024;
  static_assert(DUAL || (2 * (2 * BM * D * 4 / MAX_SPLIT) * (MAX_SPLIT - 1) <= OFF_BAR && 2 * BM * D * 4 <= OFF_BAR),
                "O parts fit the tile buffers");
  static_assert(DUAL || SPLIT_ALLOC <= 232448, "shared memory budget");
  static constexpr uint32_t TMEM_COLS = 512;
  static constexpr uint32_t TM_S = 0, TM_O = 256;       // + 128 * tile
  static_assert(SMEM_ALLOC <= 232448, "shared memory budget");
};

struct Params {
  __nv_bfloat16* o_ptr[3];
  int64_t o_sb[3], o_sh[3], o_sn[3];
  int32_t nq[3];  // query rows per role
  int32_t nk[3];  // key rows per role
  int32_t q_tiles[3];
  int32_t q_blocks[3];  // items: groups of `group` Q tiles
  int32_t group;        // Q tiles per item: 2, or 1 (KIND_DUAL)
  uint32_t per_inv[2];  // 2^32 / items per head, rounded up (with reference rows, without), or 0: divide
  int32_t b0, nb;       // samples of this launch: [b0, b0 + nb)
  int32_t per_sample;   // > 0: this many items a sample, dead ones among them; b0 + item / per_sample, nb = 1
  int32_t part;         // PART_ALL, PART_ROUNDS or PART_REST of the live items
  int32_t slots;        // CTAs of a full round
  int32_t rest_max;     // largest rest that PART_REST takes
  int32_t kv_tiles[3];
  int32_t B, H;
  int32_t mass_rows;
  int32_t mass_stride;  // count mass rows 0, k, 2k, ... (k <= 1: every row)
  int32_t mpl;
  float scale_log2;
  const float* bias;
  const int32_t* mode;
  float* mass_partial;
  int32_t* err_word;
  int32_t* a_b;
  int32_t step;
  int32_t fresh;     // refreshing samples read reference rows from tm_*f
  int32_t store_kv;  // ... and copy those K / V tiles into tm_k[1] / tm_v[1]
  int32_t store_q;   // ... and those Q tiles into tm_q[1]
  uint64_t budget_ns;
  CUtensorMap tm_q[3];
  CUtensorMap tm_k[3];
  CUtensorMap tm_v[3];
  CUtensorMap tm_qf, tm_kf, tm_vf;  // this step's reference rows (fused cache update)
};

// A launch runs all live items (reference items of reusing samples are not
// live), or the whole rounds of them that fill the GPU, or the rest. Over more
// samples than lanes every item has a CTA, and a dead one's ends after its set-up
// (launches of 32 samples each, one after another, took up to twice as long: 256
// samples of 4 heads of 128 rows 67 us, 42 in one).
enum { PART_ALL = 0, PART_ROUNDS = 1, PART_REST = 2 };

// Live items in whole rounds, given all of them.
__host__ __device__ __forceinline__ int round_items(int live, int slots, int rest_max) {
  const int rest = live % slots;
  return rest <= rest_max ? live - rest : live;
}

__device__ __forceinline__ bool refreshes(int m) { return m == RA_MODE_COMPUTE || m == RA_MODE_FULL; }

// Tile (c0 = column, c1 = row, c2 = head, c3 = sample) of a 4-D tensor map,
// shared -> global, bulk-group completion; rows past the tensor are clipped.
__device__ __forceinline__ void tma_store_4d(const void* tmap, const void* src, int32_t c0, int32_t c1,
                                             int32_t c2, int32_t c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(tmap)),
               "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ void kv_tile(const Params& p, int j, int& r, int& row0) {
  if (j < p.kv_tiles[0]) {
    r = 0;
    row0 = j * BN;
  } else if (j < p.kv_tiles[0] + p.kv_tiles[1]) {
    r = 1;
    row0 = (j - p.kv_tiles[0]) * BN;
  } else {
    r = 2;
    row0 = (j - p.kv_tiles[0] - p.kv_tiles[1]) * BN;
  }
}

// Row maximum over the 64 logits in v[] (columns col0 .. col0+63 of the tile),
// those of columns >= nvalid left out.
__device__ __forceinline__ float max64(const float (&v)[64], int col0, int nvalid, float m_in) {
  float m0 = m_in, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
  for (int c = 0; c < 64; c += 8) {
    const int e = col0 + c;
    m0 = fmax3f(m0, (e < nvalid) ? v[c] : -INFINITY, (e + 1 < nvalid) ? v[c + 1] : -INFINITY);
    m1 = fmax3f(m1, (e + 2 < nvalid) ? v[c + 2] : -INFINITY, (e + 3 < nvalid) ? v[c + 3] : -INFINITY);
    m2 = fmax3f(m2, (e + 4 < nvalid) ? v[c + 4] : -INFINITY, (e + 5 < nvalid) ? v[c + 5] : -INFINITY);
    m3 = fmax3f(m3, (e + 6 < nvalid) ? v[c + 6] : -INFINITY, (e + 7 < nvalid) ? v[c + 7] : -INFINITY);
  }
  return fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
}

// Sets the logits of columns >= nvalid (v[] holds columns col0 .. col0 + 63) to
// -inf, so their probabilities are 0; returns the maximum of the rest.
__device__ __forceinline__ float mask64(float (&v)[64], int col0, int nvalid) {
  float m0 = -INFINITY, m1 = m0;
#pragma unroll
  for (int c = 0; c < 64; c += 4) {
#pragma unroll
    for (int e = c; e < c + 4; ++e) v[e] = (col0 + e < nvalid) ? v[e] : -INFINITY;
    m0 = fmax3f(m0, v[c], v[c + 1]);
    m1 = fmax3f(m1, v[c + 2], v[c + 3]);
  }
  return fmaxf(m0, m1);
}

__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float (&v)[64]) {
  tmem_ld32(taddr, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
  tmem_ld32(taddr + 32, *reinterpret_cast<uint32_t(*)[32]>(&v[32]));
  tmem_ld_wait();
}

// Probabilities of 64 logits (columns col0 ..), p = 2^(v * sl2 + negm), packed
// to bf16 into 32 TMEM columns at p_taddr (16 at a time, so at most 16 packed
// words are live). Returns their fp32 sum. TAIL masks columns >= nvalid to
// probability 0.
template <bool TAIL>
__device__ __forceinline__ float exp64_store(const float (&v)[64], int col0, int nvalid, uint64_t scale2,
                                             uint64_t off2, uint32_t p_taddr) {
  uint64_t acc0 = f2_pack(0.f, 0.f), acc1 = acc0;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    uint32_t pk[16];
#pragma unroll
    for (int c = 0; c < 32; c += 4) {
      const int e = 32 * q + c;
      float a0, a1, b0, b1;
      f2_unpack(f2_fma(f2_pack(v[e], v[e + 1]), scale2, off2), a0, a1);
      f2_unpack(f2_fma(f2_pack(v[e + 2], v[e + 3]), scale2, off2), b0, b1);
      float p0 = ex2_approx(a0), p1 = ex2_approx(a1), p2 = ex2_approx(b0), p3 = ex2_approx(b1);
      if (TAIL) {
        const int g = col0 + e;
        p0 = (g < nvalid) ? p0 : 0.f;
        p1 = (g + 1 < nvalid) ? p1 : 0.f;
        p2 = (g + 2 < nvalid) ? p2 : 0.f;
        p3 = (g + 3 < nvalid) ? p3 : 0.f;
      }
      acc0 = f2_add(acc0, f2_pack(p0, p1));
      acc1 = f2_add(acc1, f2_pack(p2, p3));
      pk[c / 2] = pack_bf16x2(p0, p1);
      pk[c / 2 + 1] = pack_bf16x2(p2, p3);
    }
    tmem_st16(p_taddr + 16 * q, pk);
  }
  float s0, s1, s2, s3;
  f2_unpack(acc0, s0, s1);
  f2_unpack(acc1, s2, s3);
  return (s0 + s1) + (s2 + s3);
}

// Merge of a split item (the softmax threads of every rank; thread = row of
// tile t, rows of tile B follow A's). Each rank keeps its own share of the
// columns (D / nrank) and hands each other rank that one's share of its O, with
// its row maxima and sums, by bulk copies between the CTAs' shared memory (plain
// remote stores took 15k cycles for 128 KB). Then it scales the shares to the
// common maximum, adds them up in rank order, normalises and writes. Leaves the
// item's l and l_ref in l, lref. Two cluster barriers: every rank's tile buffers
// are idle and its parts written, before the copies; every part has arrived (the
// senders' buffers may go), before a CTA exits. So every rank sends and waits for
// what it receives, also after a wait of this CTA was given up. The parts are written before the
// first one: with the statistics exchanged ahead of them, behind a barrier of
// their own, the merge took 0.6 to 1.1 us longer.
template <int D>
__device__ __forceinline__ void merge_split(const WaitCtl& ctl, uint8_t* smem, uint64_t* parts_full, uint32_t o_t,
                                            bool ok, bool has_b, bool valid, int rank, int nrank, int t, int row,
                                            float m, float& l, float& lref, __nv_bfloat16* orow) {
  using C = Cfg<D>;
  const int nrows = has_b ? 2 * BM : BM, lrow = t * BM + row;
  const int cw = D / nrank;                         // columns per rank
  const uint32_t part_bytes = uint32_t(nrows) * cw * 4;  // [column / 4][row] of 16 bytes
  const uint32_t stat_bytes = uint32_t(nrows) * 16;
  uint8_t* send = smem;                             // parts for the other ranks, in rank order
  uint8_t* recv = smem + (nrank - 1) * part_bytes;  // parts from the other ranks, in rank order
  uint8_t* stats = smem + C::OFF_STATS;             // [rank][row] of (m, l, l_ref)
  constexpr uint32_t RANK_STATS = 2 * BM * 16;
  if (lrow == 0) mbar_arrive_expect_tx(parts_full, (nrank - 1) * (part_bytes + stat_bytes));
  named_bar_sync(4, 288);  // the producer's stores have read the tile buffers
  if (ok) {
    *reinterpret_cast<float4*>(stats + rank * RANK_STATS + lrow * 16) = make_float4(m, l, lref, 0.f);
    tc_fence_after();
#pragma unroll 1
    for (int c0 = 0; c0 < D; c0 += 16) {
      const int q = c0 / cw;
      if (q == rank) continue;
      uint32_t v[16];
      tmem_ld16(o_t + c0, v);
      tmem_ld_wait();
      uint4* dst = reinterpret_cast<uint4*>(send + (q - (q > rank ? 1 : 0)) * part_bytes) +
                   ((c0 - q * cw) >> 2) * nrows + lrow;
#pragma unroll
      for (int i = 0; i < 16; i += 4) dst[(i >> 2) * nrows] = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
  } else {  // what was given up is NaN on every rank
    *reinterpret_cast<float4*>(stats + rank * RANK_STATS + lrow * 16) = make_float4(0.f, NAN, NAN, 0.f);
  }
  fence_proxy_async_smem();  // the parts are next read by bulk copies
  cluster_sync_all();
  if (lrow == 0)
    for (int q = 0; q < nrank; ++q)
      if (q != rank) {
        const uint32_t bar = mapa_shared(smem_u32(parts_full), q);
        bulk_copy_to_cta(mapa_shared(smem_u32(stats + rank * RANK_STATS), q), stats + rank * RANK_STATS, stat_bytes, bar);
        bulk_copy_to_cta(mapa_shared(smem_u32(recv + (rank - (rank > q ? 1 : 0)) * part_bytes), q),
                         send + (q - (q > rank ? 1 : 0)) * part_bytes, part_bytes, bar);
      }
  const bool got = __all_sync(0xffffffffu, mbar_wait(parts_full, 0, ctl) ||
                                               mbar_wait_drain(parts_full, 0, ctl.budget_ns));
  __syncwarp();
  cluster_arrive();
  if (ok && got) {
    const float4* st = reinterpret_cast<const float4*>(stats) + lrow;
    float mx = st[0].x;
    for (int r = 1; r < nrank; ++r) mx = fmaxf(mx, st[r * 2 * BM].x);
    l = lref = 0.f;
    for (int r = 0; r < nrank; ++r) {
      const float4 v = st[r * 2 * BM];
      const float a = ex2_approx(v.x - mx);
      l = fmaf(v.y, a, l);
      lref = fmaf(v.z, a, lref);
    }
    const float inv_l = 1.f / l;
#pragma unroll 1
    for (int c0 = 0; c0 < cw; c0 += 16) {
      uint32_t v[16];
      float x[16];
      tmem_ld16(o_t + rank * cw + c0, v);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; ++i) x[i] = 0.f;
#pragma unroll 1
      for (int r = 0; r < nrank; ++r) {
        const float a = ex2_approx(st[r * 2 * BM].x - mx);
        const float4* src = reinterpret_cast<const float4*>(recv + (r - (r > rank ? 1 : 0)) * part_bytes) +
                            (c0 >> 2) * nrows + lrow;
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
          const float4 y = r == rank ? make_float4(__uint_as_float(v[i]), __uint_as_float(v[i + 1]),
                                                   __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]))
                                     : src[(i >> 2) * nrows];
          x[i] = fmaf(y.x, a, x[i]);
          x[i + 1] = fmaf(y.y, a, x[i + 1]);
          x[i + 2] = fmaf(y.z, a, x[i + 2]);
          x[i + 3] = fmaf(y.w, a, x[i + 3]);
        }
      }
      if (valid) {
        uint32_t pk[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) pk[i] = pack_bf16x2(x[2 * i] * inv_l, x[2 * i + 1] * inv_l);
        uint4* dst = reinterpret_cast<uint4*>(orow + rank * cw + c0);
        dst[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        dst[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
      }
    }
  }
  __syncwarp();
  cluster_wait();
}

// Merge of the two streams of an item (both warpgroups; thread = row): each
// reads the other's row maximum and sums (through the Q buffer), then combines
// both accumulators over its half of the columns. Leaves the item's l and l_ref
// in l, lref. The Q buffer is idle once the products are done, unless the item
// copies its Q tile into the cache slot (q_stored): then the producer says when
// that store has read it (barrier 4).
template <int D>
__device__ __forceinline__ void merge_dual(const WaitCtl& ctl, uint8_t* smem, uint64_t* o_done, uint32_t o_tmem,
                                           bool ok, bool second, bool q_stored, bool valid, int t, int row, float m,
                                           float& l, float& lref, __nv_bfloat16* orow) {
  float4* st = reinterpret_cast<float4*>(smem + Cfg<D, true>::OFF_Q);  // [stream][row]
  const bool done = __all_sync(0xffffffffu, mbar_wait(o_done, 0, ctl) && (!second || mbar_wait(o_done + 1, 0, ctl)));
  if (q_stored) named_bar_sync(4, 288);
  if (done) st[t * BM + row] = make_float4(m, ok ? l : NAN, lref, 0.f);
  named_bar_sync(3, 256);
  if (!done) return;
  tc_fence_after();
  const float4 s0 = st[row], s1 = st[BM + row];
  float a0 = 1.f, a1 = 0.f;
  l = s0.y;
  lref = s0.z;
  if (second) {
    const float mx = fmaxf(s0.x, s1.x);
    a0 = ex2_approx(s0.x - mx);
    a1 = ex2_approx(s1.x - mx);
    l = fmaf(s1.y, a1, s0.y * a0);
    lref = fmaf(s1.z, a1, s0.z * a0);
  }
  const float inv_l = 1.f / l;
  a0 *= inv_l;
  a1 *= inv_l;
#pragma unroll 1
  for (int c = t * (D / 2); c < (t + 1) * (D / 2); c += 16) {
    uint32_t v0[16], v1[16];
    tmem_ld16(o_tmem + c, v0);
    tmem_ld16(o_tmem + 128 + (second ? c : 0), v1);
    tmem_ld_wait();
    uint32_t pk[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float x = __uint_as_float(v0[2 * i]) * a0, y = __uint_as_float(v0[2 * i + 1]) * a0;
      if (second) {
        x = fmaf(__uint_as_float(v1[2 * i]), a1, x);
        y = fmaf(__uint_as_float(v1[2 * i + 1]), a1, y);
      }
      pk[i] = pack_bf16x2(x, y);
    }
    if (valid) {
      uint4* dst = reinterpret_cast<uint4*>(orow + c);
      dst[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
      dst[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
    }
  }
}

// SPLIT: a cluster of CTAs shares one item, each rank a contiguous range of
// its key tiles; the ranks' partial results meet in distributed shared memory.
// DUAL: an item is one Q tile; two streams, the even and the odd key tiles, take
// the places of the two tiles (the same issue order: one stream's products run
// while the other's softmax does) and are merged in TMEM at the end.
enum { KIND_PAIR = 0, KIND_SPLIT = 1, KIND_DUAL = 2 };
template <int D, int KIND>
__global__ void __launch_bounds__(NUM_THREADS, 1) joint_attn_kernel(const __grid_constant__ Params p) {
  constexpr bool SPLIT = KIND == KIND_SPLIT, DUAL = KIND == KIND_DUAL;
  using C = Cfg<D, DUAL>;
  constexpr int S = C::STAGES;
  // The rest of a call starts beside its whole rounds and depends on nothing of
  // theirs; it starts after their pdl_launch(), so after what they wait for: each
  // of their CTAs waits first, so what came before the call is complete and
  // written back when the rest starts, on SMs that the rounds' CTAs have left.
  // Waiting for the rounds themselves cost 2 to 12 us, as they end unevenly.
  if (!SPLIT || p.part != PART_REST) pdl_wait();
  pdl_launch();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = SPLIT ? int(cluster_rank()) : 0, nrank = SPLIT ? int(cluster_size()) : 1;
  int item = SPLIT ? int(blockIdx.x) / nrank : int(blockIdx.x), b0 = p.b0;
  if (!SPLIT && p.per_sample > 0) {
    const int s = item / p.per_sample;
    b0 += s;
    item -= s * p.per_sample;
  }
  const int lane_mode = (lane < p.nb && p.mode) ? p.mode[b0 + lane] : int(RA_MODE_FULL);

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;
  uint64_t* k_empty = bars + 1 + S;
  uint64_t* v_full = bars + 1 + 2 * S;
  uint64_t* v_empty = bars + 1 + 3 * S;
  uint64_t* s_full = bars + 1 + 4 * S;   // [tile]
  uint64_t* p_ready = bars + 3 + 4 * S;  // [tile]
  uint64_t* o_done = bars + 5 + 4 * S;   // [tile]
  uint64_t* drain = bars + 7 + 4 * S;
  uint64_t* parts_full = bars + 8 + 4 * S;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_MISC + 4);
  float* red = reinterpret_cast<float*>(smem + C::OFF_MISC + 16);  // [tile][quarter]

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < S; ++s) {
      mbar_init(k_full + s, 1);
      mbar_init(k_empty + s, 1);
      mbar_init(v_full + s, 1);
      mbar_init(v_empty + s, 1);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(s_full + t, 1);
      mbar_init(p_ready + t, 128);
      mbar_init(o_done + t, 1);
    }
    mbar_init(drain, 1);
    mbar_init(parts_full, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, C::TMEM_COLS);
  // The producer (which set the barriers up) goes on to its loads; the other
  // warps meet for the barriers and TMEM, and read its address in their roles
  // (read here for all, it cost the MMA loop 8 %). A round's first products start
  // earlier: 768 rows against 12544 keys 82.2 -> 81.2 us, image-edit reuse 435.5
  // -> 433.7.
  __syncwarp();
  if (warp == 0) {
    named_bar_arrive(5, NUM_THREADS);
  } else {
    tc_fence_before();
    named_bar_sync(5, NUM_THREADS);
    tc_fence_after();
  }
  // The item (the modes have arrived during the set-up): live items are
  // numbered sample-major, then head, then role and Q tiles (consecutive items
  // share their K/V tiles in L2).
  const uint32_t reuse = __ballot_sync(0xffffffffu, lane < p.nb && lane_mode == RA_MODE_REUSE);
  const int per_reuse = p.q_blocks[0] + p.q_blocks[2];
  {
    const int live = p.H * (p.nb * per_reuse + (p.nb - __popc(reuse)) * p.q_blocks[1]);
    const int rounds = p.part == PART_ALL ? live : round_items(live, p.slots, p.rest_max);
    if (p.part == PART_REST) item += rounds;
    if (item >= (p.part == PART_REST ? live : rounds)) {  // uniform over the cluster
      if (warp == 1) tmem_dealloc(*tmem_slot, C::TMEM_COLS);
      if (p.part == PART_REST && blockIdx.x == 0) pdl_wait();
      return;
    }
  }
  int bl = 0, per = 0;
  for (;; ++bl) {
    per = per_reuse + ((reuse >> bl) & 1 ? 0 : p.q_blocks[1]);
    if (item < p.H * per) break;
    item -= p.H * per;
  }
  const int b = b0 + bl, mode = __shfl_sync(0xffffffffu, lane_mode, bl);
  const uint32_t inv = p.per_inv[per == per_reuse ? 1 : 0];
  const int h = inv ? int(__umulhi(uint32_t(item), inv)) : item / per;
  const int first = item - h * per;  // 0: the first item of its (sample, head)
  int qb = first, role;
  const int n_ref_items = per - per_reuse;
  if (qb < p.q_blocks[0]) {
    role = 0;
  } else if (qb - p.q_blocks[0] < n_ref_items) {
    qb -= p.q_blocks[0];
    role = 1;
  } else {
    qb -= p.q_blocks[0] + n_ref_items;
    role = 2;
  }
  const int tileA = p.group * qb;
  const bool has_b = !DUAL && (tileA + 1) < p.q_tiles[role];  // a second Q tile
  const WaitCtl ctl{abort_flag, p.err_word, p.budget_ns};
  const int nkv_all = p.kv_tiles[0] + p.kv_tiles[1] + p.kv_tiles[2];
  const int j0 = SPLIT ? nkv_all * rank / nrank : 0;  // this CTA's first key tile
  const int nkv = SPLIT ? nkv_all * (rank + 1) / nrank - j0 : nkv_all;
  const bool second = DUAL ? nkv > 1 : has_b;  // the second softmax warpgroup works
  const bool store_q = p.fresh && refreshes(mode) && p.store_q && role == 1 && rank == 0;
  // Register split: warpgroup 0 (producer, MMA issuer, two idle warps) gives
  // up registers to the two softmax warpgroups: 4 x 56 + 8 x 224 = 12 x 168,
  // the launch allocation.
  if (warp < 4) {
    setmaxnreg_dec<56>();
    if (warp == 0) {
      if (lane == 0) {
        // ------------------------------------------------------------ TMA producer
        const bool fresh = p.fresh && refreshes(mode);
        const bool store_kv = fresh && p.store_kv && first == 0;
        const CUtensorMap* tq = (role == 1 && fresh) ? &p.tm_qf : &p.tm_q[role];
        if (fresh && first == 0 && h == 0 && rank == 0 && p.a_b) p.a_b[b] = p.step;
        tma_prefetch_desc(tq);
        for (int r = 0; r < 3; ++r)
          if (p.kv_tiles[r] > 0) {
            tma_prefetch_desc((r == 1 && fresh) ? &p.tm_kf : &p.tm_k[r]);
            tma_prefetch_desc((r == 1 && fresh) ? &p.tm_vf : &p.tm_v[r]);
          }
        int k_issued = 0, v_issued = 0;  // K / V tiles whose loads were issued
        uint32_t stored_stages = 0;      // stages whose last tile has a store that may still read it
        bool q_stored = !store_q;
        // Copy tile jj (loaded by now or soon) into the cache slot if it is a
        // reference tile; the Q tiles go with the first call.
        auto store_tiles = [&](int jj) -> bool {
          if (!q_stored) {
            if (!mbar_wait(q_full, 0, ctl)) return false;
            fence_proxy_async_smem();
            for (int t = 0; t < (has_b ? 2 : 1); ++t)
              for (int c = 0; c < C::CHUNKS; ++c)
                tma_store_4d(&p.tm_q[1], smem + C::OFF_Q + t * C::TILE_BYTES + c * C::CHUNK_BYTES, c * 64,
                             (tileA + t) * BM, h, b);
            bulk_commit();
            q_stored = true;
          }
          int r, row0;
          kv_tile(p, j0 + jj, r, row0);
          if (!store_kv || r != 1) return true;
          const int s = jj % S;
          const uint32_t ph = (jj / S) & 1;
          if (!mbar_wait(k_full + s, ph, ctl) || !mbar_wait(v_full + s, ph, ctl)) return false;
          fence_proxy_async_smem();
          for (int c = 0; c < C::CHUNKS; ++c) {
            tma_store_4d(&p.tm_k[1], smem + C::OFF_K + s * C::TILE_BYTES + c * C::CHUNK_BYTES, c * 64, row0, h, b);
            tma_store_4d(&p.tm_v[1], smem + C::OFF_V + s * C::TILE_BYTES + c * C::CHUNK_BYTES, c * 64, row0, h, b);
          }
          bulk_commit();
          stored_stages |= 1u << s;
          return true;
        };
        mbar_arrive_expect_tx(q_full, C::TILE_BYTES * (has_b ? 2 : 1));
        for (int t = 0; t < (has_b ? 2 : 1); ++t)
          for (int c = 0; c < C::CHUNKS; ++c)
            tma_load_4d(smem + C::OFF_Q + t * C::TILE_BYTES + c * C::CHUNK_BYTES, tq, q_full, c * 64,
                        (tileA + t) * BM, h, b);
        for (int j = 0; j < nkv; ++j) {
          const int s = j % S;
          const uint32_t ph = (j / S) & 1;
          int r, row0;
          kv_tile(p, j0 + j, r, row0);
          if (j >= S && !mbar_wait(k_empty + s, ph ^ 1, ctl)) break;
          if (stored_stages & (1u << s)) {  // stage s still feeds a store of tile j - S
            bulk_wait_read_all();
            stored_stages = 0;
          }
          mbar_arrive_expect_tx(k_full + s, C::TILE_BYTES);
          for (int c = 0; c < C::CHUNKS; ++c)
            tma_load_4d(smem + C::OFF_K + s * C::TILE_BYTES + c * C::CHUNK_BYTES,
                        (r == 1 && fresh) ? &p.tm_kf : &p.tm_k[r], k_full + s, c * 64, row0, h, b);
          ++k_issued;
          if (j >= S && !mbar_wait(v_empty + s, ph ^ 1, ctl)) break;
          mbar_arrive_expect_tx(v_full + s, C::TILE_BYTES);
          for (int c = 0; c < C::CHUNKS; ++c)
            tma_load_4d(smem + C::OFF_V + s * C::TILE_BYTES + c * C::CHUNK_BYTES,
                        (r == 1 && fresh) ? &p.tm_vf : &p.tm_v[r], v_full + s, c * 64, row0, h, b);
          ++v_issued;
          if (j >= 1 && (store_kv || store_q) && !store_tiles(j - 1)) break;
        }
        if ((store_kv || store_q) && !*abort_flag && v_issued == nkv) store_tiles(nkv - 1);
        // Shared memory must outlive the reads of every store issued.
        if (store_kv || store_q) bulk_wait_read_all();
        if (*abort_flag) {
          // Let every load this thread issued land before the CTA exits: stage s
          // received loads for j = s, s + S, ...; wait for the last one's phase.
          mbar_wait_drain(q_full, 0, p.budget_ns);
          for (int s = 0; s < S; ++s) {
            const int nk = (k_issued > s) ? (k_issued - s + S - 1) / S : 0;
            const int nv = (v_issued > s) ? (v_issued - s + S - 1) / S : 0;
            if (nk > 0) mbar_wait_drain(k_full + s, (nk - 1) & 1, p.budget_ns);
            if (nv > 0) mbar_wait_drain(v_full + s, (nv - 1) & 1, p.budget_ns);
          }
        }
      }
      if (DUAL && store_q) {  // the store of Q has read its buffer (merge_dual)
        __syncwarp();
        named_bar_arrive(4, 288);
      }
      if (lane == 0) bulk_wait_all();  // the cache slot is complete when the kernel is
    } else if (warp == 1) {
      if (lane == 0) {
        // ------------------------------------------------------------ MMA issuer
        constexpr uint32_t IDESC_QK = idesc_bf16_f32(BM, BN, 0, 0);  // Q, K both K-major
        constexpr uint32_t IDESC_PV = idesc_bf16_f32(BM, D, 0, 1);   // P K-major (TMEM), V MN-major
        const uint32_t tmem = *tmem_slot;
        const uint32_t sq = smem_u32(smem + C::OFF_Q);
        const uint32_t sk = smem_u32(smem + C::OFF_K);
        const uint32_t sv = smem_u32(smem + C::OFF_V);
        bool issued_any = false;
        // Q K_j^T into S_t, Q tile t (DUAL: the one tile).
        auto qk = [&](int j, int t) {
          const int s = j % S;
          umma_ss_ksteps<D / 16>(tmem + C::TM_S + 128 * t,
                                 sdesc_sw128(sq + (DUAL ? 0 : t) * C::TILE_BYTES, 16, 1024),
                                 sdesc_sw128(sk + s * C::TILE_BYTES, 16, 1024), IDESC_QK, 0u);
          umma_commit(s_full + t);
        };
        // O_t += P_t V_j. O_t is read only after the last P V (the epilogue); a
        // rescale reads it after s_full of the next tile, whose commit covers
        // this P V too.
        auto pv = [&](int j, int t, bool first, bool last) {
          const int s = j % S;
          umma_ts_ksteps8(tmem + C::TM_O + 128 * t, tmem + C::TM_S + 128 * t,
                          sdesc_sw128(sv + s * C::TILE_BYTES, C::CHUNK_BYTES, 1024), IDESC_PV, first ? 0u : 1u);
          if (last) umma_commit(o_done + t);
        };
        bool ok = mbar_wait(q_full, 0, ctl) && mbar_wait(k_full, 0, ctl);
        if (DUAL) {
          if (ok) {
            tc_fence_after();
            qk(0, 0);
            umma_commit(k_empty);
            issued_any = true;
            if (nkv > 1 && (ok = mbar_wait(k_full + 1, 0, ctl))) {
              tc_fence_after();
              qk(1, 1);
              umma_commit(k_empty + 1);
            }
          }
          for (int j = 0; ok && j < nkv; ++j) {
            const int s = j % S, t = j & 1;
            const bool next = j + 2 < nkv;  // S_t's next key tile
            if (!(ok = mbar_wait(v_full + s, (j / S) & 1, ctl))) break;
            if (next && !(ok = mbar_wait(k_full + (j + 2) % S, ((j + 2) / S) & 1, ctl))) break;
            if (!(ok = mbar_wait(p_ready + t, (j >> 1) & 1, ctl))) break;
            tc_fence_after();
            pv(j, t, j < 2, !next);
            umma_commit(v_empty + s);
            if (next) {
              qk(j + 2, t);  // S_t is free: PV_t was issued first
              umma_commit(k_empty + (j + 2) % S);
            }
          }
        } else {
          const int ntile = has_b ? 2 : 1;
          if (ok) {
            tc_fence_after();
            for (int t = 0; t < ntile; ++t) qk(0, t);
            umma_commit(k_empty);
            issued_any = true;
          }
          for (int j = 0; ok && j < nkv; ++j) {
            const int s = j % S;
            const bool next = j + 1 < nkv;
            if (!(ok = mbar_wait(v_full + s, (j / S) & 1, ctl))) break;
            if (next && !(ok = mbar_wait(k_full + (j + 1) % S, ((j + 1) / S) & 1, ctl))) break;
            for (int t = 0; t < ntile; ++t) {
              if (!(ok = mbar_wait(p_ready + t, j & 1, ctl))) break;
              tc_fence_after();
              pv(j, t, j == 0, !next);
              if (next) qk(j + 1, t);  // S_t is free: PV_t(j) was issued first
            }
            if (!ok) break;
            umma_commit(v_empty + s);
            if (next) umma_commit(k_empty + (j + 1) % S);
          }
        }
        if (!ok && issued_any) {
          umma_commit(drain);
          mbar_wait_drain(drain, 0, p.budget_ns);
        }
      }
    }
    if (SPLIT) {  // the softmax warps' cluster barriers (merge_split)
      __syncwarp();
      if (warp == 0) named_bar_sync(4, 288);
      cluster_sync_all();
      cluster_sync_all();
    }
  } else {
    setmaxnreg_inc<224>();
    const uint32_t tmem = *tmem_slot;
    // -------------------------------------------------------------- softmax
    const int t = (warp >= 8) ? 1 : 0;   // which Q tile this warpgroup owns
    // What only the epilogue needs waits in shared memory, not in registers.
    volatile int4* item_sh = reinterpret_cast<volatile int4*>(smem + C::OFF_ITEM) + (warp - 4);
    if (lane == 0) {
      item_sh->x = b;
      item_sh->y = h;
      item_sh->z = role + (store_q ? 4 : 0);
      item_sh->w = DUAL ? tileA : tileA + t;
    }
    __syncwarp();
    const int quarter = warp & 3;        // TMEM lane quarter this warp may access
    const int row = quarter * 32 + lane;
    const uint32_t lane_off = uint32_t(quarter * 32) << 16;
    const uint32_t s_t = tmem + lane_off + C::TM_S + 128 * t;
    const uint32_t o_t = tmem + lane_off + C::TM_O + 128 * t;
    const bool active = (t == 0) || second;
    const float sl2 = p.scale_log2;
    const float bias_l2 = (role == 2 && p.bias) ? p.bias[h] * kLog2e : 0.f;
    // The first keys may all be masked (a reference bias of -inf): the lowest
    // finite start keeps their probabilities 0.
    float m = kLowestMax, l = 0.f, lref = 0.f;
    bool ok = active;
    // DUAL: this warpgroup's key tiles are t, t + 2, ...
    for (int j = 0; ok && (DUAL ? 2 * j + t : j) < nkv; ++j) {
      int r, row0;
      kv_tile(p, DUAL ? 2 * j + t : j0 + j, r, row0);
      const int nvalid = min(BN, p.nk[r] - row0);
      const float badd = (r == 1) ? bias_l2 : 0.f;
      ok = __all_sync(0xffffffffu, mbar_wait(s_full + t, j & 1, ctl));
      if (!ok) break;
      tc_fence_after();
      // The previous P in S_t was consumed by PV_t(j-1), which completed before
      // QK_t(j) wrote S_t. The running max m only moves when the tile's max
      // exceeds it by more than 2^8 (then O, l, l_ref are rescaled by alpha).
      float alpha = 1.f;
      bool resc = false;
      // DUAL masks a tail tile's logits in registers and then takes the full
      // tile's path: a second path's cold instruction fetches cost a small launch
      // more (draft shape 16.6 -> 15.5 us); over many key tiles the extra code in
      // the loop costs more (image-edit refresh 1157 -> 1185 us).
      const bool tail = !DUAL && nvalid < BN;
      float rs;
      if (!tail) {
        // Full key tile: one TMEM read of the row with the hardware row max
        // (tcgen05.ld.red), probabilities straight from registers.
        float va[64], vb[64];
        float m0, m1, m2, m3;
        tmem_ldred32_max(s_t + 0, *reinterpret_cast<uint32_t(*)[32]>(&va[0]), m0);
        tmem_ldred32_max(s_t + 32, *reinterpret_cast<uint32_t(*)[32]>(&va[32]), m1);
        tmem_ldred32_max(s_t + 64, *reinterpret_cast<uint32_t(*)[32]>(&vb[0]), m2);
        tmem_ldred32_max(s_t + 96, *reinterpret_cast<uint32_t(*)[32]>(&vb[32]), m3);
        tmem_ld_wait();
        float mx = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
        if (DUAL && nvalid < BN) mx = fmaxf(mask64(va, 0, nvalid), mask64(vb, 64, nvalid));
        const float mt = fmaf(mx, sl2, badd);  // tile max, log2 units
        if (mt > m + kRescaleThresh) {
          alpha = ex2_approx(m - mt);  // 0 at the start
          resc = (j > 0);
          l *= alpha;
          lref *= alpha;
          m = mt;
        }
        // P_j over the first 64 columns of S_t: the logits are all in registers.
        const uint64_t scale2 = f2_pack(sl2, sl2);
        const uint64_t off2 = f2_pack(badd - m, badd - m);
        rs = exp64_store<false>(va, 0, BN, scale2, off2, s_t + 0);
        rs += exp64_store<false>(vb, 64, BN, scale2, off2, s_t + 32);
      } else {
        // Tail key tile: pass 1 takes the max over the valid columns only,
        // pass 2 re-reads the logits (half hf -> P columns [32 hf, 32 hf + 32),
        // never over logits still to be read).
        float mx = -INFINITY;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          float v[64];
          tmem_ld64(s_t + 64 * hf, v);
          mx = max64(v, 64 * hf, nvalid, mx);
        }
        const float mt = fmaf(mx, sl2, badd);
        if (mt > m + kRescaleThresh) {
          alpha = ex2_approx(m - mt);
          resc = (j > 0);
          l *= alpha;
          lref *= alpha;
          m = mt;
        }
        const uint64_t scale2 = f2_pack(sl2, sl2);
        const uint64_t off2 = f2_pack(badd - m, badd - m);
        rs = 0.f;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          float v[64];
          tmem_ld64(s_t + 64 * hf, v);
          rs += exp64_store<true>(v, 64 * hf, nvalid, scale2, off2, s_t + 32 * hf);
        }
      }
      l += rs;
      if (r == 1) lref += rs;
      if (__any_sync(0xffffffffu, resc)) {
        // PV_t(j-1) is complete: the commit that signalled s_full for this
        // tile tracks every MMA issued before QK_t(j).
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < D; c0 += 32) {
          uint32_t ov[32];
          tmem_ld32(o_t + c0, ov);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 32; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * alpha);
          tmem_st32(o_t + c0, ov);
        }
      }
      tmem_st_wait();
      tc_fence_before();
      mbar_arrive(p_ready + t);
    }
    if (ok) ok = __all_sync(0xffffffffu, mbar_wait(o_done + t, 0, ctl));
    const int eb = item_sh->x, eh = item_sh->y, erole = item_sh->z & 3, tile = item_sh->w;
    const bool q_stored = item_sh->z >= 4;
    const int grow = tile * BM + row;
    const bool valid = (active || DUAL) && grow < p.nq[erole];
    __nv_bfloat16* orow = p.o_ptr[erole] + eb * p.o_sb[erole] + eh * p.o_sh[erole] + int64_t(grow) * p.o_sn[erole];
    float inv_l;
    if (SPLIT) {
      merge_split<D>(ctl, smem, parts_full, o_t, ok && active, has_b, valid, rank, nrank, t, row, m, l, lref, orow);
      inv_l = 1.f / l;
    } else if (DUAL) {
      merge_dual<D>(ctl, smem, o_done, tmem + lane_off + C::TM_O, ok && active, second, q_stored, valid, t, row, m, l,
                    lref, orow);
      inv_l = 1.f / l;
    } else {
      inv_l = 1.f / l;
    }
    if (KIND == KIND_PAIR && ok) {
      tc_fence_after();
#pragma unroll
      for (int c0 = 0; c0 < D; c0 += 32) {
        uint32_t ov[32];
        tmem_ld32(o_t + c0, ov);
        tmem_ld_wait();
        uint32_t pk[16];
#pragma unroll
        for (int i = 0; i < 16; ++i)
          pk[i] = pack_bf16x2(__uint_as_float(ov[2 * i]) * inv_l, __uint_as_float(ov[2 * i + 1]) * inv_l);
        if (valid) {
          uint4* dst = reinterpret_cast<uint4*>(orow + c0);
          dst[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
          dst[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
          dst[2] = make_uint4(pk[8], pk[9], pk[10], pk[11]);
          dst[3] = make_uint4(pk[12], pk[13], pk[14], pk[15]);
        }
      }
    }
    // Per-tile mass partial: sum over the tile's mass rows of l_ref / l, in a
    // fixed order (warp butterfly, then quarters 0..3).
    const bool in_mass = ((erole == 2) || (erole == 0 && p.mass_rows == 1)) &&
                         (p.mass_stride <= 1 || grow % p.mass_stride == 0);
    float mv = (ok && valid && in_mass) ? lref * inv_l : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mv += __shfl_xor_sync(0xffffffffu, mv, o);
    if (lane == 0) red[4 * t + quarter] = mv;
    named_bar_sync(1 + t, 128);
    if (ok && active && erole != 1 && rank == 0 && !(DUAL && t == 1) && quarter == 0 && lane == 0) {
      const int idx = (erole == 0) ? tile : p.q_tiles[0] + tile;
      p.mass_partial[(int64_t(eb) * p.H + eh) * p.mpl + idx] =
          ((red[4 * t] + red[4 * t + 1]) + red[4 * t + 2]) + red[4 * t + 3];
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(*tmem_slot, C::TMEM_COLS);
  }
  // PART_REST starts beside the launch of the rounds (programmatic dependent
  // launch) and needs nothing of it, but must not complete before it: what
  // comes next in the stream waits for this launch alone.
  if (SPLIT && p.part == PART_REST && blockIdx.x == 0) pdl_wait();
}

// ------------------------------------------------------------------ host side
using Kernel = void (*)(Params);
struct KernelInfo {
  Kernel fn;
  int smem;
};
template <int D>
KernelInfo kernel_of(int kind) {
  if (kind == KIND_SPLIT) return {joint_attn_kernel<D, KIND_SPLIT>, Cfg<D>::SPLIT_ALLOC};
  if (kind == KIND_DUAL) return {joint_attn_kernel<D, KIND_DUAL>, Cfg<D, true>::SMEM_ALLOC};
  return {joint_attn_kernel<D, KIND_PAIR>, Cfg<D>::SMEM_ALLOC};
}
inline KernelInfo kernel_of(int d, int kind) { return d == 128 ? kernel_of<128>(kind) : kernel_of<64>(kind); }

// Clusters of cs CTAs of the split kernel that can run at once on the current
// device (they live inside one GPC, so the floorplan decides); cached per
// device, -1 with the error set on failure.
int max_clusters(int d, int cs) {
  static std::mutex mu;
  static int cache[64][2][MAX_SPLIT + 1];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    set_error("refadapt_joint_attn: no usable current device");
    return -1;
  }
  std::lock_guard<std::mutex> lk(mu);
  int& n = cache[dev][d == 128 ? 1 : 0][cs];
  if (n == 0) {
    const KernelInfo k = kernel_of(d, KIND_SPLIT);
    cudaError_t e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem);
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(cs, 1, 1);
    cfg.blockDim = dim3(NUM_THREADS, 1, 1);
    cfg.dynamicSmemBytes = k.smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int found = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&found, k.fn, &cfg);
    if (e != cudaSuccess) {
      set_error("refadapt_joint_attn: cluster occupancy query: %s", cudaGetErrorString(e));
      cudaGetLastError();
      return -1;
    }
    n = found > 0 ? found : -2;  // none fits
  }
  return n > 0 ? n : 0;
}

// Launches `items` items of p.part: one CTA each, or a cluster of cs CTAs each.
ra_status launch(const Params& p, int d, int64_t items, int cs, cudaStream_t st) {
  const char* who = "refadapt_joint_attn";
  if (items * cs > 2147483647) {
    set_error("%s: too many rows", who);
    return RA_EINVAL;
  }
  const KernelInfo k = kernel_of(d, p.group == 1 ? KIND_DUAL : cs > 1 ? KIND_SPLIT : KIND_PAIR);
  const ra_status as = ensure_dynamic_smem(reinterpret_cast<const void*>(k.fn), k.smem, who);
  if (as != RA_OK) return as;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(unsigned(items * cs), 1, 1);
  cfg.blockDim = dim3(NUM_THREADS, 1, 1);
  cfg.dynamicSmemBytes = k.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (cs > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = cs;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
  }
  attr[na++] = pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = na;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k.fn, p);
  if (e != cudaSuccess) {
    set_error("%s: launch failed: %s", who, cudaGetErrorString(e));
    cudaGetLastError();
    return RA_ECUDA;
  }
  return launch_status(who);
}

// How a call's items are launched.
struct Plan {
  int group;     // Q tiles per item: 2, or 1 with two streams of key tiles
  int cs;        // CTAs per split item, 1: nothing is split
  int rest_max;  // whole rounds unsplit and a rest of at most this many items split; 0: one launch
};

// Items of the launch's samples when every reference row runs / none does.
struct Live {
  int64_t most, least;
};
Live live_items(const Params& p, int group, int nb) {
  int64_t q[3];
  for (int r = 0; r < 3; ++r) q[r] = (p.q_tiles[r] + group - 1) / group;
  return {int64_t(p.H) * nb * (q[0] + q[1] + q[2]), int64_t(p.H) * nb * (q[0] + q[2])};
}

// The cheapest launch by a model of a CTA's time (microseconds, fitted to whole
// launches on a GB300): a fixed part (launch, mode load, set-up, first loads of
// all CTAs at once, cold instruction fetches, epilogue), so much per key tile of
// a pair of Q tiles, or per two key tiles of one Q tile in two streams, and the
// merge of a split item. What each form is for:
//   pairs unsplit         full rounds: the least traffic per product;
//   clusters              few items of many keys: every 8th target row of the
//                         image-edit shape (72 items of 98 key tiles) 81 us in
//                         clusters of two, 143 unsplit, 87 in two streams;
//   rounds, rest split    312 items of 26 key tiles (two rounds of 152 and 8)
//                         111 us, 131 in three rounds;
//   one tile, two streams items that fit few rounds: 8 heads, d = 64, of
//                         32 + 256 + 256 rows 8.2 against 11.4 us, of 77 + 1000
//                         + 500 rows 15.7 against 22.9 (half the latency per
//                         key, but twice the K and V traffic per product: 55
//                         against 46 us where it takes a second round).
// Modes are on the device, so a call with modes is weighed with all its
// reference rows, with none and (several samples) with half.
ra_status make_plan(const Params& p, int d, int nb, int slots, Plan* out) {
  const int n = p.kv_tiles[0] + p.kv_tiles[1] + p.kv_tiles[2];
  const bool wide = d == 128;
  const double merge = 6.8;
  auto cta = [&](int group, int cs) {
    if (group == 1) return (wide ? 7.5 : 5.5) + (n + 1) / 2 * (wide ? 1.64 : 1.25);
    return (wide ? 8.7 : 6.5) + (n + cs - 1) / cs * (wide ? 1.37 : 1.19) + (cs > 1 ? merge : 0.0);
  };
  auto rounds = [](int64_t items, int64_t width) { return double((items + width - 1) / width); };
  *out = Plan{2, 1, 0};
  double best = 0;
  const int least_group = n > 1 ? 1 : 2;  // one key tile has no second stream (24 heads of 128 rows 6.0 and 5.3 us)
  for (int group = 2; group >= least_group; --group) {
    const Live lv = live_items(p, group, nb);
    const int max_cs = group == 2 && nb <= MAX_SAMPLES ? MAX_SPLIT : 1;
    const int64_t cases[3] = {lv.most, p.mode ? lv.least : lv.most, (lv.most + lv.least) / 2};
    const int n_cases = p.mode ? (nb > 1 ? 3 : 2) : 1;
    for (int cs = 1; cs <= max_cs && cs <= n; cs *= 2) {
      int clusters = slots;
      if (cs > 1) {
        clusters = max_clusters(d, cs);
        if (clusters < 0) return RA_ECUDA;
        if (clusters == 0) continue;
      }
      int rest_max = 0;
      if (cs > 1 && lv.most >= slots) {
        rest_max = int(cta(group, 1) / cta(group, cs)) * clusters;
        if (rest_max > slots - 1) rest_max = slots - 1;
        if (rest_max == 0 || lv.most > 2147483647) continue;
      }
      double us = 0;
      for (int i = 0; i < n_cases; ++i) {
        const int64_t live = cases[i];
        if (rest_max == 0) {
          us += rounds(live, clusters) * cta(group, cs);
          continue;
        }
        const int64_t whole = round_items(int(live), slots, rest_max);
        us += rounds(whole, slots) * cta(group, 1);
        if (live > whole) us += rounds(live - whole, clusters) * cta(group, cs);
      }
      // A second launch has to promise a little more than the model's error, and
      // single tiles over many rounds more: with twice the traffic they end later
      // than they would alone (two samples of 24 heads, d = 64, 6525 keys: 715 us,
      // 623 in pairs).
      const double margin = rest_max > 0 ? 0.96 : group == 1 && lv.most > 3 * int64_t(slots) ? 0.90 : 0.99;
      if (best == 0 || us < margin * best) {
        best = us;
        *out = Plan{group, cs, rest_max};
      }
    }
  }
  return RA_OK;
}

// Plans and launches a call: in one go, unless its items are more than a grid has
// CTAs.
ra_status run(Params& p, int d, cudaStream_t st) {
  p.slots = num_sms();
  const int64_t most = int64_t(p.H) * (int64_t(p.q_tiles[0]) + p.q_tiles[1] + p.q_tiles[2]);  // items of a sample
  const int64_t fit = most > 0 ? 2147483647 / most : p.B;
  const int step = p.B <= MAX_SAMPLES ? p.B : int(fit < 1 ? 1 : fit < p.B ? fit : p.B);
  for (p.b0 = 0; p.b0 < p.B; p.b0 += step) {
    const int nb = p.B - p.b0 < step ? p.B - p.b0 : step;
    Plan plan;
    ra_status s = make_plan(p, d, nb, p.slots, &plan);
    if (s != RA_OK) return s;
    p.group = plan.group;
    for (int r = 0; r < 3; ++r) p.q_blocks[r] = (p.q_tiles[r] + plan.group - 1) / plan.group;
    for (int i = 0; i < 2; ++i) {
      // exact while item * per < 2^32 for every item < H * per
      const uint64_t per = uint64_t(p.q_blocks[0]) + p.q_blocks[2] + (i == 0 ? p.q_blocks[1] : 0);
      p.per_inv[i] = per > 1 && per * per * p.H < (uint64_t(1) << 32) ? uint32_t(((uint64_t(1) << 32) + per - 1) / per) : 0;
    }
    const Live lv = live_items(p, plan.group, nb);
    p.nb = nb;
    p.per_sample = 0;
    if (nb > MAX_SAMPLES) {
      p.nb = 1;
      p.per_sample = int32_t(lv.most / nb);
    }
    if (plan.rest_max == 0) {
      if (plan.group == 1) note_launch("two streams");
      else if (plan.cs > 1) note_launch("clusters of %d", plan.cs);
      else note_launch("pairs");
      p.part = PART_ALL;
      s = launch(p, d, lv.most, plan.cs, st);
    } else {
      // No modes leave more whole rounds than all items do, or a larger split rest.
      note_launch("rounds of pairs, up to %d in clusters of %d", plan.rest_max, plan.cs);
      p.rest_max = plan.rest_max;
      p.part = PART_ROUNDS;
      s = launch(p, d, round_items(int(lv.most), p.slots, p.rest_max), 1, st);
      p.part = PART_REST;
      if (s == RA_OK) s = launch(p, d, p.rest_max, plan.cs, st);
    }
    if (s != RA_OK) return s;
  }
  return RA_OK;
}

}  // namespace attn
}  // namespace ra

extern "C" int32_t refadapt_mass_partial_len(int32_t n_text, int32_t n_tgt) {
  if (n_text < 0 || n_tgt < 0) return 0;
  return (n_text + RA_MASS_TILE_ROWS - 1) / RA_MASS_TILE_ROWS + (n_tgt + RA_MASS_TILE_ROWS - 1) / RA_MASS_TILE_ROWS;
}

extern "C" ra_status refadapt_joint_attn(const ra_attn_args* a, void* stream) {
  using namespace ra;
  using namespace ra::attn;
  clear_error();
  if (!a) {
    set_error("refadapt_joint_attn: args is NULL");
    return RA_EINVAL;
  }
  if (a->d != 64 && a->d != 128) {
    set_error("refadapt_joint_attn: d = %d (supported: 64, 128)", a->d);
    return RA_EINVAL;
  }
  if (a->B < 1 || a->H < 1 || a->B > 65535 || a->H > 65535) {
    set_error("refadapt_joint_attn: B = %d, H = %d out of range", a->B, a->H);
    return RA_EINVAL;
  }
  if (a->mass_rows != 0 && a->mass_rows != 1) {
    set_error("refadapt_joint_attn: mass_rows must be 0 or 1");
    return RA_EINVAL;
  }
  if (a->mass_row_stride < 0) {
    set_error("refadapt_joint_attn: mass_row_stride must be >= 0");
    return RA_EINVAL;
  }
  if (!(a->softmax_scale >= 0.f) || std::isinf(a->softmax_scale)) {
    set_error("refadapt_joint_attn: softmax_scale must be finite and >= 0");
    return RA_EINVAL;
  }
  if (!a->mass_partial) {
    set_error("refadapt_joint_attn: mass_partial is NULL");
    return RA_EINVAL;
  }
  static const char* names[3] = {"text", "ref", "tgt"};
  char what[64];
  Params p;
  std::memset(&p, 0, sizeof(p));
  bool ref_rows = true;
  for (int r = 0; r < 3; ++r) {
    if (a->v[r].n != a->k[r].n || a->o[r].n != a->q[r].n) {
      set_error("refadapt_joint_attn: %s: k and v (key rows) or q and o (query rows) disagree on n", names[r]);
      return RA_EINVAL;
    }
    const ra_seg* segs[4] = {&a->q[r], &a->k[r], &a->v[r], &a->o[r]};
    const char* kinds[4] = {"q", "k", "v", "o"};
    for (int i = 0; i < 4; ++i) {
      snprintf(what, sizeof(what), "refadapt_joint_attn: %s[%s]", kinds[i], names[r]);
      const bool may_skip = (r == RA_REF) && (i == 0 || i == 3);
      if (may_skip && segs[i]->ptr == nullptr) {
        ref_rows = false;
        continue;
      }
      if (!check_seg(*segs[i], what)) return RA_EINVAL;
    }
  }
  if (a->k[RA_TGT].n < 1) {
    set_error("refadapt_joint_attn: the target segment needs at least one key row");
    return RA_EINVAL;
  }
  const int d = a->d;
  for (int r = 0; r < 3; ++r) {
    const int nk = a->k[r].n, nq = (r == RA_REF && !ref_rows) ? 0 : a->q[r].n;
    p.nk[r] = nk;
    p.nq[r] = nq;
    p.kv_tiles[r] = (nk + BN - 1) / BN;
    p.q_tiles[r] = (nq + BM - 1) / BM;
    if (nk > 0 && (!encode_seg(&p.tm_k[r], a->k[r], a->B, a->H, d, 64, BN, true) ||
                   !encode_seg(&p.tm_v[r], a->v[r], a->B, a->H, d, 64, BN, true)))
      return RA_EINVAL;
    if (nq == 0) continue;
    if (!encode_seg(&p.tm_q[r], a->q[r], a->B, a->H, d, 64, BM, true)) return RA_EINVAL;
    p.o_ptr[r] = static_cast<__nv_bfloat16*>(a->o[r].ptr);
    p.o_sb[r] = a->o[r].stride_b;
    p.o_sh[r] = a->o[r].stride_h;
    p.o_sn[r] = a->o[r].stride_n;
  }
  if (a->ref_fresh_q.ptr != nullptr || a->ref_fresh_k.ptr != nullptr || a->ref_fresh_v.ptr != nullptr ||
      a->a_b != nullptr) {
    // Fused cache update: this step's reference rows, read by refreshing
    // samples and copied into the segments k/v/q[RA_REF] point at.
    const ra_seg* fr[3] = {&a->ref_fresh_q, &a->ref_fresh_k, &a->ref_fresh_v};
    const ra_seg* ca[3] = {&a->q[RA_REF], &a->k[RA_REF], &a->v[RA_REF]};
    const char* kinds[3] = {"q", "k", "v"};
    bool copy[3] = {false, false, false};
    for (int i = 0; i < 3; ++i) {
      if (i == 0 && !ref_rows) {
        if (fr[0]->ptr != nullptr || fr[0]->n != 0) {
          set_error("refadapt_joint_attn: ref_fresh_q given without reference query rows (q[ref] is NULL)");
          return RA_EINVAL;
        }
        continue;
      }
      snprintf(what, sizeof(what), "refadapt_joint_attn: ref_fresh_%s", kinds[i]);
      if (!check_seg(*fr[i], what)) return RA_EINVAL;
      if (fr[i]->n != ca[i]->n) {
        set_error("refadapt_joint_attn: ref_fresh_%s has n = %d, %s[ref] has %d", kinds[i], fr[i]->n, kinds[i],
                  ca[i]->n);
        return RA_EINVAL;
      }
      if (fr[i]->ptr == ca[i]->ptr) {
        if (fr[i]->stride_b != ca[i]->stride_b || fr[i]->stride_h != ca[i]->stride_h ||
            fr[i]->stride_n != ca[i]->stride_n) {
          set_error("refadapt_joint_attn: ref_fresh_%s shares its pointer with %s[ref] but not its strides",
                    kinds[i], kinds[i]);
          return RA_EINVAL;
        }
        continue;  // read in place
      }
      copy[i] = true;
      if (fr[i]->n > 0) {
        CUtensorMap* tm = (i == 0) ? &p.tm_qf : (i == 1) ? &p.tm_kf : &p.tm_vf;
        if (!encode_seg(tm, *fr[i], a->B, a->H, d, 64, (i == 0) ? BM : BN, true)) return RA_EINVAL;
      }
    }
    if (copy[1] != copy[2]) {
      set_error("refadapt_joint_attn: ref_fresh_k and ref_fresh_v must both be in place or both be copied");
      return RA_EINVAL;
    }
    // Segments read in place keep their own maps as the fresh ones.
    if (!copy[0]) p.tm_qf = p.tm_q[RA_REF];
    if (!copy[1]) {
      p.tm_kf = p.tm_k[RA_REF];
      p.tm_vf = p.tm_v[RA_REF];
    }
    p.fresh = 1;
    p.store_kv = copy[1] ? 1 : 0;
    p.store_q = copy[0] ? 1 : 0;
    p.a_b = a->a_b;
    p.step = a->step;
  }
  p.B = a->B;
  p.H = a->H;
  p.mass_rows = a->mass_rows;
  p.mass_stride = a->mass_row_stride;
  p.mpl = refadapt_mass_partial_len(a->q[RA_TEXT].n, a->q[RA_TGT].n);
  const float scale = a->softmax_scale > 0.f ? a->softmax_scale : 1.0f / std::sqrt(float(d));
  p.scale_log2 = scale * kLog2e;
  p.bias = a->ref_logit_bias;
  p.mode = a->mode;
  p.mass_partial = a->mass_partial;
  p.err_word = a->err_word;
  p.budget_ns = wait_budget_ns();
  return run(p, d, static_cast<cudaStream_t>(stream));
}
