// refadapt_ln_modulate: the DiT block's modulated LayerNorm,
//   x = (h - mean(h)) / sqrt(var(h) + eps) * (1 + scale[sample]) + shift[sample]
// over the C features of every row (no affine of its own; the AdaLN shift and
// scale of the block, stream and sample modulate it). Reference segments may be
// gated on the per-sample mode (skipped when REUSE).
//
// HBM-bound: 4 C bytes per row. One warp per row, the row in registers as
// packed bf16, mean and variance in fp32 in two passes over them. What keeps
// HBM busy (ln_mod_kernel): one persistent CTA per SM that takes a contiguous
// share of the live rows, each warp with a ring of rows that bulk copies fill
// ahead of it; and the modulation (8 C bytes, twice a row's own bytes) held in
// shared memory per (segment, sample) piece instead of read through L1 for every
// row. At C = 3072: 12544 rows 34.8 -> 25.8 us (6 TB/s; a plain copy of them
// 24.3), 4352 rows 12.3 -> 9.3, 1024 rows 6.4 -> 4.0, against one row per warp and
// no ring (ln_row_kernel). Its set-up and its walk over the pieces cost more where
// rows are short or samples many: two rows of 256 1.3 us by row, 1.9 persistent; 64
// samples of 1 and of 205 rows of 2560 47 and 242. by_row() chooses; a row's
// arithmetic is the same in both.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstring>

#include "api_common.h"
#include "tc_ptx.cuh"

namespace ra {
namespace lnmod {

constexpr int MAX_GROUPS = 16;  // 8 features per lane per group: C <= 4096

// Shared memory of a CTA: shift, 1 + scale (fp32, C each), a ring of S rows per
// warp, the rings' barriers. Above C = 3072 twelve warps leave room for two rows
// each.
template <int G>
struct Layout {
  static constexpr int ROW_BYTES = 512 * G;
  static constexpr int MOD_BYTES = 2 * 1024 * G;
  static constexpr int WARPS = G > 12 ? 12 : 16;
  static constexpr int FIT = (232448 - MOD_BYTES - 1024) / (WARPS * ROW_BYTES);
  static constexpr int S = FIT > 4 ? 4 : FIT;
  static constexpr int OFF_BAR = MOD_BYTES + WARPS * S * ROW_BYTES;
  static constexpr int BYTES = OFF_BAR + WARPS * S * 8;
  static_assert(S >= 2 && BYTES <= 232448, "shared memory budget");
};

struct Seg {
  const __nv_bfloat16* h;
  int64_t h_ss, h_sr;
  __nv_bfloat16* x;
  int64_t x_ss, x_sr;
  const float* shift;
  const float* scale;
  int64_t mod_ss;
  int32_t rows, gated;
};

struct Params {
  Seg seg[3];
  int32_t n_seg, B, C, groups;
  uint64_t budget_ns;
  float eps;
  const int32_t* mode;
};

__device__ __forceinline__ bool live(const Params& p, int g, int s) {
  return !p.seg[g].gated || p.mode[s] != RA_MODE_REUSE;
}

// Live rows in order: segments, samples within, rows within. A piece is the
// rows of one live (segment, sample), from row `begin` of the order on.
struct Piece {
  int g = 0, s = 0, begin = 0;
  // Moves to the piece that holds row i (i at or past begin, below the total).
  __device__ __forceinline__ void seek(const Params& p, int i) {
    while (i - begin >= p.seg[g].rows || !live(p, g, s)) {
      if (live(p, g, s)) begin += p.seg[g].rows;
      if (++s == p.B || p.seg[g].rows == 0) {
        s = 0;
        ++g;
      }
    }
  }
  // The same over many samples (the whole warp, from a segment's first): those of
  // a segment that is not gated are counted off by a division, others 32 at a
  // time. seek() takes 0.1 us for each (256 samples of one row: 50 us).
  __device__ __forceinline__ void jump(const Params& p, int i) {
    for (;; ++g, s = 0) {
      const int rows = p.seg[g].rows;
      if (rows == 0) continue;
      const int k = int(uint32_t(i - begin) / uint32_t(rows));  // live samples to pass
      if (!p.seg[g].gated) {
        s = min(k, p.B);
        begin += s * rows;
        if (s < p.B) return;
        continue;
      }
      int passed = 0;
      for (; s < p.B; s += 32) {
        const int t = s + (threadIdx.x & 31);
        const int n = __popc(__ballot_sync(0xffffffffu, t < p.B && live(p, g, t)));
        if (passed + n > k) break;
        passed += n;
      }
      begin += passed * rows;
      if (s < p.B) return;  // one of the 32 samples from s on: seek() finds it
    }
  }
};

// A warp whose own copy of row i did not end within the budget: it lets the
// copies on their way (of its next S - 1 rows) land, and its rows from i on
// become NaN.
template <int G>
__device__ __noinline__ void give_up(const Params& p, uint64_t* full, int stage, uint32_t phase, int i, int hi) {
  using L = Layout<G>;
  for (int k = 1; k < L::S && i + k * L::WARPS < hi; ++k) {
    if (++stage == L::S) {
      stage = 0;
      phase ^= 1;
    }
    mbar_wait_drain(full + stage, phase, p.budget_ns);
  }
  Piece w;
  for (; i < hi; i += L::WARPS) {
    w.seek(p, i);
    const Seg& sg = p.seg[w.g];
    uint4* dst = reinterpret_cast<uint4*>(sg.x + w.s * sg.x_ss + int64_t(i - w.begin) * sg.x_sr);
    for (int q = 0; q < G; ++q) dst[q * 32 + (threadIdx.x & 31)] = make_uint4(~0u, ~0u, ~0u, ~0u);
  }
}

// -mean and 1 / standard deviation of a warp's row (8-feature group q of the
// lane in u[q]), each twice in a pair.
template <int G>
__device__ __forceinline__ void row_stats(const uint4 (&u)[G], int C, float eps, uint64_t& neg_mean, uint64_t& rstd2) {
  uint64_t acc0 = f2_pack(0.f, 0.f), acc1 = acc0;
#pragma unroll
  for (int q = 0; q < G; ++q) {
    acc0 = f2_add(acc0, f2_add(bf2_unpack(u[q].x), bf2_unpack(u[q].y)));
    acc1 = f2_add(acc1, f2_add(bf2_unpack(u[q].z), bf2_unpack(u[q].w)));
  }
  float a0, a1;
  f2_unpack(f2_add(acc0, acc1), a0, a1);
  float sum = a0 + a1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const float mean = sum / float(C);
  neg_mean = f2_pack(-mean, -mean);
  acc0 = acc1 = f2_pack(0.f, 0.f);
#pragma unroll
  for (int q = 0; q < G; ++q) {
    const uint32_t e[4] = {u[q].x, u[q].y, u[q].z, u[q].w};
#pragma unroll
    for (int k = 0; k < 4; k += 2) {
      const uint64_t d0 = f2_add(bf2_unpack(e[k]), neg_mean), d1 = f2_add(bf2_unpack(e[k + 1]), neg_mean);
      acc0 = f2_fma(d0, d0, acc0);
      acc1 = f2_fma(d1, d1, acc1);
    }
  }
  f2_unpack(f2_add(acc0, acc1), a0, a1);
  float sq = a0 + a1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  const float rstd = rsqrtf(sq / float(C) + eps);
  rstd2 = f2_pack(rstd, rstd);
}

// Eight modulated features: sc is 1 + scale, sh the shift, four features each.
__device__ __forceinline__ uint4 row_out(uint4 u, uint64_t neg_mean, uint64_t rstd2, ulonglong2 sc0, ulonglong2 sc1,
                                         ulonglong2 sh0, ulonglong2 sh1) {
  auto two = [&](uint32_t e, uint64_t sc, uint64_t sh) {
    float y0, y1;
    f2_unpack(f2_fma(f2_mul(f2_add(bf2_unpack(e), neg_mean), rstd2), sc, sh), y0, y1);
    return pack_bf16x2(y0, y1);
  };
  return make_uint4(two(u.x, sc0.x, sh0.x), two(u.y, sc0.y, sh0.y), two(u.z, sc1.x, sh1.x), two(u.w, sc1.y, sh1.y));
}

// One row per warp, the modulation read through L1: for calls of few rows, or of
// few rows per sample. Every row of the call has a warp, a dead one's ends.
template <int G>
constexpr int kRowWarps = G < 3 ? 8 : 4;
template <int G>
__global__ void __launch_bounds__(32 * kRowWarps<G>) ln_row_kernel(const __grid_constant__ Params p) {
  pdl_launch();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  int64_t i = int64_t(blockIdx.x) * kRowWarps<G> + (threadIdx.x >> 5);
  int g = 0;
  for (; g < p.n_seg && i >= int64_t(p.B) * p.seg[g].rows; ++g) i -= int64_t(p.B) * p.seg[g].rows;
  if (g == p.n_seg) return;
  const Seg& sg = p.seg[g];
  const int s = int(i / sg.rows);
  if (!live(p, g, s)) return;
  const int64_t r = i - int64_t(s) * sg.rows;
  uint4 u[G];
  const uint4* src = reinterpret_cast<const uint4*>(sg.h + s * sg.h_ss + r * sg.h_sr);
#pragma unroll
  for (int q = 0; q < G; ++q) u[q] = src[q * 32 + lane];
  const ulonglong2* shift = reinterpret_cast<const ulonglong2*>(sg.shift + s * sg.mod_ss) + 2 * lane;
  const ulonglong2* scale = reinterpret_cast<const ulonglong2*>(sg.scale + s * sg.mod_ss) + 2 * lane;
  uint4* dst = reinterpret_cast<uint4*>(sg.x + s * sg.x_ss + r * sg.x_sr);
  const uint64_t one = f2_pack(1.f, 1.f);
  // Modulation of the next AHEAD groups: no load waits behind a store of x.
  constexpr int AHEAD = G < 3 ? G : 3;
  ulonglong2 m[AHEAD][4];
  auto fetch = [&](int q) {
    ulonglong2(&v)[4] = m[q % AHEAD];
    v[0] = scale[64 * q], v[1] = scale[64 * q + 1], v[2] = shift[64 * q], v[3] = shift[64 * q + 1];
  };
#pragma unroll
  for (int q = 0; q < AHEAD; ++q) fetch(q);
  uint64_t neg_mean, rstd2;
  row_stats<G>(u, p.C, p.eps, neg_mean, rstd2);
#pragma unroll
  for (int q = 0; q < G; ++q) {
    ulonglong2(&v)[4] = m[q % AHEAD];
#pragma unroll
    for (int z = 0; z < 2; ++z) v[z].x = f2_add(v[z].x, one), v[z].y = f2_add(v[z].y, one);
    const uint4 y = row_out(u[q], neg_mean, rstd2, v[0], v[1], v[2], v[3]);
    if (q + AHEAD < G) fetch(q + AHEAD);
    dst[q * 32 + lane] = y;
  }
}

template <int G>  // 8-feature groups per lane: C = 256 G
__global__ void __launch_bounds__(32 * Layout<G>::WARPS, 1) ln_mod_kernel(const __grid_constant__ Params p) {
  using L = Layout<G>;
  constexpr int S = L::S, W = L::WARPS;
  extern __shared__ __align__(128) uint8_t smem[];
  float* shift_sh = reinterpret_cast<float*>(smem);
  float* scale_sh = shift_sh + 256 * G;
  pdl_launch();
  pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* ring = smem + L::MOD_BYTES + warp * S * L::ROW_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + L::OFF_BAR) + warp * S;
  if (lane < S) mbar_init(full + lane, 1);
  fence_mbar_init();
  __syncwarp();
  // Live rows of the call (the modes are on the device), and this CTA's share.
  int total = 0;
  for (int g = 0; g < p.n_seg; ++g) {
    int n = p.B;
    if (p.seg[g].gated) {
      n = 0;
      for (int s0 = 0; s0 < p.B; s0 += 32)
        n += __popc(__ballot_sync(0xffffffffu, s0 + lane < p.B && live(p, g, s0 + lane)));
    }
    total += n * p.seg[g].rows;
  }
  const int share = total / int(gridDim.x), more = total - share * int(gridDim.x), cta = int(blockIdx.x);
  const int lo = share * cta + min(cta, more);
  const int hi = lo + share + (cta < more ? 1 : 0);
  if (lo == hi) return;
  Piece ld;
  if (p.B > 4) ld.jump(p, lo);
  Piece w = ld;
  int i = lo + warp, ld_i = i;  // this warp's rows: lo + warp, + W, ...; loads run up to S rows ahead
  auto load = [&](int stage) {
    if (ld_i < hi && lane == 0) {
      ld.seek(p, ld_i);
      const Seg& sg = p.seg[ld.g];
      mbar_arrive_expect_tx(full + stage, L::ROW_BYTES);
      bulk_load(ring + stage * L::ROW_BYTES, sg.h + ld.s * sg.h_ss + int64_t(ld_i - ld.begin) * sg.h_sr, L::ROW_BYTES,
                full + stage);
    }
    ld_i += W;
  };
  for (int k = 0; k < S; ++k) load(k);
  int stage = 0;
  uint32_t phase = 0;
  for (int piece_lo = lo; piece_lo < hi;) {
    w.seek(p, piece_lo);
    const Seg& sg = p.seg[w.g];
    const int piece_hi = min(hi, w.begin + sg.rows);
    if (piece_lo != lo) __syncthreads();  // every warp is done with the last piece's modulation
    const float* shift = sg.shift + w.s * sg.mod_ss;
    const float* scale = sg.scale + w.s * sg.mod_ss;
    for (int f = threadIdx.x; f < 64 * G; f += 32 * W) {
      // Four columns: half f % 2 of lane (f / 2) % 32 in group f / 64; kept as
      // [group][half][lane], so the rows' 16-byte reads have no bank conflicts.
      const int at = ((f >> 6) * 2 + (f & 1)) * 32 + ((f >> 1) & 31);
      const float4 sh = reinterpret_cast<const float4*>(shift)[f];
      float4 sc = reinterpret_cast<const float4*>(scale)[f];
      sc.x += 1.f, sc.y += 1.f, sc.z += 1.f, sc.w += 1.f;
      reinterpret_cast<float4*>(shift_sh)[at] = sh;
      reinterpret_cast<float4*>(scale_sh)[at] = sc;
    }
    __syncthreads();
    for (; i < piece_hi; i += W) {
      if (!__all_sync(0xffffffffu, mbar_wait_drain(full + stage, phase, p.budget_ns))) {
        give_up<G>(p, full, stage, phase, i, hi);
        i = hi;
        break;
      }
      uint4 u[G];
      const uint4* src = reinterpret_cast<const uint4*>(ring + stage * L::ROW_BYTES);
#pragma unroll
      for (int q = 0; q < G; ++q) u[q] = src[q * 32 + lane];
      __syncwarp();  // the row is in registers: its stage takes the next one
      load(stage);
      if (++stage == S) {
        stage = 0;
        phase ^= 1;
      }
      uint64_t neg_mean, rstd2;
      row_stats<G>(u, p.C, p.eps, neg_mean, rstd2);
      uint4* dst = reinterpret_cast<uint4*>(sg.x + w.s * sg.x_ss + int64_t(i - w.begin) * sg.x_sr);
#pragma unroll
      for (int q = 0; q < G; ++q) {
        const ulonglong2* sh = reinterpret_cast<const ulonglong2*>(shift_sh) + 2 * q * 32 + lane;
        const ulonglong2* sc = reinterpret_cast<const ulonglong2*>(scale_sh) + 2 * q * 32 + lane;
        dst[q * 32 + lane] = row_out(u[q], neg_mean, rstd2, sc[0], sc[32], sh[0], sh[32]);
      }
    }
    piece_lo = piece_hi;
  }
}

ra_status launch(void (*fn)(Params), const Params& p, int64_t ctas, int threads, int smem, cudaStream_t st) {
  if (smem > 0) {
    const ra_status as = ensure_dynamic_smem(reinterpret_cast<const void*>(fn), smem, "refadapt_ln_modulate");
    if (as != RA_OK) return as;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(ctas));
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr = pdl_attribute();
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, fn, p);
  if (e != cudaSuccess) {
    set_error("refadapt_ln_modulate: launch failed: %s", cudaGetErrorString(e));
    cudaGetLastError();
    return RA_ECUDA;
  }
  return launch_status("refadapt_ln_modulate");
}

template <int G>
ra_status run(const Params& p, int64_t rows, bool one_row_per_warp, cudaStream_t st) {
  using L = Layout<G>;
  note_launch(one_row_per_warp ? "one row per warp" : "persistent");
  if (one_row_per_warp)
    return launch(ln_row_kernel<G>, p, (rows + kRowWarps<G> - 1) / kRowWarps<G>, 32 * kRowWarps<G>, 0, st);
  const int64_t sms = num_sms();
  return launch(ln_mod_kernel<G>, p, rows < sms ? rows : sms, 32 * L::WARPS, L::BYTES, st);
}

// One row per warp, or the persistent kernel: models of the two (microseconds,
// fitted at C = 256 to 4096, 1 to 94,000 rows and 1 to 768 pieces). A CTA of the
// persistent kernel pays 3.5 us for every further piece of its share, so a
// segment of few rows per sample and many samples is better off by row (64
// samples of 1 and of 205 rows of 2560: 242 us persistent, 47 by row).
bool by_row(const Params& p, int64_t rows, int sms) {
  const double c = p.C / 1024.0, k = rows / 1000.0, share = double(rows) / sms;
  double crossed = 0;  // pieces of the CTA that meets most
  int segs = 0;
  for (int g = 0; g < p.n_seg; ++g) {
    if (p.seg[g].rows == 0) continue;
    const double n = share / p.seg[g].rows < p.B ? share / p.seg[g].rows : p.B;
    crossed = n > crossed ? n : crossed;
    ++segs;
  }
  const double walk = 3.5 * crossed + (p.B > 4 ? 0.9 : 0.19 * p.B) * segs;
  const double row = 1.2 + 0.37 * c + k * (c > 0.28 ? 0.95 * c : 0.26);
  const double persistent = 1.75 + 0.33 * c + walk + k * (c > 0.47 ? 0.62 * c : 0.29);
  return row < persistent || rows > 2147483647 - 65536;  // the persistent kernel counts rows in 32 bits
}

bool aligned16(const void* ptr) { return (reinterpret_cast<uintptr_t>(ptr) & 15u) == 0; }

}  // namespace lnmod
}  // namespace ra

extern "C" ra_status refadapt_ln_modulate(const ra_lnmod_args* a, void* stream) {
  using namespace ra;
  using namespace ra::lnmod;
  clear_error();
  if (!a) {
    set_error("refadapt_ln_modulate: args is NULL");
    return RA_EINVAL;
  }
  if (a->B < 1 || a->n_seg < 1 || a->n_seg > 3 || a->C < 256 || a->C % 256 != 0 || a->C > 256 * MAX_GROUPS ||
      !(a->eps >= 0.f)) {
    set_error("refadapt_ln_modulate: need B >= 1, 1 <= n_seg <= 3, C a multiple of 256 in [256, 4096], "
              "eps >= 0 (B=%d n_seg=%d C=%d)", a->B, a->n_seg, a->C);
    return RA_EINVAL;
  }
  Params p;
  std::memset(&p, 0, sizeof(p));
  p.n_seg = a->n_seg;
  p.B = a->B;
  p.C = a->C;
  p.groups = a->C / 256;
  p.eps = a->eps;
  p.mode = a->mode;
  p.budget_ns = wait_budget_ns();
  int64_t rows = 0;
  for (int g = 0; g < a->n_seg; ++g) {
    const ra_lnmod_seg& s = a->seg[g];
    Seg& d = p.seg[g];
    if (s.rows < 0) {
      set_error("refadapt_ln_modulate: seg %d rows < 0", g);
      return RA_EINVAL;
    }
    d.rows = s.rows;
    d.gated = s.gated ? 1 : 0;
    if (s.gated && !a->mode) {
      set_error("refadapt_ln_modulate: seg %d is gated but mode is NULL", g);
      return RA_EINVAL;
    }
    if (s.rows == 0) continue;
    if (!s.h || !s.x || !s.shift || !s.scale || !aligned16(s.h) || !aligned16(s.x) || !aligned16(s.shift) ||
        !aligned16(s.scale) || s.h_stride_r % 8 || s.h_stride_s % 8 || s.x_stride_r % 8 || s.x_stride_s % 8 ||
        s.mod_stride_s % 4 || s.h_stride_r < a->C || s.x_stride_r < a->C) {
      set_error("refadapt_ln_modulate: seg %d: pointers must be 16-byte aligned, row strides >= C and "
                "multiples of 8 elements (mod_stride_s of 4)", g);
      return RA_EINVAL;
    }
    d.h = static_cast<const __nv_bfloat16*>(s.h);
    d.h_ss = s.h_stride_s;
    d.h_sr = s.h_stride_r;
    d.x = static_cast<__nv_bfloat16*>(s.x);
    d.x_ss = s.x_stride_s;
    d.x_sr = s.x_stride_r;
    d.shift = s.shift;
    d.scale = s.scale;
    d.mod_ss = s.mod_stride_s;
    rows += int64_t(a->B) * s.rows;
  }
  if (rows == 0) return RA_OK;
  if ((rows + 3) / 4 > 2147483647) {
    set_error("refadapt_ln_modulate: too many rows");
    return RA_EINVAL;
  }
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  switch (p.groups) {
#define RA_LNMOD_CASE(G) \
  case G: return run<G>(p, rows, by_row(p, rows, num_sms()), st);
    RA_LNMOD_CASE(1) RA_LNMOD_CASE(2) RA_LNMOD_CASE(3) RA_LNMOD_CASE(4) RA_LNMOD_CASE(5) RA_LNMOD_CASE(6)
    RA_LNMOD_CASE(7) RA_LNMOD_CASE(8) RA_LNMOD_CASE(9) RA_LNMOD_CASE(10) RA_LNMOD_CASE(11) RA_LNMOD_CASE(12)
    RA_LNMOD_CASE(13) RA_LNMOD_CASE(14) RA_LNMOD_CASE(15) RA_LNMOD_CASE(16)
#undef RA_LNMOD_CASE
    default: return RA_EINVAL;  // C was checked above
  }
}
