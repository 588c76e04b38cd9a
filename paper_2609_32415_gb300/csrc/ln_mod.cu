// refadapt_ln_modulate: the DiT block's modulated LayerNorm,
//   x = (h - mean(h)) / sqrt(var(h) + eps) * (1 + scale[sample]) + shift[sample]
// over the C features of every row (no affine of its own; the AdaLN shift and
// scale of the block, stream and sample modulate it). Reference segments may be
// gated on the per-sample mode (skipped when REUSE).
//
// HBM-bound: 4 C bytes per row. One warp per row, the row in registers as
// packed bf16, mean and variance in fp32 in two passes over them. What keeps
// HBM busy: one persistent CTA per SM that takes a contiguous share of the live
// rows, each warp with a ring of rows that bulk copies fill ahead of it; and
// the modulation (8 C bytes, twice a row's own bytes) held in shared memory per
// (segment, sample) piece instead of read through L1 for every row. At C = 3072:
// 12544 rows 44.7 -> 26.6 us (5.8 TB/s; a plain copy of them 24.3), 4352 rows
// 18.4 -> 13.0, 1280 rows 8.8 -> 5.4, against one row per warp and no ring.
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
// rows of one live (segment, sample); rows [begin, begin + rows) of the order.
struct Piece {
  int g, s;
  int64_t begin;
  // Moves to the piece that holds row i (i at or past begin, below the total).
  __device__ __forceinline__ void seek(const Params& p, int64_t i) {
    while (i - begin >= p.seg[g].rows || !live(p, g, s)) {
      if (live(p, g, s)) begin += p.seg[g].rows;
      if (++s == p.B) {
        s = 0;
        ++g;
      }
    }
  }
};

// A warp whose own copy of row i did not end within the budget: it lets the
// copies on their way (of its next S - 1 rows) land, and its rows from i on
// become NaN.
template <int G>
__device__ __noinline__ void give_up(const Params& p, uint64_t* full, int stage, uint32_t phase, int64_t i, int64_t hi) {
  using L = Layout<G>;
  for (int k = 1; k < L::S && i + k * L::WARPS < hi; ++k) {
    if (++stage == L::S) {
      stage = 0;
      phase ^= 1;
    }
    mbar_wait_drain(full + stage, phase, p.budget_ns);
  }
  Piece w{0, 0, 0};
  for (; i < hi; i += L::WARPS) {
    w.seek(p, i);
    const Seg& sg = p.seg[w.g];
    uint4* dst = reinterpret_cast<uint4*>(sg.x + w.s * sg.x_ss + (i - w.begin) * sg.x_sr);
    for (int q = 0; q < G; ++q) dst[q * 32 + (threadIdx.x & 31)] = make_uint4(~0u, ~0u, ~0u, ~0u);
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
  int64_t total = 0;
  for (int g = 0; g < p.n_seg; ++g) {
    int n = p.B;
    if (p.seg[g].gated) {
      n = 0;
      for (int s0 = 0; s0 < p.B; s0 += 32)
        n += __popc(__ballot_sync(0xffffffffu, s0 + lane < p.B && live(p, g, s0 + lane)));
    }
    total += int64_t(n) * p.seg[g].rows;
  }
  const uint32_t share = uint32_t(total) / gridDim.x, more = uint32_t(total) - share * gridDim.x;
  const int64_t lo = int64_t(share) * blockIdx.x + min(blockIdx.x, more);
  const int64_t hi = lo + share + (blockIdx.x < more ? 1 : 0);
  if (lo == hi) return;
  Piece ld{0, 0, 0}, w{0, 0, 0};
  int64_t i = lo + warp, ld_i = i;  // this warp's rows: lo + warp, + W, ...; loads run up to S rows ahead
  auto load = [&](int stage) {
    if (ld_i < hi && lane == 0) {
      ld.seek(p, ld_i);
      const Seg& sg = p.seg[ld.g];
      mbar_arrive_expect_tx(full + stage, L::ROW_BYTES);
      bulk_load(ring + stage * L::ROW_BYTES, sg.h + ld.s * sg.h_ss + (ld_i - ld.begin) * sg.h_sr, L::ROW_BYTES,
                full + stage);
    }
    ld_i += W;
  };
  for (int k = 0; k < S; ++k) load(k);
  int stage = 0;
  uint32_t phase = 0;
  for (int64_t piece_lo = lo; piece_lo < hi;) {
    w.seek(p, piece_lo);
    const Seg& sg = p.seg[w.g];
    const int64_t piece_hi = min(hi, w.begin + sg.rows);
    if (piece_lo != lo) __syncthreads();  // every warp is done with the last piece's modulation
    const float* shift = sg.shift + w.s * sg.mod_ss;
    const float* scale = sg.scale + w.s * sg.mod_ss;
    for (int f = threadIdx.x; f < 64 * G; f += 32 * W) {
      // Four columns: half f % 2 of lane (f / 2) % 32 in group f / 64; kept as
      // [group][half][lane], so the rows' 16-byte reads have no bank conflicts.
      const int at = ((f >> 6) * 2 + (f & 1)) * 32 + ((f >> 1) & 31);
      reinterpret_cast<float4*>(shift_sh)[at] = reinterpret_cast<const float4*>(shift)[f];
      float4 v = reinterpret_cast<const float4*>(scale)[f];
      v.x += 1.f, v.y += 1.f, v.z += 1.f, v.w += 1.f;
      reinterpret_cast<float4*>(scale_sh)[at] = v;
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
      const float mean = sum / float(p.C);
      const uint64_t neg_mean = f2_pack(-mean, -mean);
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
      const float rstd = rsqrtf(sq / float(p.C) + p.eps);
      const uint64_t rstd2 = f2_pack(rstd, rstd);
      uint4* dst = reinterpret_cast<uint4*>(sg.x + w.s * sg.x_ss + (i - w.begin) * sg.x_sr);
#pragma unroll
      for (int q = 0; q < G; ++q) {
        const uint32_t e[4] = {u[q].x, u[q].y, u[q].z, u[q].w};
        uint32_t pk[4];
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
          const ulonglong2 sh = reinterpret_cast<const ulonglong2*>(shift_sh)[(2 * q + k / 2) * 32 + lane];
          const ulonglong2 sc = reinterpret_cast<const ulonglong2*>(scale_sh)[(2 * q + k / 2) * 32 + lane];
          float y0, y1;
          f2_unpack(f2_fma(f2_mul(f2_add(bf2_unpack(e[k]), neg_mean), rstd2), sc.x, sh.x), y0, y1);
          pk[k] = pack_bf16x2(y0, y1);
          f2_unpack(f2_fma(f2_mul(f2_add(bf2_unpack(e[k + 1]), neg_mean), rstd2), sc.y, sh.y), y0, y1);
          pk[k + 1] = pack_bf16x2(y0, y1);
        }
        dst[q * 32 + lane] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
      }
    }
    piece_lo = piece_hi;
  }
}

template <int G>
ra_status launch(const Params& p, int64_t rows, cudaStream_t st) {
  using L = Layout<G>;
  const ra_status as =
      ensure_dynamic_smem(reinterpret_cast<const void*>(ln_mod_kernel<G>), L::BYTES, "refadapt_ln_modulate");
  if (as != RA_OK) return as;
  const int64_t sms = num_sms();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(rows < sms ? rows : sms));
  cfg.blockDim = dim3(32 * L::WARPS);
  cfg.dynamicSmemBytes = L::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr = pdl_attribute();
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, ln_mod_kernel<G>, p);
  if (e != cudaSuccess) {
    set_error("refadapt_ln_modulate: launch failed: %s", cudaGetErrorString(e));
    cudaGetLastError();
    return RA_ECUDA;
  }
  return launch_status("refadapt_ln_modulate");
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
  if (rows > 4294967295ll) {
    set_error("refadapt_ln_modulate: too many rows");
    return RA_EINVAL;
  }
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  switch (p.groups) {
#define RA_LNMOD_CASE(G) \
  case G: return launch<G>(p, rows, st);
    RA_LNMOD_CASE(1) RA_LNMOD_CASE(2) RA_LNMOD_CASE(3) RA_LNMOD_CASE(4) RA_LNMOD_CASE(5) RA_LNMOD_CASE(6)
    RA_LNMOD_CASE(7) RA_LNMOD_CASE(8) RA_LNMOD_CASE(9) RA_LNMOD_CASE(10) RA_LNMOD_CASE(11) RA_LNMOD_CASE(12)
    RA_LNMOD_CASE(13) RA_LNMOD_CASE(14) RA_LNMOD_CASE(15) RA_LNMOD_CASE(16)
#undef RA_LNMOD_CASE
    default: return RA_EINVAL;  // C was checked above
  }
}
