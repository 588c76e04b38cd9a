"""GPU parity of the DiT block's layers (refadapt_rope_table,
refadapt_ln_modulate, refadapt_gemm and its epilogues) against the oracle's
fp64 layers (oracle/dit.py) on the same seeded bf16 inputs.

Tolerance: every output is one bf16 rounding of a value the GPU forms in fp32
and the oracle in fp64, so the two agree except where the fp32 value lands on
the other side of a bf16 rounding boundary, a difference of one bf16 ulp
(at most 2^-7 |ref|): |got - ref| <= 2^-7 |ref| + 1e-3 rms(ref) (fp32
cancellation in long dot products), and at least 98 % of the elements are
equal."""
import math

import numpy as np
import pytest
import torch

import oracle
from oracle import BOUNDARY, COMPUTE, FULL, REUSE
from oracle import dit
from _helpers import bits, f64

pytestmark = pytest.mark.gpu


def _close(got, ref, frac=0.98):
    got = np.asarray(got, np.float64)
    ref = np.asarray(ref, np.float64)
    rms = math.sqrt(float(np.mean(ref ** 2))) + 1e-30
    bad = np.abs(got - ref) > 2.0 ** -7 * np.abs(ref) + 1e-3 * rms
    eq = float(np.mean(got == ref))
    return (not bad.any()) and eq >= frac, int(bad.sum()), eq


def _bf(shape, g, scale=1.0):
    return (torch.randn(shape, generator=g) * scale).to(torch.bfloat16)


def test_rope_table_matches_angles(cuda_ok):
    from paper_2609_32415_gb300 import api
    for n_pos, d in ((33272, 128), (100, 64)):
        t = api.rope_table(n_pos, d).cpu().double().numpy()
        ang = dit.rope_angles(np.arange(n_pos), d)
        assert np.abs(t[..., 0] - np.cos(ang)).max() < 1e-6
        assert np.abs(t[..., 1] - np.sin(ang)).max() < 1e-6


@pytest.mark.parametrize("C", [256, 3072])
def test_ln_modulate_segments_and_gating(cuda_ok, C):
    from paper_2609_32415_gb300 import api
    g = torch.Generator().manual_seed(C)
    B = 2
    rows = {"text": 40, "ref": 130, "tgt": 77}
    mode = torch.tensor([REUSE, BOUNDARY], dtype=torch.int32, device="cuda")
    segs, keep = [], {}
    for r, n in rows.items():
        # strided input: rows of a wider buffer
        wide = (_bf((B, n, C + 64), g) * 2.0 + 0.5).cuda()
        h = wide[:, :, 32:32 + C]
        x = torch.full((B, n, C), float("nan"), dtype=torch.bfloat16, device="cuda")
        shift = (torch.randn((B, C), generator=g) * 0.1).cuda()
        scale = (torch.randn((B, C), generator=g) * 0.1).cuda()
        segs.append({"h": h, "x": x, "shift": shift, "scale": scale, "gated": r == "ref"})
        keep[r] = (h, x, shift, scale)
    api.refadapt_ln_modulate(segs, C, eps=1e-6, mode=mode)
    torch.cuda.synchronize()
    for r, (h, x, shift, scale) in keep.items():
        for s in range(B):
            got = f64(x[s])
            if r == "ref" and s == 0:
                assert np.isnan(got).all()
                continue
            ref = dit.round_bf16(dit.layer_norm_modulate(f64(h[s]), shift[s].double().cpu().numpy(),
                                                         scale[s].double().cpu().numpy(), 1e-6))
            ok, nbad, eq = _close(got, ref, 0.99)
            assert ok, (r, s, nbad, eq)


@pytest.mark.parametrize("C,B,rows", [(256, 40, (3, 5, 2)), (512, 1, (1, 0, 0)), (1280, 3, (1, 900, 130)),
                                      (2304, 2, (700, 4, 33)), (3328, 2, (5, 600, 1500)), (4096, 1, (17, 9, 3000))])
def test_ln_modulate_pieces(cuda_ok, C, B, rows):
    """Row shares of a CTA that cross segments and samples, more samples than
    lanes, rings of two to four rows, fewer rows than SMs."""
    from paper_2609_32415_gb300 import api
    g = torch.Generator().manual_seed(C + B)
    mode = torch.tensor([REUSE if s % 3 == 1 else COMPUTE for s in range(B)], dtype=torch.int32, device="cuda")
    segs = [{"h": _bf((B, n, C), g).cuda(), "x": torch.full((B, n, C), float("nan"), dtype=torch.bfloat16, device="cuda"),
             "shift": (torch.randn((B, C), generator=g) * 0.1).cuda(),
             "scale": (torch.randn((B, C), generator=g) * 0.1).cuda(), "gated": i == 1} for i, n in enumerate(rows)]
    api.refadapt_ln_modulate(segs, C, mode=mode)
    torch.cuda.synchronize()
    for i, sd in enumerate(segs):
        for s in range(B):
            got = f64(sd["x"][s])
            if i == 1 and s % 3 == 1:
                assert np.isnan(got).all()
                continue
            if got.size == 0:
                continue
            ref = dit.round_bf16(dit.layer_norm_modulate(f64(sd["h"][s]), sd["shift"][s].double().cpu().numpy(),
                                                         sd["scale"][s].double().cpu().numpy(), 1e-6))
            ok, nbad, eq = _close(got, ref, 0.99)
            assert ok, (i, s, nbad, eq)


@pytest.mark.parametrize("C", [256, 512, 768, 2048, 3072, 4096])
def test_ln_modulate_by_row_and_persistent_agree(cuda_ok, C):
    """A call of many rows of a few samples, and calls of one and of a few rows of
    each: a row's result does not depend on the kernel that the call takes."""
    from paper_2609_32415_gb300 import api
    g = torch.Generator().manual_seed(C)
    B, n = 2, 9000
    h, mods = _bf((B, n, C), g).cuda(), [torch.randn((B, C), generator=g).cuda() for _ in range(2)]
    seg = {"shift": mods[0], "scale": mods[1]}
    x = torch.empty_like(h)
    api.refadapt_ln_modulate([dict(seg, h=h, x=x)], C)
    _launched("persistent" if C > 256 else "one row per warp")
    for lo, hi in ((0, 1), (4000, 4007), (n - 1, n)):
        y = torch.empty((B, hi - lo, C), dtype=torch.bfloat16, device="cuda")
        api.refadapt_ln_modulate([dict(seg, h=h[:, lo:hi], x=y)], C)
        _launched("one row per warp")
        assert torch.equal(y, x[:, lo:hi])
    ref = torch.nn.functional.layer_norm(h[:, ::500].double(), (C,), eps=1e-6)
    ref = ref * (1 + mods[1].double()[:, None]) + mods[0].double()[:, None]
    assert (x[:, ::500].double() - ref).abs().max() <= 2.0 ** -8 * ref.abs().max()


@pytest.mark.parametrize("C,B,rows,form", [(1280, 300, (3, 0, 20), 0), (3072, 70, (1, 200, 2), 0), (512, 33, (0, 1, 400), 0),
                                           (3072, 9, (40, 300, 2000), 1), (4096, 40, (0, 90, 300), 1),
                                           (3328, 2, (3000, 600, 150), 1), (1280, 3, (500, 3000, 4000), 1),
                                           (2304, 34, (0, 400, 350), 1)])
def test_ln_modulate_many_samples(cuda_ok, C, B, rows, form):
    """By row, and persistent with rings of two to four rows and shares that cross
    segments, samples and skipped samples."""
    from paper_2609_32415_gb300 import api
    g = torch.Generator().manual_seed(B)
    modes = [int(m) for m in torch.randint(0, 4, (B,), generator=g)]
    segs = [{"h": _bf((B, n, C), g).cuda(), "x": torch.full((B, n, C), float("nan"), dtype=torch.bfloat16, device="cuda"),
             "shift": torch.randn((B, C), generator=g).cuda(), "scale": torch.randn((B, C), generator=g).cuda(),
             "gated": i == 1} for i, n in enumerate(rows)]
    api.refadapt_ln_modulate(segs, C, mode=torch.tensor(modes, dtype=torch.int32, device="cuda"))
    _launched("persistent" if form else "one row per warp")
    reuse = torch.tensor([m == REUSE for m in modes], device="cuda")
    for i, sd in enumerate(segs):
        if sd["h"].numel() == 0:
            continue
        ref = torch.nn.functional.layer_norm(sd["h"].double(), (C,), eps=1e-6)
        ref = ref * (1 + sd["scale"].double()[:, None]) + sd["shift"].double()[:, None]
        live = ~reuse if i == 1 else torch.ones_like(reuse)
        assert bool(torch.isnan(sd["x"][~live]).all())
        assert (sd["x"][live].double() - ref[live]).abs().max() <= 2.0 ** -8 * ref.abs().max()


def test_ln_modulate_with_a_short_wait_budget(cuda_ok):
    """The rows' own copies end; a wait budget that does not cover them leaves no row unwritten."""
    from paper_2609_32415_gb300 import api
    g = torch.Generator().manual_seed(3)
    C, n = 3072, 1500
    sd = {"h": _bf((2, n, C), g).cuda(), "shift": torch.randn((2, C), generator=g).cuda(),
          "scale": torch.randn((2, C), generator=g).cuda()}
    x = [torch.full((2, n, C), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    api.refadapt_ln_modulate([dict(sd, x=x[0])], C)
    api.refadapt_set_wait_budget_ns(1)
    try:
        for _ in range(10):
            api.refadapt_ln_modulate([dict(sd, x=x[1])], C)
            _launched("persistent")
            torch.cuda.synchronize()
            assert torch.equal(x[0].view(torch.int16), x[1].view(torch.int16))
            x[1].fill_(float("nan"))
    finally:
        api.refadapt_set_wait_budget_ns(500_000_000)


def _launched(form):
    """The last call took this launch form."""
    from paper_2609_32415_gb300 import api
    got = api.refadapt_last_launch()
    assert got == form, (form, got)


def _gemm_case(B, K, N, rows_list, epi, g, gated=None, modes=None, inplace=False, tile_mode=0):
    from paper_2609_32415_gb300 import api
    from paper_2609_32415_gb300._lib import RA_EPI_GELU, RA_EPI_RESID, RA_EPI_STORE
    segs, keep = [], []
    for i, rows in enumerate(rows_list):
        a = _bf((B, rows, K), g).cuda()
        w = _bf((N, K), g, 1.0 / math.sqrt(K)).cuda()
        bias = (torch.randn(N, generator=g) * 0.1).cuda() if i != 1 else None
        sd = {"a": a, "w": w, "bias": bias, "gated": bool(gated and gated[i])}
        if epi == RA_EPI_RESID:
            resid = _bf((B, rows, N), g).cuda()
            gate = (0.3 + 0.1 * torch.randn((B, N), generator=g)).cuda()
            sd.update(resid=resid, gate=gate)
            sd["out"] = resid if inplace else torch.full((B, rows, N), float("nan"), dtype=torch.bfloat16,
                                                         device="cuda")
            keep.append((a, w, bias, resid.clone(), gate, sd["out"]))
        else:
            sd["out"] = torch.full((B, rows, N), float("nan"), dtype=torch.bfloat16, device="cuda")
            keep.append((a, w, bias, None, None, sd["out"]))
        segs.append(sd)
    mode = None if modes is None else torch.tensor(modes, dtype=torch.int32, device="cuda")
    api.refadapt_gemm(segs, N, K, epi, mode=mode, tile_mode=tile_mode)
    torch.cuda.synchronize()
    for i, (a, w, bias, resid, gate, out) in enumerate(keep):
        for s in range(B):
            got = f64(out[s])
            if got.size == 0:
                continue
            if gated and gated[i] and modes[s] == REUSE:
                if epi == RA_EPI_RESID and inplace:
                    np.testing.assert_array_equal(got, f64(resid[s]))
                else:
                    assert np.isnan(got).all()
                continue
            y = dit.linear(f64(a[s]), f64(w), None if bias is None else bias.double().cpu().numpy())
            if epi == RA_EPI_GELU:
                y = dit.gelu_tanh(y)
            elif epi == RA_EPI_RESID:
                y = f64(resid[s]) + gate[s].double().cpu().numpy() * y
            ok, nbad, eq = _close(got, dit.round_bf16(y))
            assert ok, (epi, i, s, nbad, eq)


# tile_mode 1: one CTA per 128 x 256 tile; 2: CTA pairs (cta_group::2) on 256 x 256 tiles.
TILE_MODES = [1, 2]


@pytest.mark.parametrize("tile_mode", TILE_MODES)
@pytest.mark.parametrize("K,N,rows", [(64, 256, [1]), (256, 768, [40, 130, 77]), (3072, 512, [300]),
                                      (512, 2048, [2500]), (128, 512, [4500, 70]), (192, 512, [700])])
def test_gemm_store_matches_oracle(cuda_ok, K, N, rows, tile_mode):
    """Tiles are numbered in bands of 16 tile rows: 4500 rows make a full band
    and a partial one of 256-row tiles (18 = 16 + 2) and of 128-row tiles
    (36 = 16 + 16 + 4), followed by a second segment."""
    from paper_2609_32415_gb300._lib import RA_EPI_STORE
    _gemm_case(2, K, N, rows, RA_EPI_STORE, torch.Generator().manual_seed(K + N), tile_mode=tile_mode)


@pytest.mark.parametrize("tile_mode", TILE_MODES)
def test_gemm_gelu_matches_oracle(cuda_ok, tile_mode):
    from paper_2609_32415_gb300._lib import RA_EPI_GELU
    _gemm_case(1, 256, 1024, [129, 200], RA_EPI_GELU, torch.Generator().manual_seed(5), tile_mode=tile_mode)


@pytest.mark.parametrize("tile_mode", TILE_MODES)
@pytest.mark.parametrize("inplace", [False, True])
def test_gemm_gated_residual_matches_oracle(cuda_ok, inplace, tile_mode):
    from paper_2609_32415_gb300._lib import RA_EPI_RESID
    _gemm_case(2, 1024, 256, [40, 256, 200], RA_EPI_RESID, torch.Generator().manual_seed(6),
               gated=[False, True, False], modes=[REUSE, COMPUTE], inplace=inplace, tile_mode=tile_mode)


@pytest.mark.parametrize("tile_mode", TILE_MODES)
def test_gemm_skips_gated_tiles_in_a_long_schedule(cuda_ok, tile_mode):
    """Three segments, the middle one gated off for one sample, enough tiles
    that every CTA walks several (both accumulators, several phases)."""
    from paper_2609_32415_gb300._lib import RA_EPI_STORE
    _gemm_case(2, 192, 1024, [700, 1500, 900], RA_EPI_STORE, torch.Generator().manual_seed(7),
               gated=[False, True, False], modes=[COMPUTE, REUSE], tile_mode=tile_mode)


@pytest.mark.parametrize("tile_mode", TILE_MODES)
@pytest.mark.parametrize("B,rows,gated", [(41, [6, 0, 16], [False, True, False]), (33, [0, 130, 3], [False, True, False]),
                                          (70, [0, 0, 20], [False] * 3), (9, [300, 40, 0], [True, False, False])])
def test_gemm_many_samples(cuda_ok, B, rows, gated, tile_mode):
    """Tiles are found past many samples, empty segments and skipped samples."""
    g = torch.Generator().manual_seed(B)
    _gemm_case(B, 256, 512, rows, 0, g, gated=gated, modes=[int(m) for m in torch.randint(0, 4, (B,), generator=g)],
               tile_mode=tile_mode)


# One row tile and just more columns than a round of the next narrower tiles
# holds (76 pairs, 152 single CTAs): every tile width from 64 to 256, the last
# tile of most of them reaching past N.
@pytest.mark.parametrize("tile_mode,N", [(2, 512), (2, 5120), (2, 7424), (2, 9984), (2, 12288), (2, 14848),
                                         (2, 17152), (1, 512), (1, 9984), (1, 14848)])
@pytest.mark.parametrize("epi", ["gelu", "resid"])
def test_gemm_tile_widths_match_oracle(cuda_ok, epi, tile_mode, N):
    from paper_2609_32415_gb300._lib import RA_EPI_GELU, RA_EPI_RESID
    _gemm_case(1, 512, N, [40], RA_EPI_GELU if epi == "gelu" else RA_EPI_RESID, torch.Generator().manual_seed(N),
               tile_mode=tile_mode)
    widths = {512: 64, 5120: 96, 7424: 128, 9984: 160, 12288: 192, 14848: 224, 17152: 256}
    if tile_mode == 1:
        widths.update({9984: 96, 14848: 128})
    _launched("%s, %d columns" % ("CTA pairs" if tile_mode == 2 else "single CTAs", widths[N]))


@pytest.mark.parametrize("rows,N,narrow", [([5], 14336, False), ([40, 3], 12288, False), ([40], 12288, True), ([5], 4096, True)])
def test_gemm_few_rows_take_wide_tiles(cuda_ok, rows, N, narrow):
    """Many column tiles do not share a handful of rows of A."""
    from paper_2609_32415_gb300 import api
    _gemm_case(1, 512, N, rows, 0, torch.Generator().manual_seed(N))
    assert ("256 columns" in api.refadapt_last_launch()) != narrow, api.refadapt_last_launch()


# Calls of few tiles and a long K, whose tiles are shared by the CTAs of a cluster: one row, ragged
# rows, K steps that do not divide by the CTAs, tiles of 64 to 256 columns, a gated segment.
@pytest.mark.parametrize("epi", [0, 1, 2])
@pytest.mark.parametrize("B,K,N,rows", [(1, 4160, 256, [1]), (1, 4160, 256, [1, 129, 77]), (2, 4096, 1024, [77, 300]),
                                        (2, 4160, 1024, [77, 500, 300]), (1, 12352, 768, [130, 257]),
                                        (1, 16384, 512, [640])])
def test_gemm_split_k_matches_oracle(cuda_ok, epi, B, K, N, rows):
    gated = [i == 1 for i in range(len(rows))]
    _gemm_case(B, K, N, rows, epi, torch.Generator().manual_seed(K + N), gated=gated, modes=[REUSE, COMPUTE][:B],
               inplace=epi == 2)
    _launched("clusters of %d, %d columns" % (2 if rows == [77, 500, 300] else 4, 256 if N == 1024 else 128))


# A little more than whole rounds of pair tiles (81 or 84 of them): the rest is split, its tiles
# cut into quarters, of which some have no rows; with modes that leave no rest or no whole round.
@pytest.mark.parametrize("epi,B,N,rows,modes", [(2, 1, 3072, [1024, 256, 300], [COMPUTE]),
                                                (2, 1, 3072, [1024, 256, 300], [REUSE]),
                                                (1, 2, 1536, [100, 700, 700], [COMPUTE, COMPUTE]),
                                                (0, 2, 1536, [100, 700, 700], [REUSE, COMPUTE]),
                                                (2, 3, 2304, [385, 130], [COMPUTE, REUSE, COMPUTE]),
                                                (0, 3, 2304, [385, 130], [COMPUTE, COMPUTE, COMPUTE])])
def test_gemm_split_rest_matches_oracle(cuda_ok, epi, B, N, rows, modes):
    _gemm_case(B, 8256, N, rows, epi, torch.Generator().manual_seed(N + B), gated=[i == 1 for i in range(len(rows))],
               modes=modes, inplace=epi == 2)
    _launched("rounds of CTA pairs, up to 9 tiles in clusters of 4")


@pytest.mark.parametrize("tile_mode", TILE_MODES)
@pytest.mark.parametrize("H,d,modes", [(4, 64, [FULL, BOUNDARY]), (2, 128, [REUSE, COMPUTE])])
def test_gemm_qkv_epilogue_matches_oracle(cuda_ok, H, d, modes, tile_mode):
    """QKV projection with per-head RMS norm and RoPE at the rows' joint
    positions; the reference segment is gated: REUSE writes nothing,
    BOUNDARY writes only its query (K/V stay the cached ones)."""
    _qkv_case(H, d, modes, tile_mode, {"text": 37, "ref": 256, "tgt": 300})


@pytest.mark.parametrize("tile_mode", TILE_MODES)
@pytest.mark.parametrize("H,d,tgt", [(12, 64, 200), (12, 64, 700), (4, 64, 2100), (4, 64, 4500), (2, 128, 3500)])
def test_gemm_qkv_wide_tiles_match_oracle(cuda_ok, H, d, tgt, tile_mode):
    """Enough rows that tiles of one to four heads are picked."""
    _qkv_case(H, d, [BOUNDARY, COMPUTE], tile_mode, {"text": 37, "ref": 300, "tgt": tgt})


def test_gemm_qkv_position_offset_is_any_number(cuda_ok):
    """pos_offset is taken as int() takes it."""
    from paper_2609_32415_gb300 import api
    from paper_2609_32415_gb300._lib import RA_EPI_QKV
    H, d, C = 4, 64, 256
    g = torch.Generator().manual_seed(4)
    sd = {"a": _bf((1, 9, C), g).cuda(), "w": _bf((3 * C, C), g).cuda(), "q_norm": torch.ones(d, device="cuda"),
          "k_norm": torch.ones(d, device="cuda")}
    got = []
    for pos in (7, 7.0, np.float32(7.5), "7"):
        out = {z: torch.empty((1, H, 9, d), dtype=torch.bfloat16, device="cuda") for z in "qkv"}
        api.refadapt_gemm([dict(sd, **out, pos_offset=pos)], 3 * C, C, RA_EPI_QKV, rope=api.rope_table(16, d), H=H, d=d)
        got.append(out)
    with pytest.raises(TypeError):
        api.refadapt_gemm([dict(sd, **out, pos_offset=None)], 3 * C, C, RA_EPI_QKV, rope=api.rope_table(16, d), H=H, d=d)
    torch.cuda.synchronize()
    assert all(torch.equal(o[z], got[0][z]) for o in got for z in "qkv")


def _qkv_case(H, d, modes, tile_mode, n):
    from paper_2609_32415_gb300 import api
    from paper_2609_32415_gb300._lib import RA_EPI_QKV
    g = torch.Generator().manual_seed(H * d)
    B, C = 2, H * d
    pos0 = {"text": 0, "ref": n["text"], "tgt": n["text"] + n["ref"]}
    rope = api.rope_table(sum(n.values()), d)
    mode = torch.tensor(modes, dtype=torch.int32, device="cuda")
    segs, keep = [], {}
    for i, (r, rows) in enumerate(n.items()):
        x = _bf((B, rows, C), g).cuda()
        w = _bf((3 * C, C), g, 1.0 / math.sqrt(C)).cuda()
        bias = (torch.randn(3 * C, generator=g) * 0.02).cuda()
        qn = (1.0 + 0.1 * torch.randn(d, generator=g)).cuda()
        kn = (1.0 + 0.1 * torch.randn(d, generator=g)).cuda()
        out = [torch.full((B, H, rows, d), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
        segs.append({"a": x, "w": w, "bias": bias, "q": out[0], "k": out[1], "v": out[2], "q_norm": qn,
                     "k_norm": kn, "pos_offset": pos0[r], "gated": r == "ref"})
        keep[r] = (x, w, bias, qn, kn, out)
    api.refadapt_gemm(segs, 3 * C, C, RA_EPI_QKV, mode=mode, rope=rope, H=H, d=d, norm_eps=1e-6,
                      tile_mode=tile_mode)
    torch.cuda.synchronize()
    for r, (x, w, bias, qn, kn, out) in keep.items():
        pos = pos0[r] + np.arange(n[r])
        for s in range(B):
            y = dit.linear(f64(x[s]), f64(w), bias.double().cpu().numpy())
            parts = [y[:, z * C:(z + 1) * C].reshape(n[r], H, d).transpose(1, 0, 2) for z in range(3)]
            want = [dit.round_bf16(dit.apply_rope(dit.rms_norm(parts[0], qn.double().cpu().numpy()), pos)),
                    dit.round_bf16(dit.apply_rope(dit.rms_norm(parts[1], kn.double().cpu().numpy()), pos)),
                    dit.round_bf16(parts[2])]
            for z in range(3):
                got = f64(out[z][s])
                skip = r == "ref" and (modes[s] == REUSE or (modes[s] == BOUNDARY and z > 0))
                if skip:
                    assert np.isnan(got).all(), (r, s, z)
                    continue
                ok, nbad, eq = _close(got, want[z])
                assert ok, (r, s, z, nbad, eq)


def test_gemm_rejects_bad_shapes(cuda_ok):
    from paper_2609_32415_gb300 import api
    from paper_2609_32415_gb300._lib import RA_EINVAL, RA_EPI_STORE, RefAdaptError
    a = torch.zeros((1, 10, 96), dtype=torch.bfloat16, device="cuda")
    w = torch.zeros((256, 96), dtype=torch.bfloat16, device="cuda")
    out = torch.zeros((1, 10, 256), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(RefAdaptError) as e:
        api.refadapt_gemm([{"a": a, "w": w, "out": out}], 256, 96, RA_EPI_STORE)   # K not a multiple of 64
    assert e.value.status == RA_EINVAL
    w2 = torch.zeros((128, 64), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(RefAdaptError) as e:
        api.refadapt_gemm([{"a": a[:, :, :64], "w": w2, "out": out[:, :, :128]}], 128, 64,
                          RA_EPI_STORE)                                         # N not a multiple of 256
    assert e.value.status == RA_EINVAL
