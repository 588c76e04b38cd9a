"""Launches of the attention that split an item's keys over a cluster, run whole
rounds and a split rest, or take one Q tile per item in two streams of key
tiles: against the oracle on a few heads, and bit for bit on a second run.

Element bound: P and the output are rounded to bf16 (unit roundoff 2^-9 each),
two independent errors that leave O with a 2-norm error of at most 2^-9 sqrt(2)
= 0.0028 of its rms; a million elements of it stay within 5.4 standard
deviations, so |got - ref| <= 0.015 (|ref| + rms), and 0.003 in the 2-norm."""
import numpy as np
import pytest
import torch

from _helpers import M_ABS, ROLES, empty_outputs, make_segments, mass_from_partials, o_close, oracle_block
from test_gpu_attention import BOUNDARY, COMPUTE, FULL, REUSE, _run

pytestmark = pytest.mark.gpu


def _assert_close(got, ref, what=""):
    ok, worst, normwise = o_close(got.double().cpu().numpy(), ref, 0.015)
    assert ok and normwise <= 3e-3, (what, worst, normwise)

def _launched(form):
    """The last attention call took this launch form (what the launch model picks
    for a case is asserted, or the case would not test it)."""
    from paper_2609_32415_gb300 import api
    got = api.refadapt_last_launch()
    assert got.startswith(form), (form, got)


TWO, ROUNDS, PAIRS = "two streams", "rounds of pairs, up to ", "pairs"
# text, ref, tgt rows, heads, d, modes, launch form.
CASES = [
    ((33, 5000, 130), 2, 128, [REUSE], TWO),           # 43 key tiles
    ((33, 5000, 130), 2, 64, [BOUNDARY, REUSE], TWO),  # the same, reference items live in one sample
    ((33, 700, 1500), 24, 64, None, TWO),              # three rounds, 19 key tiles
    ((40, 100, 200), 3, 64, [COMPUTE, REUSE], TWO),    # few key tiles
    ((0, 0, 77), 3, 128, None, PAIRS),                 # one key tile: no second stream
    ((0, 0, 200), 2, 64, None, TWO),                   # two: one each
    ((100, 900, 1900), 12, 128, [FULL], ROUNDS + "36 in clusters of 4"),   # 152 items and a rest of 4
    ((200, 900, 1700), 22, 128, [REUSE], ROUNDS + "36 in clusters of 4"),  # a rest of 24 that only reusing leaves
    ((100, 1800, 1800), 12, 128, [FULL], ROUNDS + "76 in clusters of 2"),  # a rest of 52
    ((100, 300, 1900), 10, 64, [REUSE, COMPUTE], ROUNDS),                  # mixed modes over more than a round
]


def _heads(segs, out, mp, hs):
    return ({r: [x[:, hs] for x in segs[r]] for r in ROLES}, {r: out[r][:, hs] for r in ROLES}, mp[:, hs])


@pytest.mark.parametrize("rows,H,d,modes,form", CASES, ids=lambda x: str(x).replace(" ", ""))
def test_split_launches_match_oracle(cuda_ok, rows, H, d, modes, form):
    n = dict(zip(ROLES, rows))
    B = len(modes) if modes else 1
    segs = make_segments(B, H, d, n, gen=torch.Generator().manual_seed(H * d + rows[1]), std=1.0)
    out, mp = _run(segs, B, H, d, n, modes)
    _launched(form)
    hs = sorted({0, H // 2, H - 1})
    s2, o2, m2 = _heads(segs, out, mp, hs)
    for s in range(B):
        ref = oracle_block(s2, s, modes[s] if modes else FULL, d ** -0.5)
        for r in ROLES:
            if ref["O"][r] is None:
                assert torch.isnan(o2[r][s].float()).all()
            else:
                _assert_close(o2[r][s], ref["O"][r], (s, r))
        assert np.abs(mass_from_partials(m2, n["tgt"])[s] - ref["M"]).max() <= M_ABS
    again, mp2 = _run(segs, B, H, d, n, modes)
    assert torch.equal(mp, mp2)
    for r in ROLES:
        assert torch.equal(out[r].view(torch.int16), again[r].view(torch.int16)), r


@pytest.mark.parametrize("H,d", [(8, 64), (8, 128), (24, 128)])
def test_split_item_without_reference_queries(cuda_ok, H, d):
    """Sampled target rows, no reference queries, 72 key tiles: 16 items in
    clusters of four, 48 in clusters of two. Head 0's reference bias of -inf
    leaves whole key ranges of its items with probability 0."""
    from paper_2609_32415_gb300 import api
    B, n = 1, {"text": 40, "ref": 8000, "tgt": 1000}
    segs = make_segments(B, H, d, n, gen=torch.Generator().manual_seed(d), std=1.0)
    q = [segs["text"][0], None, segs["tgt"][0][:, :, ::5, :]]
    out = [torch.zeros_like(q[0]), None, torch.zeros((B, H, 200, d), dtype=torch.bfloat16, device="cuda")]
    mp = api.alloc_mass_partial(B, H, 40, 200)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    bias = torch.zeros(H, device="cuda")
    bias[0] = float("-inf")
    api.refadapt_joint_attn(q, [segs[r][1] for r in ROLES], [segs[r][2] for r in ROLES], out, mp, err_word=err,
                            ref_logit_bias=bias)
    _launched("clusters of %d" % (2 if H == 24 else 4))
    torch.cuda.synchronize()
    api.refadapt_check_error(err)
    hs = [1, H - 1]
    ref = oracle_block({r: [x[:, hs] for x in segs[r]] for r in ROLES}, 0, FULL, d ** -0.5)
    _assert_close(out[2][0, hs], ref["O"]["tgt"][:, ::5])
    _assert_close(out[0][0, hs], ref["O"]["text"])
    cut = {r: [x[:, :1, :0] if r == "ref" else x[:, :1] for x in segs[r]] for r in ROLES}
    _assert_close(out[2][0, :1], oracle_block(cut, 0, REUSE, d ** -0.5)["O"]["tgt"][:, ::5])
    assert float(mp[0, 0].abs().max()) == 0.0


@pytest.mark.parametrize("d", [64, 128])
def test_split_range_of_masked_keys(cuda_ok, d):
    """A reference bias of -inf: a stream of key tiles starts with keys of
    probability 0; the target rows attend to text and target keys alone."""
    B, H, n = 1, 2, {"text": 33, "ref": 5000, "tgt": 130}
    segs = make_segments(B, H, d, n, gen=torch.Generator().manual_seed(d + 1), std=1.0)
    out, mp = _run(segs, B, H, d, n, [REUSE], bias=[float("-inf"), 0.5])
    _launched(TWO)
    cut = {r: [x[:, :1, :0] if r == "ref" else x[:, :1] for x in segs[r]] for r in ROLES}
    ref = oracle_block(cut, 0, REUSE, d ** -0.5)
    _assert_close(out["tgt"][0, :1], ref["O"]["tgt"])
    assert float(mp[0, 0].abs().max()) == 0.0
    s2, o2, m2 = _heads(segs, out, mp, [1])
    full = oracle_block(s2, 0, REUSE, d ** -0.5, np.array([0.5]))
    _assert_close(o2["tgt"][0], full["O"]["tgt"])
    assert abs(float(m2.double().sum()) / n["tgt"] - full["M"][0]) <= M_ABS


@pytest.mark.parametrize("rows,H,modes", [((33, 5000, 130), 2, [COMPUTE, REUSE]), ((100, 1800, 1800), 12, [FULL])])
def test_split_launches_write_the_cache(cuda_ok, rows, H, modes):
    """The fused cache write from two streams, and from whole rounds and split
    rest items (each rank of a cluster stores its own key range): a refreshing
    sample's slot equals the fresh rows, a reusing one's is untouched, a_b is
    stamped."""
    from paper_2609_32415_gb300 import api
    B, d, n = len(modes), 128, dict(zip(ROLES, rows))
    segs = make_segments(B, H, d, n, gen=torch.Generator().manual_seed(H))
    slot = [torch.full_like(x, 0.25) for x in segs["ref"]]
    a_b = torch.full((B,), -1, dtype=torch.int32, device="cuda")
    out = empty_outputs(B, H, d, n)
    mp = api.alloc_mass_partial(B, H, n["text"], n["tgt"])
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    mode = torch.tensor(modes, dtype=torch.int32, device="cuda")
    api.refadapt_joint_attn([segs["text"][0], slot[0], segs["tgt"][0]], [segs["text"][1], slot[1], segs["tgt"][1]],
                            [segs["text"][2], slot[2], segs["tgt"][2]], [out[r] for r in ROLES], mp, mode=mode,
                            err_word=err, ref_fresh=tuple(segs["ref"]), a_b=a_b, step=5)
    _launched(TWO if B == 2 else ROUNDS)
    torch.cuda.synchronize()
    api.refadapt_check_error(err)
    assert a_b.tolist() == [5 if m != REUSE else -1 for m in modes]
    for got, fresh in zip(slot, segs["ref"]):
        for s, m in enumerate(modes):
            assert torch.equal(got[s], fresh[s]) if m != REUSE else bool((got[s] == 0.25).all())
    hs = [0, H - 1]
    ref = oracle_block({r: [x[:, hs] for x in segs[r]] for r in ROLES}, 0, COMPUTE, d ** -0.5)
    for r in ROLES:
        _assert_close(out[r][0, hs], ref["O"][r], r)


@pytest.mark.parametrize("rows,H", [((0, 128, 20), 76), ((0, 90, 128), 20), ((5, 100, 40), 50), ((20, 250, 20), 30)])
@pytest.mark.parametrize("d", [64, 128])
def test_two_streams_keep_the_stored_query(cuda_ok, rows, H, d):
    """Two to four key tiles: a reference-row item's merge comes soon after the
    copy of its Q tile into the cache slot left the buffer the merge writes to.
    The slot equals the fresh rows bit for bit, over repeated launches."""
    from paper_2609_32415_gb300 import api
    n = dict(zip(ROLES, rows))
    segs = make_segments(1, H, d, n, gen=torch.Generator().manual_seed(H + d))
    slot = [torch.zeros_like(x) for x in segs["ref"]]
    a_b = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    out = empty_outputs(1, H, d, n)
    mp = api.alloc_mass_partial(1, H, n["text"], n["tgt"])
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    mode = torch.tensor([COMPUTE], dtype=torch.int32, device="cuda")
    for step in range(20):
        for x in slot:
            x.fill_(0.25)
        api.refadapt_joint_attn([segs["text"][0], slot[0], segs["tgt"][0]], [segs["text"][1], slot[1], segs["tgt"][1]],
                                [segs["text"][2], slot[2], segs["tgt"][2]], [out[r] for r in ROLES], mp, mode=mode,
                                err_word=err, ref_fresh=tuple(segs["ref"]), a_b=a_b, step=step)
        _launched(TWO)
        for got, fresh in zip(slot, segs["ref"]):
            assert torch.equal(got, fresh)
    api.refadapt_check_error(err)
    assert a_b.tolist() == [19]


@pytest.mark.parametrize("rows,H,d,form", [((0, 128, 4000), 24, 64, PAIRS), ((0, 130, 5000), 8, 128, ROUNDS),
                                           ((0, 128, 77), 3, 64, TWO), ((0, 1800, 1800), 12, 128, ROUNDS)])
def test_masked_reference_without_text(cuda_ok, rows, H, d, form):
    """A reference bias of -inf where the first key tile is the reference's:
    target rows attend to the target keys alone, in every launch form (pairs,
    two streams, whole rounds and a split rest)."""
    n = dict(zip(ROLES, rows))
    segs = make_segments(1, H, d, n, gen=torch.Generator().manual_seed(d + H), std=1.0)
    bias = [float("-inf")] + [0.25] * (H - 1)
    out, mp = _run(segs, 1, H, d, n, [FULL], bias=bias)
    _launched(form)
    cut = {r: [x[:, :1, :0] if r == "ref" else x[:, :1] for x in segs[r]] for r in ROLES}
    _assert_close(out["tgt"][0, :1], oracle_block(cut, 0, REUSE, d ** -0.5)["O"]["tgt"])
    assert float(mp[0, 0].abs().max()) == 0.0
    s2, o2, m2 = _heads(segs, out, mp, [H - 1])
    full = oracle_block(s2, 0, FULL, d ** -0.5, np.array([0.25]))
    for r in ("ref", "tgt"):
        _assert_close(o2[r][0], full["O"][r], r)
    assert abs(float(m2.double().sum()) / n["tgt"] - full["M"][0]) <= M_ABS


@pytest.mark.parametrize("B,rows,H,d,form", [(33, (3, 130, 140), 2, 64, PAIRS), (40, (0, 20, 30), 3, 128, TWO),
                                             (70, (20, 300, 10), 2, 128, PAIRS), (257, (0, 140, 5), 1, 64, PAIRS)])
def test_more_samples_than_lanes(cuda_ok, B, rows, H, d, form):
    """More than 32 samples: mixed modes, the fused cache write and the stamps;
    a sample's results are those of a call of its own."""
    from paper_2609_32415_gb300 import api
    n = dict(zip(ROLES, rows))
    g = torch.Generator().manual_seed(B)
    segs = make_segments(B, H, d, n, gen=g, std=1.0)
    modes = [int(m) for m in torch.randint(0, 4, (B,), generator=g)]
    slot = [torch.randn(x.shape, generator=g).to(torch.bfloat16).cuda() for x in segs["ref"]]
    old = [x.clone() for x in slot]
    a_b = torch.full((B,), -1, dtype=torch.int32, device="cuda")
    out = empty_outputs(B, H, d, n)
    mp = api.alloc_mass_partial(B, H, n["text"], n["tgt"])
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.refadapt_joint_attn([segs["text"][0], slot[0], segs["tgt"][0]], [segs["text"][1], slot[1], segs["tgt"][1]],
                            [segs["text"][2], slot[2], segs["tgt"][2]], [out[r] for r in ROLES], mp,
                            mode=torch.tensor(modes, dtype=torch.int32, device="cuda"), err_word=err,
                            ref_fresh=tuple(segs["ref"]), a_b=a_b, step=5)
    _launched(form)
    torch.cuda.synchronize()
    api.refadapt_check_error(err)
    fresh = [m in (COMPUTE, FULL) for m in modes]
    assert a_b.tolist() == [5 if f else -1 for f in fresh]
    for got, new, was in zip(slot, segs["ref"], old):
        for s in range(B):
            assert torch.equal(got[s], new[s] if fresh[s] else was[s]), s
    for s in sorted({0, 1, 31, 32, B // 2, B - 1}):
        seen = dict(segs, ref=[x for x in slot])
        ref = oracle_block(seen, s, modes[s], d ** -0.5)
        for r in ROLES:
            if n[r] == 0:
                continue
            if ref["O"][r] is None:
                assert torch.isnan(out[r][s].float()).all()
            else:
                _assert_close(out[r][s], ref["O"][r], (s, r))
        assert np.abs(mass_from_partials(mp, n["tgt"])[s] - ref["M"]).max() <= M_ABS
    assert not any(torch.isnan(out["tgt"][s].float()).any() for s in range(B))


@pytest.mark.parametrize("B,rows,H,d", [(16, (2, 0, 1068), 16, 64), (4, (0, 307, 1363), 24, 64), (8, (0, 308, 310), 24, 128)])
def test_single_tiles_only_over_few_rounds(cuda_ok, B, rows, H, d):
    """Over many rounds one Q tile per item (twice the K and V traffic) loses to pairs."""
    n = dict(zip(ROLES, rows))
    segs = make_segments(B, H, d, n, gen=torch.Generator().manual_seed(B), std=1.0)
    out, mp = _run(segs, B, H, d, n, [FULL] * B)
    _launched(PAIRS)
    s2, o2, m2 = _heads(segs, out, mp, [0, H - 1])
    ref = oracle_block(s2, B - 1, FULL, d ** -0.5)
    for r in ROLES:
        if n[r] > 0:
            _assert_close(o2[r][B - 1], ref["O"][r], r)
