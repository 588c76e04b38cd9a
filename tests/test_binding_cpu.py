"""The native argument marshalling refuses what the entry points' contract
refuses, before anything reaches the library (no GPU needed)."""
import pytest
import torch


def _attn(q=None, **kw):
    from paper_2609_32415_gb300 import api
    x = torch.zeros((1, 2, 4, 64), dtype=torch.bfloat16)
    return api.refadapt_joint_attn(q or (x, x, x), (x, x, x), (x, x, x), (x, x, x), torch.zeros(2), **kw)


def test_attention_tensors_must_be_bf16_cuda():
    with pytest.raises(ValueError, match=r"expected a \[B, H, n, d\] bf16 CUDA tensor .* got \(1, 2, 4, 64\) "
                                         r"torch.bfloat16 cpu"):
        _attn()
    with pytest.raises(ValueError, match="a_b is written only with ref_fresh"):
        _attn(a_b=torch.zeros(1, dtype=torch.int32))
    with pytest.raises(IndexError):
        _attn(q=(torch.zeros(1, 2, 4, 64),))
    with pytest.raises(TypeError):
        _attn(q=(1, 2, 3))


def test_row_segments_are_checked():
    from paper_2609_32415_gb300 import api
    x, v = torch.zeros((1, 3, 256), dtype=torch.bfloat16), torch.zeros((1, 256))
    with pytest.raises(ValueError, match=r"h: expected a \[B, rows, F\] CUDA tensor .* got \(1, 3, 256\)"):
        api.refadapt_ln_modulate([{"h": x, "x": x, "shift": v, "scale": v}], 256)
    with pytest.raises(KeyError, match="h"):
        api.refadapt_ln_modulate([{"x": x}], 256)
    with pytest.raises(ValueError, match=r"a: expected a \[B, rows, F\] CUDA tensor"):
        api.refadapt_gemm([{"a": x, "w": x[0], "out": x}], 256, 256, 0)
    with pytest.raises(TypeError):
        api.refadapt_gemm([], 256, 256, 0)


def test_a_binding_for_another_torch_is_rebuilt(monkeypatch):
    from paper_2609_32415_gb300 import build
    build.build()
    assert build.up_to_date()
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    assert not build.up_to_date()
