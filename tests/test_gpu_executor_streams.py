"""Where the Executor's hooks run, and which buffers its launches take."""
import pytest
import torch

pytestmark = pytest.mark.gpu

ROLES = ("text", "ref", "tgt")


def _setup(n_blocks, n_steps=2, **kw):
    from paper_2609_32415_gb300 import Executor, roles_from_joint, synth
    wl = synth.custom_workload(1, 2, 64, 5, 100, 70, n_blocks=n_blocks, n_steps=n_steps, ref_drift=0.05,
                               tgt_drift=[0.05] * n_blocks, theta=0.08, delta_max=3)
    traj = synth.Trajectory(wl, device="cuda")
    ex = Executor(wl.n_blocks, wl.B, wl.H, wl.d, wl.n_text, wl.n_ref, wl.n_tgt, wl.theta, wl.delta_max, wl.eps,
                  log_steps=wl.n_steps, **kw)
    xs = [[roles_from_joint(traj.get(t, b), wl.offsets(), wl.n) for b in range(n_blocks)] for t in range(n_steps)]
    torch.cuda.synchronize()
    return wl, ex, xs


@pytest.mark.parametrize("n_blocks", [1, 3])
@pytest.mark.parametrize("explicit", [False, True])
def test_hooks_run_behind_the_attention(cuda_ok, n_blocks, explicit):
    """attn_hook and after_block see the attention's stream as the current one:
    what they enqueue is ordered behind it."""
    wl, ex, xs = _setup(n_blocks)
    stream = torch.cuda.Stream() if explicit else None
    allowed = [stream if explicit else torch.cuda.current_stream()] if n_blocks == 1 else ex._mains
    seen, copies = [], []
    ex.attn_hook = lambda phase, t, b: seen.append(torch.cuda.current_stream())
    outs = [{r: torch.full((wl.B, wl.H, wl.n[r], wl.d), float("nan"), dtype=torch.bfloat16, device="cuda")
             for r in ROLES} for _ in range(n_blocks)]

    def after(t, b):
        seen.append(torch.cuda.current_stream())
        copies.append(outs[b]["tgt"].clone())

    torch.cuda.synchronize()
    ex.step(0, xs[0], outs, stream=stream, after_block=after)
    torch.cuda.synchronize()
    ex.check()
    assert len(seen) == 3 * n_blocks and all(any(s == a for a in allowed) for s in seen)
    assert all(torch.equal(c, o["tgt"]) for c, o in zip(copies, outs))


@pytest.mark.parametrize("fused", [True, False])
def test_assigned_buffers_are_used(cuda_ok, fused):
    """A buffer that the caller assigns to the executor is the one that its next launches take."""
    wl, ex, xs = _setup(2, fused_cache=fused)
    _, same, _ = _setup(2, fused_cache=fused)
    names = ("cache_k", "cache_v", "cache_x", "a_b", "mass", "D", "modes", "gbar", "M")
    old = {k: getattr(ex, k) for k in names}
    kept = {k: x.clone() for k, x in old.items()}
    for k in names:
        setattr(ex, k, old[k].clone())
    for t in range(2):
        ex.step(t, xs[t])
        same.step(t, xs[t])
    torch.cuda.synchronize()
    ex.check()
    for k in names:
        assert torch.equal(old[k], kept[k]), k
        assert torch.equal(getattr(ex, k).nan_to_num(), getattr(same, k).nan_to_num()), k
    assert (ex.modes[0] == 3).all() and (ex.a_b >= 0).all()
