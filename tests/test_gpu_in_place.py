"""Prefill in place: the outputs stored over q, k or v."""
import pytest
import torch

from paper_2406_07368_b200 import binding, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io,d,W,H,T", [("f32", 64, 3, 2, 20), ("f32", 64, 32, 3, 700), ("f32", 128, 32, 3, 300),
                                        ("bf16", 64, 5, 2, 333), ("f32", 64, 4, 300, 130), ("bf16", 128, 3, 2, 300),
                                        ("bf16", 128, 8, 2, 300), ("bf16", 128, 4, 20, 900),
                                        # cut into 24, 10 and 16 segments, and into 3 that are too many for clusters
                                        ("bf16", 128, 3, 2, 3000), ("bf16", 128, 32, 8, 2400), ("bf16", 128, 5, 9, 2048),
                                        ("bf16", 128, 9, 47, 900)])
@pytest.mark.parametrize("over", ["q", "k", "v"])
def test_outputs_over_an_input(io, d, W, H, T, over):
    ctx = binding.Context(H, d, W, "elu1", 0.0, io)
    need = ctx.la_prefill_workspace_bytes(1, T)
    if need:
        ctx.la_set_workspace(torch.empty(need, dtype=torch.uint8, device="cuda"))
    x = {n: torch.from_numpy(a).to(ctx.dtype).cuda() for n, a in zip("qkv", wl.qkv(9, (1, H, T, d), 0.5, io))}
    w = torch.from_numpy(wl.conv_weights(9, H, d, W)).cuda()
    sts = []
    for init in (False, True):
        st = ctx.new_state(1)
        ctx.la_prefill(x["q"], x["k"], x["v"], w, st)
        sts.append(st)
        st2 = st.clone()
        want = ctx.la_prefill(x["q"], x["k"], x["v"], w, st, init_state=init)
        y = {n: a.clone() for n, a in x.items()}
        got = ctx.la_prefill(y["q"], y["k"], y["v"], w, st2, init_state=init, out=y[over])
        assert got is y[over] and torch.equal(got, want)
        for n in ("S", "z", "win", "pos"):
            assert torch.equal(getattr(st2, n), getattr(st, n)), n


@pytest.mark.parametrize("spare", [0, 1])
def test_over_v_with_just_too_little_workspace(spare):
    """One byte less than la_prefill_workspace_bytes: still cut where the outputs go elsewhere, one block per chain over v."""
    H, d, W, T = 3, 128, 4, 2000
    ctx = binding.Context(H, d, W, "elu1", 0.0, "bf16")
    q, k, v = (torch.from_numpy(a).to(ctx.dtype).cuda() for a in wl.qkv(9, (1, H, T, d), 0.5, "bf16"))
    w = torch.from_numpy(wl.conv_weights(9, H, d, W)).cuda()
    call = lambda out=None: ctx.la_prefill(q, k, v, w, ctx.new_state(1), out=out)                 # noqa: E731
    uncut = call()
    ctx.la_set_workspace(torch.empty(ctx.la_prefill_workspace_bytes(1, T) - 1 + spare, dtype=torch.uint8, device="cuda"))
    cut = call()
    assert not torch.equal(cut, uncut)
    assert torch.equal(call(out=v), cut if spare else uncut)
