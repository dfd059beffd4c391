"""The prefill cut along the sequence with few segments per chain (one cluster per chain, whose blocks form the segments'
sums and add them up as they load their state), at the smallest lengths that are cut, ragged and not, fresh and
continuing; and with up to 8 segments, which is as many as a cluster has, and more, which take launches of their own."""
import numpy as np
import pytest
import torch

from oracle import la_oracle as orc
from paper_2406_07368_b200 import binding, workloads as wl
from tests._util import rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,T,W,first", [(36, 768, 3, 0), (36, 641, 3, 70), (74, 700, 1, 130), (37, 769, 5, 3), (40, 900, 32, 33),
                                         (49, 2000, 2, 0), (18, 1024, 3, 0), (18, 1024, 4, 5), (16, 1152, 8, 40), (21, 900, 6, 0),
                                         (13, 1400, 3, 128)])
def test_split_with_few_segments(H, T, W, first):
    """`first` tokens in a call of their own, then T in one that is cut; against the oracle on all of them (bf16: 2e-2, the
    tolerance of every tensor-core path) and against the same call without the workspace (only the order of fp32 sums and
    the roundings behind it differ: a few bf16 ulps)."""
    d, io = 128, "bf16"
    q, k, v = wl.qkv(H + T, (1, H, first + T, d), d ** -0.5, io, v_mean=0.5)
    w = wl.conv_weights(5, H, d, W)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(torch.bfloat16).cuda()   # noqa: E731
    wd = torch.from_numpy(w).cuda()
    ctx = binding.Context(H, d, W, "elu1", 0.0, io)
    outs, states = [], []
    for lend in (True, False):
        st = ctx.new_state(1)
        need = ctx.la_prefill_workspace_bytes(1, T)
        assert need > 0
        ctx.la_set_workspace(None)
        if first:
            ctx.la_prefill(dev(q[:, :, :first]), dev(k[:, :, :first]), dev(v[:, :, :first]), wd, st)
        if lend:
            ctx.la_set_workspace(torch.full((need,), 0xff, dtype=torch.uint8, device="cuda"))
        outs.append(ctx.la_prefill(dev(q[:, :, first:]), dev(k[:, :, first:]), dev(v[:, :, first:]), wd, st, init_state=first > 0))
        states.append(st)
    assert ctx.la_last_device_status() == binding.LA_OK
    want, ost = orc.prefill_quadratic(q, k, v, w, "elu1", 0.0)
    got = outs[0].float().cpu().numpy()
    assert rel_err(got, want[:, :, first:]) < 2e-2
    assert rel_err(got, outs[1].float().cpu().numpy()) < 1.2e-2
    for st in states:
        assert rel_err(st.S.cpu().numpy(), ost.S) < 2e-2 and rel_err(st.z.cpu().numpy(), ost.z) < 2e-2
        assert st.pos.tolist() == [first + T]
    assert torch.equal(states[0].win, states[1].win)


def test_state_sums_of_many_tiles_over_and_over():
    """The passes that only form sums run ahead of the products as far as two buffers allow: segments of two tiles and more,
    many calls, every one bit for bit the same and none with a wait that ran out."""
    ctx = binding.Context(36, 128, 3, "elu1", 0.0, "bf16")
    for T in (900, 2500, 6000):                                  # one launch of clusters; per-segment sums of 2 to 12 tiles
        q, k, v = (torch.from_numpy(x).to(torch.bfloat16).cuda() for x in wl.qkv(T, (1, 36, T, 128), 0.1, "bf16"))
        w = torch.from_numpy(wl.conv_weights(5, 36, 128, 3)).cuda()
        ctx.la_set_workspace(torch.empty(ctx.la_prefill_workspace_bytes(1, T), dtype=torch.uint8, device="cuda"))
        first = None
        for _ in range(50):
            st = ctx.new_state(1)
            got = (ctx.la_prefill(q, k, v, w, st), st.S, *ctx.la_segment_state(k, v))
            first = first or got
            assert all(torch.equal(a, b) for a, b in zip(got, first))
    assert ctx.la_last_device_status() == binding.LA_OK
