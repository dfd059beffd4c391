"""The three-branch block with several groups per 128-token tile (groups of 32 and 64 on the tensor cores), at the edges of
groups and tiles, and cut along the sequence."""
import numpy as np
import pytest
import torch

from oracle import la_oracle as orc
from paper_2406_07368_b200 import binding, workloads as wl
from tests._util import TOL, rel_err

pytestmark = pytest.mark.gpu


def _run(C, T, W, phi, eps, alpha, first=0, B=1, H=3, workspace=False):
    d, io = 128, "bf16"
    q, k, v = wl.qkv(41 + T, (B, H, first + T, d), 0.5, io, v_mean=1.0)
    w = wl.conv_weights(41, H, d, W)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(torch.bfloat16).cuda()   # noqa: E731
    wd = torch.from_numpy(w).cuda()
    ctx = binding.Context(H, d, W, phi, eps, io)
    st = ctx.new_state(B)
    args = (C, alpha, d ** -0.5)
    if first:
        ctx.la_prefill_grouped(dev(q[:, :, :first]), dev(k[:, :, :first]), dev(v[:, :, :first]), wd, st, *args)
    if workspace:
        need = ctx.la_prefill_workspace_bytes(B, T)
        assert need > 0
        ws = torch.full((need,), 0xff, dtype=torch.uint8, device="cuda")
        ctx.la_set_workspace(ws)
    o = ctx.la_prefill_grouped(dev(q[:, :, first:]), dev(k[:, :, first:]), dev(v[:, :, first:]), wd, st, *args,
                               init_state=first > 0)
    assert ctx.la_last_device_status() == binding.LA_OK
    if workspace:
        assert (ws != 0xff).any()                                # the cut was made
    want, ost = orc.prefill_grouped_block(q, k, v, w, phi, eps, C, alpha, d ** -0.5)
    got = o.float().cpu().numpy()
    assert rel_err(got, want[:, :, first:]) < TOL[io]
    for a in range(0, T, C):                                     # group by group: one wrong group cannot hide
        assert rel_err(got[:, :, a:a + C], want[:, :, first + a:first + a + C]) < TOL[io], a
    assert rel_err(st.S.cpu().numpy(), ost.S) < TOL[io] and rel_err(st.z.cpu().numpy(), ost.z) < TOL[io]
    assert st.pos.tolist() == [first + T] * B
    np.testing.assert_array_equal(st.win.float().cpu().numpy(), ost.win)


@pytest.mark.parametrize("C", [32, 64])
@pytest.mark.parametrize("T", [1, 31, 32, 33, 63, 65, 96, 127, 128, 129, 161, 390])
def test_edges(C, T):
    _run(C, T, 3, "elu1", 0.0, 0.8)


@pytest.mark.parametrize("C,W,phi,eps,alpha,first", [(32, 8, "elu1", 0.0, 1.0, 0), (64, 1, "relu", 1e-6, 0.7, 64),
                                                     (32, 3, "relu", 1e-6, 1.3, 96), (64, 3, "elu1", 0.0, 0.0, 128),
                                                     (32, 16, "elu1", 0.0, 0.0, 32)])
def test_options_and_continuation(C, W, phi, eps, alpha, first):
    _run(C, 300, W, phi, eps, alpha, first)


@pytest.mark.parametrize("C,T,first,H", [(64, 900, 0, 36), (32, 770, 64, 2), (128, 1000, 0, 3), (100, 1200, 100, 40)])
def test_cut_along_the_sequence(C, T, first, H):
    """With a workspace: packed groups, one group per tile, and partly filled tiles (100 tokens)."""
    _run(C, T, 3, "elu1", 0.0, 1.0, first, H=H, workspace=True)


@pytest.mark.parametrize("C", [32, 64])
def test_scores_against_earlier_groups_of_a_tile_keep_the_precision_of_the_state(C):
    """The global branch where its values cancel: the tokens of group 0 come in pairs of nearly equal keys and opposite
    values, all other values are zero, so that the output of a later row of the tile is a small difference of large sums.
    ReLU of bf16 is exact, and what is left is the output's own rounding (2^-9 of it) and that of the scores: 2^-17 each in
    two bf16 parts, of a mean of values of size 1; one more bit for the sums."""
    d, H, T = 128, 3, 128
    g = np.random.default_rng(5)
    bf = lambda x: torch.from_numpy(x.astype(np.float32)).to(torch.bfloat16)              # noqa: E731
    q, k = bf(g.normal(0.5, 1.0, (1, H, T, d))), bf(g.normal(0.5, 1.0, (1, H, T, d)))
    k[:, :, 1:C:2] = k[:, :, 0:C:2] + bf(g.normal(0.0, 0.05, (1, H, C // 2, d)))
    v = torch.zeros(1, H, T, d, dtype=torch.bfloat16)
    v[:, :, 0:C:2], v[:, :, 1:C:2] = 1.0, -1.0
    ctx = binding.Context(H, d, 1, "relu", 1e-6, "bf16")
    o = ctx.la_prefill_grouped(q.cuda(), k.cuda(), v.cuda(), torch.zeros(H, d, 1, device="cuda"), ctx.new_state(1), C, 1.0,
                               d ** -0.5)
    f = lambda x: x.double().numpy()                                                       # noqa: E731
    want, _ = orc.prefill_grouped_block(f(q), f(k), f(v), np.zeros((H, d, 1)), "relu", 1e-6, C, 1.0, d ** -0.5)
    got, want = o.double().cpu().numpy()[:, :, C:], np.asarray(want)[:, :, C:]
    assert 1e-4 < np.abs(want).max() < 2e-2                      # small, as intended
    assert (np.abs(got - want) <= 2.0 ** -9 * np.abs(want) + 2.0 ** -16).all()


@pytest.mark.parametrize("C,T,W", [(32, 128, 3), (64, 128, 3), (32, 200, 8), (64, 250, 1)])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_values_that_are_not_finite_stay_behind_their_group(C, T, W, bad):
    """A value of a later group, in the same tile or the next one, that is not finite: the groups before it do not change."""
    d, H = 128, 2
    q, k, v = (torch.from_numpy(x).to(torch.bfloat16).cuda() for x in wl.qkv(7, (1, H, T, d), 0.5, "bf16", v_mean=1.0))
    w = torch.from_numpy(wl.conv_weights(7, H, d, W)).cuda()
    ctx = binding.Context(H, d, W, "elu1", 0.0, "bf16")
    clean = ctx.la_prefill_grouped(q, k, v, w, ctx.new_state(1), C, 1.0, d ** -0.5)
    for tok in range(C, T, C + 5):
        v2 = v.clone()
        v2[0, 1, tok, 77] = bad
        o = ctx.la_prefill_grouped(q, k, v2, w, ctx.new_state(1), C, 1.0, d ** -0.5)
        end = tok // C * C
        assert torch.equal(o[:, :, :end], clean[:, :, :end]), tok
        assert torch.equal(o[:, 0], clean[:, 0]) and not o[0, 1, tok, 77].isfinite()


@pytest.mark.parametrize("C,T,first,H", [(100, 1280, 0, 18), (96, 2306, 96, 8), (33, 700, 0, 32), (48, 2048, 48, 16)])
def test_cut_with_the_workspace_asked_for_without_a_group(C, T, first, H):
    """Tiles of other than 128 tokens: the number of segments must fit the workspace that la_prefill_workspace_bytes names."""
    _run(C, T, 3, "elu1", 0.0, 1.0, first, H=H, workspace=True)


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_values_that_are_not_finite_stay_behind_their_segment(bad):
    """Ten segments of seven 40-token groups, whose sums are formed in 128-token tiles by a launch of its own: the last tile of
    a segment overlaps the next one's first groups, a value of which must not enter the segment's sums."""
    C, T, H, d = 40, 2660, 8, 128
    q, k, v = (torch.from_numpy(x).to(torch.bfloat16).cuda() for x in wl.qkv(7, (1, H, T, d), 0.5, "bf16", v_mean=1.0))
    w = torch.from_numpy(wl.conv_weights(7, H, d, 3)).cuda()
    ctx = binding.Context(H, d, 3, "elu1", 0.0, "bf16")
    ws = torch.full((ctx.la_prefill_workspace_bytes(1, T),), 0xff, dtype=torch.uint8, device="cuda")
    ctx.la_set_workspace(ws)
    clean = ctx.la_prefill_grouped(q, k, v, w, ctx.new_state(1), C, 1.0, d ** -0.5)
    assert (ws != 0xff).any()
    for tok in (325, 370, 605):
        v2 = v.clone()
        v2[0, 1, tok, 77] = bad
        o = ctx.la_prefill_grouped(q, k, v2, w, ctx.new_state(1), C, 1.0, d ** -0.5)
        end = tok // C * C
        assert torch.equal(o[:, :, :end], clean[:, :, :end]), tok
