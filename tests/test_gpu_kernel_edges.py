"""Sizes at which single kernels can go wrong: the tap sums of long windows, the pass over a segment that forms its sums, the
commit of paths of every length."""
import numpy as np
import pytest
import torch

from oracle import la_oracle as orc
from paper_2406_07368_b200 import binding, workloads as wl
from tests._util import TOL, rel_err

pytestmark = pytest.mark.gpu


def _dev(x, io="bf16"):
    return torch.from_numpy(np.ascontiguousarray(x)).to(binding.TORCH_DTYPE[io]).cuda()


@pytest.mark.parametrize("W", [6, 8, 9, 10, 16, 17, 18, 24, 25, 26, 31, 32])
@pytest.mark.parametrize("T,first", [(1, 0), (127, 0), (129, 3), (300, 40)])
def test_tap_sums_of_long_windows(W, T, first):
    """ReLU of negative queries: no attention term, the output is the tap sum alone, rounded to bf16 (up to 2^-8 of it: 8 bits).  Up
    to 32 products are added in fp32, 2^-24 each of a partial sum no larger than that of the magnitudes: 2^-16 covers them."""
    H, d = 3, 128
    _, k, v = wl.qkv(W + T, (1, H, first + T, d), 1.0, "bf16")
    w = wl.conv_weights(W, H, d, W)
    q = -np.ones_like(v)
    ctx = binding.Context(H, d, W, "relu", 1e-6, "bf16")
    st, wd = ctx.new_state(1), torch.from_numpy(w).cuda()
    if first:
        ctx.la_prefill(*(_dev(x[:, :, :first]) for x in (q, k, v)), wd, st)
    got = ctx.la_prefill(*(_dev(x[:, :, first:]) for x in (q, k, v)), wd, st, init_state=first > 0).double().cpu().numpy()
    want, mag = np.zeros(v.shape), np.zeros(v.shape)
    for t in range(W):
        term = w[None, :, :, t][:, :, None].astype(np.float64) * np.pad(v, ((0, 0), (0, 0), (t, 0), (0, 0)))[:, :, :first + T]
        want += term
        mag += np.abs(term)
    want, mag = want[:, :, first:], mag[:, :, first:]
    assert ctx.la_last_device_status() == binding.LA_OK
    assert (np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 2.0 ** -16 * mag).all()
    np.testing.assert_array_equal(st.win.float().cpu().numpy(), np.pad(v, ((0, 0), (0, 0), (W - 1, 0), (0, 0)))[:, :, first + T:])


@pytest.mark.parametrize("C,T,W", [(32, 200, 20), (64, 300, 32 - 8), (32, 128, 10)])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_tap_sums_keep_values_that_are_not_finite_to_their_window(C, T, W, bad):
    """In the three-branch mode nothing but the window joins a token with the groups before its own: bit for bit the same
    there, and in the other channels everywhere."""
    d, H = 128, 2
    q, k, v = (_dev(x) for x in wl.qkv(7, (1, H, T, d), 0.5, "bf16", v_mean=1.0))
    w = torch.from_numpy(wl.conv_weights(7, H, d, W)).cuda()
    ctx = binding.Context(H, d, W, "elu1", 0.0, "bf16")
    clean = ctx.la_prefill_grouped(q, k, v, w, ctx.new_state(1), C, 1.0, d ** -0.5)
    for tok in range(C, T, C + 5):
        v2 = v.clone()
        v2[0, 1, tok, 77] = bad
        o = ctx.la_prefill_grouped(q, k, v2, w, ctx.new_state(1), C, 1.0, d ** -0.5)
        end = tok // C * C
        assert torch.equal(o[:, :, :end], clean[:, :, :end]), tok
        assert torch.equal(o[0, 1, :, :77], clean[0, 1, :, :77]) and torch.equal(o[0, 1, :, 78:], clean[0, 1, :, 78:]), tok
        assert not o[0, 1, tok:tok + W, 77].isfinite().any(), tok


@pytest.mark.parametrize("tiles", [2, 3, 4, 5, 7])
@pytest.mark.parametrize("W,group", [(3, 0), (9, 0), (3, 64), (3, 100)])
def test_segments_of_few_tiles(tiles, W, group):
    """32 chains in four segments of `tiles` tiles, the last one ragged, continuing: as the call that is not cut (only the order
    of fp32 sums and the roundings behind it differ: a few bf16 ulps)."""
    H, d, tile = 32, 128, 100 if group == 100 else 128
    T, first = 4 * tiles * tile - 19, 192 if group == 64 else 200       # (781 tokens in tiles of 100 are still seven of 128)
    q, k, v = (_dev(x) for x in wl.qkv(tiles, (1, H, first + T, d), d ** -0.5, "bf16", v_mean=0.5))
    w = torch.from_numpy(wl.conv_weights(5, H, d, W)).cuda()
    ctx = binding.Context(H, d, W, "elu1", 0.0, "bf16")
    cut = lambda x, a, b: x[:, :, a:b].contiguous()                                        # noqa: E731

    def call(a, b, st):
        x = [cut(y, a, b) for y in (q, k, v)]
        if group:
            return ctx.la_prefill_grouped(*x, w, st, group, 1.0, d ** -0.5, init_state=a > 0)
        return ctx.la_prefill(*x, w, st, init_state=a > 0)

    got = []
    for lend in (True, False):
        st = ctx.new_state(1)
        ctx.la_set_workspace(None)
        call(0, first, st)
        if lend:
            ws = torch.full((ctx.la_prefill_workspace_bytes(1, T),), 0xff, dtype=torch.uint8, device="cuda")
            ctx.la_set_workspace(ws)
        got.append((call(first, first + T, st), st))
    assert ctx.la_last_device_status() == binding.LA_OK
    S_seg = ws[:32 * 4 * d * d * 4].view(32, 4, -1)                     # a state per chain and segment: the first three are formed
    assert (S_seg[:, :3] != 0xff).any(-1).all()
    (a, sa), (b, sb) = got
    assert rel_err(a.float().cpu().numpy(), b.float().cpu().numpy()) < 1.2e-2
    assert rel_err(sa.S.cpu().numpy(), sb.S.cpu().numpy()) < 1e-4 and rel_err(sa.z.cpu().numpy(), sb.z.cpu().numpy()) < 1e-4
    assert torch.equal(sa.win, sb.win) and torch.equal(sa.pos, sb.pos)


@pytest.mark.parametrize("io,d", [("f32", 64), ("f32", 128), ("bf16", 64), ("bf16", 128)])
@pytest.mark.parametrize("W", [1, 3, 12])
@pytest.mark.parametrize("H,depth,phi", [(2, 64, "elu1"), (2, 64, "relu"), (10, 16, "relu"), (10, 33, "elu1"), (20, 16, "elu1")])
def test_commit_of_paths_of_every_length(io, d, W, H, depth, phi):
    """Chains of 64 nodes, accepted up to every node there is (rank-1 updates in order, and the window's rows).  With d = 128 on 148
    SMs: 38 units fit in one wave of five blocks per SM, 190 in one of six (not with paths of 33), 380 take three waves of five."""
    N = 64
    lens = [0, 1, 2, 3, 4, 5, 7, 8, 9, 12, 15, 16, 17, 31, 32, 33, 48, 63, 64]
    lens = [min(n, depth) for n in lens]
    B = len(lens)
    _, k, v = wl.qkv(11, (B, H, N, d), 0.3, io)
    parent, accept = np.stack([wl.chain_tree(N)] * B), np.array(lens, dtype=np.int32) - 1
    ctx = binding.Context(H, d, W, phi, 0.0, io, max_nodes=64, max_depth=depth)
    st = ctx.new_state(B)
    g = np.random.default_rng(3)
    S, z = g.normal(size=st.S.shape).astype(np.float32), g.uniform(1, 2, st.z.shape).astype(np.float32)
    win = g.integers(-4, 5, st.win.shape).astype(np.float32)
    st.S.copy_(torch.from_numpy(S)), st.z.copy_(torch.from_numpy(z)), st.win.copy_(torch.from_numpy(win))
    path, n = ctx.la_commit(_dev(k, io), _dev(v, io), torch.from_numpy(parent).cuda(), torch.from_numpy(accept).cuda(), st)
    assert ctx.la_last_device_status() == binding.LA_OK
    assert n.tolist() == lens
    fk = np.where(k > 0, k + 1.0, np.exp(np.minimum(k, 0.0))) if phi == "elu1" else np.maximum(k, 0.0)
    for b, L in enumerate(lens):
        assert path[b].tolist() == list(range(L)) + [-1] * (depth - L)
        assert rel_err(st.S[b].cpu().numpy(), S[b] + np.einsum("hna,hnc->hac", fk[b, :, :L], v[b, :, :L])) < TOL["f32"]
        assert rel_err(st.z[b].cpu().numpy(), z[b] + fk[b, :, :L].sum(1)) < TOL["f32"]
        rows = np.concatenate([win[b], v[b, :, :L]], axis=1)
        np.testing.assert_array_equal(st.win[b].float().cpu().numpy(), rows[:, rows.shape[1] - (W - 1):])
    assert st.pos.tolist() == lens
