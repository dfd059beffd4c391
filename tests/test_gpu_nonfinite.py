"""Inputs that are not finite: a NaN must show in everything that depends on it, and only there."""
import pytest
import torch

from paper_2406_07368_b200 import binding, workloads as wl

pytestmark = pytest.mark.gpu

NAN = float("nan")


def _make(io, d, tokens, B=2, H=2, W=3, **kw):
    ctx = binding.Context(H, d, W, "elu1", 0.0, io, **kw)
    q, k, v = (torch.from_numpy(x).to(ctx.dtype).cuda() for x in wl.qkv(3, (B, H, *tokens, d), 0.5, io))
    w = torch.from_numpy(wl.conv_weights(3, H, d, W)).cuda()
    st = ctx.new_state(B)
    st.S.normal_()
    st.z.uniform_(1, 2)
    return ctx, q, k, v, w, st


def _state_hit(st, b, h, a):
    """Feature a of (b, h) is NaN in S and z, everything else is finite."""
    assert st.z[b, h, a].isnan() and st.z.isnan().sum() == 1
    assert st.S[b, h, a].isnan().all() and st.S.isnan().sum() == st.S.shape[3]


@pytest.mark.parametrize("io,d", [("f32", 64), ("f32", 128), ("bf16", 64), ("bf16", 128)])
def test_nan_in_k_reaches_the_state(io, d):
    ctx, q, k, v, w, st = _make(io, d, ())
    k[1, 0, 5] = NAN
    o = ctx.la_decode_step(q, k, v, w, st)
    _state_hit(st, 1, 0, 5)
    assert o[1, 0].isnan().all() and o[0].isfinite().all() and o[1, 1].isfinite().all()

    parent = torch.arange(-1, 3, dtype=torch.int32).repeat(2, 1).cuda()
    ctx, q, k, v, w, st = _make(io, d, (4,))
    k[0, 1, 2, 7] = NAN
    ctx.la_commit(k, v, parent, torch.tensor([3, 3], dtype=torch.int32).cuda(), st)
    _state_hit(st, 0, 1, 7)

    ctx, q, k, v, w, st = _make(io, d, (40,))
    k[0, 1, 20, 7] = NAN
    o = ctx.la_prefill(q, k, v, w, st)
    _state_hit(st, 0, 1, 7)
    assert o[0, 1, 20:].isnan().all() and o[0, 1, :20].isfinite().all() and o[1].isfinite().all()
    dS, dz = ctx.la_segment_state(k, v)
    assert dz[0, 1, 7].isnan() and dz.isnan().sum() == 1 and dS[0, 1, 7].isnan().all()


@pytest.mark.parametrize("io,d,cuda_cores", [("f32", 64, False), ("f32", 128, False), ("bf16", 64, False), ("bf16", 128, True),
                                             ("bf16", 128, False)])
def test_nan_in_q_or_k_reaches_the_outputs(io, d, cuda_cores):
    parent = torch.tensor([-1, 0, 0, 1], dtype=torch.int32).repeat(2, 1).cuda()
    for name, hit in (("q", [1]), ("k", [1, 3])):              # node 1 itself; node 1 and its child, not its sibling
        ctx, q, k, v, w, st = _make(io, d, (4,))
        ctx.la_set_prefill_kernel(int(cuda_cores))
        dict(q=q, k=k)[name][1, 0, 1, 9] = NAN
        o = ctx.la_verify_tree(q, k, v, parent, w, st)
        if cuda_cores or io == "f32" or d == 64:
            assert o[1, 0, hit].isnan().all() and o.isnan().sum() == len(hit) * d
        else:
            assert o[1, 0, hit].isnan().all()
    ctx, q, k, v, w, st = _make(io, d, (40,))
    ctx.la_set_prefill_kernel(int(cuda_cores))
    q[1, 0, 33, 9] = NAN
    o = ctx.la_prefill(q, k, v, w, st)
    assert o[1, 0, 33].isnan().all() and o.isnan().sum() == d
    o = ctx.la_prefill_grouped(q, k, v, w, st, 16, 1.0, d ** -0.5)
    assert o[1, 0, 33].isnan().all() and o.isnan().sum() == d


@pytest.mark.parametrize("io,d", [("f32", 64), ("f32", 128), ("bf16", 64)])
@pytest.mark.parametrize("bad", [float("inf"), NAN])
def test_value_that_is_not_finite_reaches_no_earlier_token(io, d, bad):
    """The CUDA-core prefill: the outputs before a token whose value is not finite do not change."""
    T = 150
    ctx, q, k, v, w, st = _make(io, d, (T,))
    clean = ctx.la_prefill(q, k, v, w, st)
    for tok in (0, 1, 15, 16, 31, 32, 33, 47, 63, 64, 100, 127, 128, 149):
        v2 = v.clone()
        v2[0, 1, tok, 3] = bad
        o = ctx.la_prefill(q, k, v2, w, st)
        assert torch.equal(o[0, 1, :tok], clean[0, 1, :tok]) and torch.equal(o[1], clean[1]), tok
        assert not o[0, 1, tok:, 3].isfinite().any(), tok
        assert torch.equal(o[0, 1, :, :3], clean[0, 1, :, :3]) and torch.equal(o[0, 1, :, 4:], clean[0, 1, :, 4:])
