"""The native side of the binding: what it refuses, and the output buffers it makes."""
import numpy as np
import pytest
import torch

from paper_2406_07368_b200 import binding, workloads as wl

pytestmark = pytest.mark.gpu


def _inputs(io="bf16", B=2, H=2, d=128, N=8, W=3):
    ctx = binding.Context(H, d, W, "elu1", 0.0, io, max_nodes=16, max_depth=4)
    q, k, v = (torch.from_numpy(x).to(ctx.dtype).cuda() for x in wl.qkv(11, (B, H, N, d), 1.0, io))
    w = torch.from_numpy(wl.conv_weights(11, H, d, W)).cuda()
    return ctx, q, k, v, w, ctx.new_state(B)


def test_refusals():
    ctx, q, k, v, w, st = _inputs()
    for bad, what in ((q.float(), "dtype"), (q[:, :, :5], "contiguous"), (q.cpu(), "CUDA"), (q[:1], "shape")):
        with pytest.raises(ValueError, match=what):
            ctx.la_prefill(q, bad, v, w, st)
    with pytest.raises(ValueError, match="state.S"):
        ctx.la_prefill(q[:1].contiguous(), k[:1].contiguous(), v[:1].contiguous(), w, st)
    with pytest.raises(ValueError):
        ctx.la_decode_step(q, k, v, w, st)                       # one dimension too many
    with pytest.raises(TypeError):
        ctx.la_prefill("q", k, v, w, st)
    with pytest.raises(binding.LaError) as e:                    # a missing tensor is the library's to refuse
        ctx.la_prefill(q, None, v, w, st)
    assert e.value.code == binding.LA_ERR_INVALID_ARG
    ctx.close()
    with pytest.raises(binding.LaError) as e:
        ctx.la_prefill(q, k, v, w, st)
    assert e.value.code == binding.LA_ERR_INVALID_ARG


@pytest.mark.parametrize("given_path", [False, True])
@pytest.mark.parametrize("given_len", [False, True])
def test_commit_outputs_of_skipped_sequences(given_path, given_len):
    """A malformed tree leaves the caller's buffers alone; buffers the binding makes read "no path, length 0"."""
    ctx, q, k, v, w, st = _inputs()
    parent = np.stack([wl.chain_tree(8)] * 2)
    parent[1, 2] = 5                                             # parent after child
    dirty = torch.full((1 << 16,), 77, dtype=torch.int32, device="cuda")
    del dirty                                                    # what a new buffer gets is not zero by luck
    path = torch.full((2, 4), 55, dtype=torch.int32, device="cuda") if given_path else None
    length = torch.full((2,), 55, dtype=torch.int32, device="cuda") if given_len else None
    path, length = ctx.la_commit(k, v, torch.from_numpy(parent).cuda(), torch.full((2,), 2, dtype=torch.int32, device="cuda"),
                                 st, path_out=path, commit_len=length)
    assert ctx.la_last_device_status() == binding.LA_ERR_BAD_TREE
    assert path.tolist() == [[0, 1, 2, -1], [55] * 4 if given_path else [-1] * 4]
    assert length.tolist() == [3, 55 if given_len else 0]


def test_calls_on_a_given_stream():
    ctx, q, k, v, w, st = _inputs()
    want = ctx.la_prefill(q, k, v, w, st)
    st2, out, s = ctx.new_state(2), torch.full_like(q, 7.0), torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        torch.cuda._sleep(200_000_000)                           # about 0.1 s in front of the call on its stream
    got = ctx.la_prefill(q, k, v, w, st2, out=out, stream=s)
    before = out.clone()                                         # on the current stream, which the call must not be on
    torch.cuda.current_stream().synchronize()
    assert not s.query()
    assert (before == 7.0).all()
    s.synchronize()
    assert got is out and torch.equal(got, want)


def test_state_whose_tensors_are_views_made_on_access():
    """A state out of a larger pool: every access makes a new view, which nothing but the call itself keeps alive."""
    ctx, q, k, v, w, st = _inputs()
    want = ctx.la_prefill(q, k, v, w, st)
    pool = ctx.new_state(6)

    class Slice:
        S = property(lambda self: pool.S[2:4])
        z = property(lambda self: pool.z[2:4])
        win = property(lambda self: pool.win[2:4])
        pos = property(lambda self: pool.pos[2:4])

    for _ in range(20):
        assert torch.equal(ctx.la_prefill(q, k, v, w, Slice()), want)
    assert torch.equal(pool.S[2:4], st.S) and torch.equal(pool.win[2:4], st.win) and pool.pos.tolist() == [0, 0, 8, 8, 0, 0]
    assert not pool.S[:2].any() and not pool.S[4:].any()


def test_numbers_are_taken_as_int_and_float_take_them():
    ctx, q, k, v, w, st = _inputs()
    want = ctx.la_prefill_grouped(q, k, v, w, st, 32, 1.0, 0.5)
    for group, alpha, scale in ((32.0, 1, np.float32(0.5)), (np.int64(32), torch.tensor(1.0), "0.5"), (torch.tensor(32), True, 0.5)):
        assert torch.equal(ctx.la_prefill_grouped(q, k, v, w, st, group, alpha, scale), want)
    with pytest.raises(TypeError):
        ctx.la_prefill_grouped(q, k, v, w, st, None, 1.0, 0.5)
    with pytest.raises(ValueError):
        ctx.la_prefill_grouped(q, k, v, w, st, 32, "one", 0.5)
