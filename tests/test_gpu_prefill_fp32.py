"""The chunked CUDA-core prefill at the edges of its chunks and of its cut along the sequence (clusters of up to 8 CTAs,
segments of whole chunks: 64 tokens at d = 64, 32 at d = 128)."""
import numpy as np
import pytest
import torch

from oracle import la_oracle as orc
from paper_2406_07368_b200 import binding, workloads as wl
from tests._util import rel_err

pytestmark = pytest.mark.gpu

# 1e-5: sums of up to ~600 products in fp32, 2^-24 each, in two nested orders, with room for the division (fp32 io); the
# bf16 case differs from the oracle by its rounded output alone (2^-8 of the value).
TOL = {"f32": 1e-5, "bf16": 5e-3}


def _run(io, d, T, W, phi, eps, B, H, first):
    q, k, v = wl.qkv(31, (B, H, T, d), 1.0 if io == "f32" else d ** -0.5, io, v_mean=0.5)
    w = wl.conv_weights(31, H, d, W)
    ctx = binding.Context(H, d, W, phi, eps, io)
    st, dev = ctx.new_state(B), lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(ctx.dtype).cuda()
    wd = torch.from_numpy(w).cuda()
    outs = []
    for a, b in ((0, first), (first, T)) if first else ((0, T),):
        outs.append(ctx.la_prefill(dev(q[:, :, a:b]), dev(k[:, :, a:b]), dev(v[:, :, a:b]), wd, st, init_state=a > 0))
    want, ost = orc.prefill_quadratic(q, k, v, w, phi, eps)
    assert rel_err(torch.cat(outs, 2).float().cpu().numpy(), want) < TOL[io]
    assert rel_err(st.S.cpu().numpy(), ost.S) < 1e-5 and rel_err(st.z.cpu().numpy(), ost.z) < 1e-5
    assert st.pos.tolist() == [T] * B
    if W > 1:
        tail = np.concatenate([np.zeros((B, H, W - 1, d), np.float32), v], 2)[:, :, -(W - 1):]
        assert np.array_equal(st.win.float().cpu().numpy(), tail)


@pytest.mark.parametrize("T", [1, 31, 32, 33, 63, 64, 65, 127, 129, 511, 512, 513, 577])
@pytest.mark.parametrize("d", [64, 128])
def test_chunk_and_segment_edges(d, T):
    _run("f32", d, T, 3, "elu1", 0.0, 1, 2, 0)


@pytest.mark.parametrize("io,d,W,phi,eps,first", [
    ("f32", 64, 1, "relu", 1e-6, 0), ("f32", 64, 32, "elu1", 0.0, 20), ("f32", 128, 32, "relu", 1e-6, 7),
    ("bf16", 64, 5, "elu1", 0.0, 65), ("bf16", 64, 32, "relu", 1e-6, 100), ("f32", 128, 2, "elu1", 0.0, 160)])
def test_options_and_continuation(io, d, W, phi, eps, first):
    _run(io, d, 200, W, phi, eps, 1, 3, first)


@pytest.mark.parametrize("d,B,H", [(64, 32, 7), (128, 10, 8)])
def test_one_block_per_chain_when_chains_abound(d, B, H):
    _run("f32", d, 100, 3, "elu1", 0.0, B, H, 40)


@pytest.mark.parametrize("d,phi,B,H,edges", [
    (64, "elu1", 1, 2, (25,)), (64, "relu", 1, 2, (22,)), (64, "elu1", 25, 8, (28,)), (64, "relu", 25, 8, (25,)),
    (64, "elu1", 64, 8, (41, 86)), (128, "elu1", 1, 2, (14, 34)), (128, "relu", 19, 8, (23, 52, 80)), (128, "elu1", 50, 8, (19, 44))])
def test_both_sides_of_the_lines_between_walking_and_chunks(d, phi, B, H, edges):
    """Short calls walk their tokens; the lines depend on the head dimension, the number of chains and phi.  A call on either
    side of each line continues 5 tokens (which are walked) and must agree with the oracle."""
    for T in (t + x for t in edges for x in (0, 1)):
        _run("f32", d, T + 5, 3, phi, 1e-6 if phi == "relu" else 0.0, B, H, 5)
