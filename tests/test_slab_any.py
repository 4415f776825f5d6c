"""The slab kernel fed through registers (odd vocabularies, unaligned matrices) and with k > 32: what the automatic
choice runs where no other fast kernel takes the shape.  Against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_10453_b200 import binding, synth
from parity import check_topk

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    c = binding.Context(max_M=140, max_d=2048, max_V=160000, max_k=64)
    yield c
    c.close()


def unaligned(t, off):
    """The same matrix `off` elements into a buffer with NaN around it: reading outside would show."""
    buf = torch.full((t.numel() + 64,), float("nan"), dtype=t.dtype, device=DEV)
    v = buf[off:off + t.numel()].view(t.shape)
    v.copy_(t)
    return v


# M, d, r, V, k, offsets (elements) of h, A, B
SHAPES = [
    (1, 8, 2, 37, 37, (0, 0, 0)),             # one stage, V below a box
    (2, 33, 7, 1001, 10, (1, 3, 5)),          # odd d and r, everything unaligned
    (8, 64, 32, 16003, 33, (0, 0, 0)),        # exactly one stage; three selection variants from here on
    (9, 96, 33, 20001, 64, (0, 8, 1)),        # one row past a stage
    (16, 72, 65, 8 * 2401 + 2, 20, (0, 0, 2)),
    (17, 130, 40, 8 * 3001 + 4, 12, (0, 0, 4)),
    (33, 64, 48, 50257, 25, (0, 0, 0)),
    (64, 64, 24, 30011, 40, (0, 0, 7)),
    (70, 100, 20, 9973, 5, (0, 0, 0)),        # two launches
    (3, 128, 64, 8 * 2000, 48, (0, 0, 0)),    # TMA, k > 32
    (140, 64, 16, 8 * 900, 64, (0, 0, 0)),    # TMA, k > 32, three launches, narrow slabs
    (2, 64, 16, 8 * 1100, 9, (0, 0, 3)),      # a good shape at a bad address
]


@pytest.mark.parametrize("M,d,r,V,k,off", SHAPES)
def test_any_shape_matches_oracle(ctx, M, d, r, V, k, off):
    x = synth.make_inputs(M, d, r, V, seed=31)
    b = {n: oracle.bf16_bits(t) for n, t in x.items()}
    h, A, B = (unaligned(x[n], o) for n, o in zip(("h", "A", "B"), off))
    ids, lp = ctx.slimspec_head_topk(h, A, B, k)
    again = ctx.slimspec_head_topk(h, A, B, k)
    torch.cuda.synchronize()
    assert ctx.last_error() == binding.OK and ctx.last_path() == binding.PATH_GENERIC
    st = check_topk(oracle.head_topk(b["h"], b["A"], b["B"], k), ids.cpu().numpy(), lp.cpu().numpy())
    # the code keeps 24 bits; fp32 sums of at most 130 terms
    assert st["max_lp_err"] < 2e-5
    assert torch.equal(ids, again[0]) and torch.equal(lp, again[1])
    buf = torch.full((M * V + 512,), 12345.0, dtype=torch.float32, device=DEV)
    out = ctx.slimspec_head_logits(h, A, B, out_logits=buf[256:256 + M * V].view(M, V))
    torch.cuda.synchronize()
    assert torch.all(buf[:256] == 12345.0) and torch.all(buf[256 + M * V:] == 12345.0)
    ref = oracle.slimspec_logits(b["h"], b["A"], b["B"])
    assert np.max(np.abs(out.cpu().numpy().astype(np.float64) - ref)) < 1e-4     # (k <= 32 at a good shape: 17 bits of the code)


@pytest.mark.parametrize("M,d,V,k", [(3, 37, 1003, 9), (20, 256, 30011, 50)])
def test_any_fullhead_and_equal_logits(ctx, M, d, V, k):
    h = synth.make_h(M, d, 3)
    h[M // 2:] = 0                  # all logits of these rows are equal: the lowest ids win
    W = synth.make_W(d, V, 3)
    ids, lp = ctx.fullhead_topk(h.to(DEV), W.to(DEV), k)
    torch.cuda.synchronize()
    assert ctx.last_error() == binding.OK and ctx.last_path() == binding.PATH_GENERIC
    st = check_topk(oracle.fullhead_topk(oracle.bf16_bits(h), oracle.bf16_bits(W), k), ids.cpu().numpy(), lp.cpu().numpy())
    assert st["max_lp_err"] < 2e-5
    assert ids[M // 2:].cpu().tolist() == [list(range(k))] * (M - M // 2)
