"""The slab kernel (vocabulary on the tensor cores' M side): sizes at the edges of its tiles, stages, row groups and
selection variants, against the fp64 oracle."""
import pytest
import torch

import oracle
from paper_2605_10453_b200 import binding, synth
from parity import check_topk

pytestmark = pytest.mark.gpu

DEV = "cuda:0"

# M, d, r, V, k
SHAPES = [
    (3, 256, 16, 8 * 149, 1),          # one stage, half of it past K; slabs of 8 columns
    (7, 128, 48, 8 * 600, 13),         # K no multiple of a stage; second selection variant (k > 12)
    (8, 512, 64, 64 * 593, 12),        # units of 64 columns, the last slabs one unit narrower
    (9, 256, 80, 8 * 1300, 32),        # stacked parts, 16 rows
    (16, 512, 96, 129 * 148 * 8, 10),  # just over eight tiles
    (17, 256, 64, 8 * 2500, 10),       # 32-row group, mostly empty
    (31, 256, 128, 8 * 1501, 5),
    (33, 256, 128, 8 * 1501, 10),      # three groups of 16
    (48, 192, 64, 8 * 4001, 10),
    (49, 128, 112, 8 * 801, 10),
    (64, 512, 256, 8 * 5000, 32),
    (64, 128, 64, 64, 10),             # one unit per CTA, fewer CTAs than SMs
    (130, 72, 32, 8 * 777, 4),         # three launches (the tensor path does not take this hidden size)
]


@pytest.fixture(scope="module")
def ctx():
    c = binding.Context(max_M=130, max_d=2048, max_V=160000, max_k=32)
    yield c
    c.close()


def _check(ref, ids, lp):
    # the code keeps 17 bits, sums are fp32 over at most 2048 terms of size 1: 1e-4 is ten times what that gives
    assert check_topk(ref, ids.cpu().numpy(), lp.cpu().numpy())["max_lp_err"] < 1e-4


@pytest.mark.parametrize("M,d,r,V,k", SHAPES)
def test_slab_head_matches_oracle(ctx, M, d, r, V, k):
    x = synth.make_inputs(M, d, r, V, seed=23)
    g = {n: t.to(DEV) for n, t in x.items()}
    b = {n: oracle.bf16_bits(t) for n, t in x.items()}
    ids, lp = ctx.slimspec_head_topk(g["h"], g["A"], g["B"], k)
    again = ctx.slimspec_head_topk(g["h"], g["A"], g["B"], k)
    torch.cuda.synchronize()
    assert ctx.last_error() == binding.OK and ctx.last_path() == binding.PATH_STREAM
    _check(oracle.head_topk(b["h"], b["A"], b["B"], k), ids, lp)
    assert torch.equal(ids, again[0]) and torch.equal(lp, again[1])


@pytest.mark.parametrize("M,d,V,k", [(5, 200, 8 * 1300, 10), (40, 264, 8 * 901, 7)])
def test_slab_fullhead_and_equal_logits(ctx, M, d, V, k):
    """Full rank (one part, K no multiple of a stage); the second half of the rows are zero: all their logits
    are equal, more candidates than any list takes, and the lowest ids win."""
    h = synth.make_h(M, d, 3)
    h[M // 2:] = 0
    W = synth.make_W(d, V, 3)
    ids, lp = ctx.fullhead_topk(h.to(DEV), W.to(DEV), k)
    torch.cuda.synchronize()
    assert ctx.last_error() == binding.OK and ctx.last_path() == binding.PATH_STREAM
    _check(oracle.fullhead_topk(oracle.bf16_bits(h), oracle.bf16_bits(W), k), ids, lp)
    assert ids[M // 2:].cpu().tolist() == [list(range(k))] * (M - M // 2)


@pytest.mark.parametrize("M", [20, 64])
def test_slab_logits(ctx, M):
    d, r, V = 256, 64, 8 * 1337
    x = synth.make_inputs(M, d, r, V, seed=2)
    buf = torch.full((M * V + 512,), 12345.0, dtype=torch.float32, device=DEV)
    out = ctx.slimspec_head_logits(x["h"].to(DEV), x["A"].to(DEV), x["B"].to(DEV), out_logits=buf[256:256 + M * V].view(M, V))
    torch.cuda.synchronize()
    assert ctx.last_error() == binding.OK
    assert torch.all(buf[:256] == 12345.0) and torch.all(buf[256 + M * V:] == 12345.0)
    b = {n: oracle.bf16_bits(t) for n, t in x.items()}
    ref = torch.from_numpy(oracle.slimspec_logits(b["h"], b["A"], b["B"]))
    assert (out.cpu().double() - ref).abs().max() < 1e-4
