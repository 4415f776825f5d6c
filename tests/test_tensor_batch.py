"""The tensor-core path for batches (more rows than the streaming kernels take): sizes at the edges of its row blocks, column
tiles, K chunks and K splits, against the fp64 oracle."""
import pytest
import torch

import oracle
from paper_2605_10453_b200 import binding, synth
from parity import check_topk

pytestmark = pytest.mark.gpu

DEV = "cuda:0"

# M, d, r, V, k
SHAPES = [
    (65, 64, 64, 64, 10),              # one K chunk, one column tile, a quarter of it filled
    (96, 512, 72, 8 * 997, 32),        # K no multiple of a chunk; last tile ragged
    (128, 576, 128, 256 * 149, 10),    # nine chunks: uneven K splits; a second tile for one CTA
    (129, 256, 64, 256 * 150, 10),     # CTA pairs, one row in the second CTA
    (255, 200, 96, 8 * 2501, 1),       # d no multiple of a chunk
    (256, 512, 256, 8 * 4001, 31),
    (257, 256, 64, 8 * 1500, 12),      # two row blocks of a pair, one row in the second; code as bf16
    (600, 384, 520, 8 * 600, 32),      # X does not fit shared memory; fewer tiles than pairs
    (130, 516, 68, 8 * 700, 5),        # A's rows are no multiple of 16 bytes: the other down-projection
]


@pytest.fixture(scope="module")
def ctx():
    c = binding.Context(max_M=600, max_d=1024, max_V=40000, max_k=32)
    yield c
    c.close()


def _lp_tol(M):
    # Up to 256 rows the code keeps 17 bits and sums are fp32: 1e-4 as on the streaming path.  Beyond, each element of the code is
    # rounded to bf16: at most 2^-9 of it, uniform, rms 2^-9 / sqrt(3) = 1.1e-3.  A logit is a sum of r products of a normal code
    # and normal weights, its error 1.1e-3 |z| / sqrt(r); |z| / sqrt(r) reaches 1.4 over 257 rows at r = 64, and the
    # largest of 3 million such sums 8 of their standard deviations (products of normals: heavier tails than one normal's 5).
    return 1e-4 if M <= 256 else 8 * 1.1e-3 * 1.4


@pytest.mark.parametrize("M,d,r,V,k", SHAPES)
def test_batch_matches_oracle(ctx, M, d, r, V, k):
    x = synth.make_inputs(M, d, r, V, seed=31)
    g = {n: t.to(DEV) for n, t in x.items()}
    b = {n: oracle.bf16_bits(t) for n, t in x.items()}
    ids, lp = ctx.slimspec_head_topk(g["h"], g["A"], g["B"], k)
    again = ctx.slimspec_head_topk(g["h"], g["A"], g["B"], k)
    logits = ctx.slimspec_head_logits(g["h"], g["A"], g["B"])
    torch.cuda.synchronize()
    assert ctx.last_error() == binding.OK and ctx.last_path() == binding.PATH_TENSOR
    ref = oracle.head_topk(b["h"], b["A"], b["B"], k)
    assert check_topk(ref, ids.cpu().numpy(), lp.cpu().numpy())["max_lp_err"] < _lp_tol(M)
    assert torch.equal(ids, again[0]) and torch.equal(lp, again[1])
    assert abs(logits.cpu().double().numpy() - ref["logits"]).max() < _lp_tol(M)


@pytest.mark.parametrize("M", [100, 300])
def test_batch_equal_logits(ctx, M):
    """Zero rows: every logit is the same, no bound keeps the lists short, and the lowest ids win.  The calls before leave
    larger bounds behind; they must not count."""
    d, V, k = 264, 8 * 1201, 16
    W = synth.make_W(d, V, 3).to(DEV)
    h = synth.make_h(M, d, 3)
    ctx.fullhead_topk(h.to(DEV), W, k)
    h[M // 2:] = 0
    ids, lp = ctx.fullhead_topk(h.to(DEV), W, k)
    torch.cuda.synchronize()
    assert ctx.last_error() == binding.OK and ctx.last_path() == binding.PATH_TENSOR
    assert check_topk(oracle.fullhead_topk(oracle.bf16_bits(h), oracle.bf16_bits(W.cpu()), k), ids.cpu().numpy(), lp.cpu().numpy())["max_lp_err"] < 1e-4
    assert ids[M // 2:].cpu().tolist() == [list(range(k))] * (M - M // 2)


@pytest.mark.parametrize("M,d,r,V,k,path", [
    (33, 512, 328, 8 * 1001, 10, binding.PATH_TENSOR),       # 33 to 64 rows: from a rank of 320 on
    (64, 1024, 320, 256 * 150, 20, binding.PATH_TENSOR),
    (17, 4104, 528, 8 * 3000, 10, binding.PATH_STREAM),      # slab kernel behind the tensor cores' down-projection
    (3, 4104, 1040, 8 * 1777, 5, binding.PATH_STREAM),
])
def test_few_rows_matches_oracle(M, d, r, V, k, path):
    ctx = binding.Context(max_M=M, max_d=d, max_V=V, max_k=k)
    x = synth.make_inputs(M, d, r, V, seed=37)
    g = {n: t.to(DEV) for n, t in x.items()}
    b = {n: oracle.bf16_bits(t) for n, t in x.items()}
    ids, lp = ctx.slimspec_head_topk(g["h"], g["A"], g["B"], k)
    torch.cuda.synchronize()
    assert ctx.last_error() == binding.OK and ctx.last_path() == path
    ctx.close()
    assert check_topk(oracle.head_topk(b["h"], b["A"], b["B"], k), ids.cpu().numpy(), lp.cpu().numpy())["max_lp_err"] < 1e-4


@pytest.mark.parametrize("M,d,r,V", [(4, 4104, 1024, 8 * 1601), (3, 512, 8192, 8 * 640), (2, 4096, 2048, 8 * 1601), (1, 2056, 2048, 8 * 1601)])
def test_few_rows_large_A_keep_the_whole_code(M, d, r, V):
    """One to four rows over a large A: the slab kernel, with the code in three parts, which is all of fp32."""
    k = 10
    ctx = binding.Context(max_M=M, max_d=max(d, r), max_V=V, max_k=k)
    x = synth.make_inputs(M, d, r, V, seed=41)
    g = {n: t.to(DEV) for n, t in x.items()}
    b = {n: oracle.bf16_bits(t) for n, t in x.items()}
    ids, lp = ctx.slimspec_head_topk(g["h"], g["A"], g["B"], k)
    torch.cuda.synchronize()
    assert ctx.last_error() == binding.OK and ctx.last_path() == binding.PATH_STREAM
    ctx.close()
    # fp32 sums of d and r products: 2^-24 sqrt(8192) = 5e-6 of a logit of at most 6; a code of 17 bits would show 1e-4 or less too,
    # so the bound is what fp32 sums give and no more
    assert check_topk(oracle.head_topk(b["h"], b["A"], b["B"], k), ids.cpu().numpy(), lp.cpu().numpy())["max_lp_err"] < 4e-5
