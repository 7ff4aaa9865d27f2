"""The causal attention kernel of prefill chunks (16-bit cache) against the one-warp-per-key-group kernel, which keeps
the query and the probabilities in fp32, through one layer: tile edges, positions before the chunk, groups of 1 to 16
query heads, score distributions sharp enough that the running maximum moves by more than a factor of 2^8."""
import pytest
import torch

from synthetic import ModelShape, make_weights

from helpers import to_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dmtd():
    import paper_2510_11958_b200 as pkg
    pkg.load_library()
    return pkg


@pytest.mark.parametrize("kv", ["f16", "bf16"])
@pytest.mark.parametrize("nq,nkv,B,pos0,R,sharp", [
    (8, 2, 1, 0, 16, 1.0),         # less than one block of positions
    (8, 2, 1, 0, 33, 1.0),         # one position more than a block
    (8, 2, 2, 0, 128, 1.0),        # whole key tiles
    (8, 2, 1, 127, 17, 1.0),       # the chunk begins with the last key of a tile
    (8, 2, 1, 128, 40, 6.0),
    (8, 2, 3, 301, 97, 1.0),
    (8, 2, 1, 0, 600, 12.0),
    (4, 4, 2, 5, 130, 3.0),        # one query head per kv head: 128 positions a block
    (8, 4, 1, 64, 70, 1.0),
    (8, 1, 1, 3, 50, 4.0),
    (16, 1, 2, 130, 24, 1.0),      # 8 positions a block
])
def test_prefill_attention_against_fp32_probabilities(dmtd, kv, nq, nkv, B, pos0, R, sharp):
    shape = ModelShape(n_layers=1, hidden=256, n_q_heads=nq, n_kv_heads=nkv, head_dim=128, intermediate=256, vocab=64)
    w = make_weights(shape, seed=3, norm_jitter=0.1, std=0.05)
    w["layers"][0]["q_norm"] *= sharp
    g = torch.Generator().manual_seed(7)
    before = torch.randn(B, max(pos0, 1), shape.hidden, generator=g).cuda()
    rows = torch.randn(B, R, shape.hidden, generator=g).cuda()
    eng = dmtd.Dmtd(shape, to_cuda(w), L_d=1, tau=1, max_batch=B, max_seq=pos0 + R + 1, kv_dtype=kv)
    outs = []
    for tc in (0, 1):
        eng.set_option("tc_attention", tc)
        for p in range(0, pos0, 15):                        # short chunks: the decode kernels
            eng.step_layers(0, 1, before[:, p:min(p + 15, pos0)].clone(memory_format=torch.contiguous_format), p)
        outs.append(eng.step_layers(0, 1, rows.clone(), pos0))
    torch.cuda.synchronize()
    ref, got = outs[0].double(), outs[1].double()
    # query, probabilities (and, before the chunk, the rows that the decode kernel wrote) rounded to 16 bits once:
    # 2^-8 relative for bf16 on either side of a product, as in the layer tests; fp16 has three bits more
    tol = 4e-3 if kv == "bf16" else 1e-3
    # a sharp softmax turns an error of the score (2^-9 of |q||k| for bf16) into one of the probability
    tol *= max(1.0, sharp)
    assert (got - ref).abs().max() <= tol * max(1.0, ref.abs().max().item())


@pytest.mark.parametrize("kv", ["f16", "bf16"])
@pytest.mark.parametrize("nq,nkv,B,pos0,R,sharp", [
    (4, 2, 1, 0, 300, 1.0),
    (4, 2, 2, 127, 140, 12.0),     # the reference maximum of a row moves by far more than 2^8
    (8, 2, 1, 128, 200, 6.0),
    (8, 1, 1, 3, 129, 12.0),
    (4, 4, 1, 250, 150, 12.0),
])
def test_prefill_attention_rows_alone(dmtd, kv, nq, nkv, B, pos0, R, sharp):
    """The kernel's output without the residual and the MLP (no down projection, an identity for the O projection), row by
    row against the decode kernel, which reads the same rounded Q, K and V in chunks of 15 positions (its own test holds it
    to fp64).  The bound does not grow with the sharpness of the softmax."""
    shape = ModelShape(n_layers=1, hidden=nq * 128, n_q_heads=nq, n_kv_heads=nkv, head_dim=128, intermediate=256, vocab=64)
    w = make_weights(shape, seed=3, norm_jitter=0.1, std=0.05)
    layer = w["layers"][0]
    layer["q_norm"] *= sharp
    layer["down_proj"].zero_()
    layer["o_proj"].copy_(torch.eye(shape.hidden))
    g = torch.Generator().manual_seed(7)
    rows = torch.randn(B, pos0 + R, shape.hidden, generator=g).cuda()
    eng = dmtd.Dmtd(shape, to_cuda(w), L_d=1, tau=1, max_batch=B, max_seq=pos0 + R + 1, kv_dtype=kv)
    def layer_on(p, n):
        return eng.step_layers(0, 1, rows[:, p:p + n].clone(memory_format=torch.contiguous_format), p)

    ref = torch.cat([layer_on(p, min(15, pos0 + R - p)) for p in range(0, pos0 + R, 15)], 1)[:, pos0:]
    got = layer_on(pos0, R)
    ref, got = (x - rows[:, pos0:] for x in (ref, got))
    err = (got - ref).abs().amax(-1) / ref.abs().max()
    # the probabilities are rounded once on either side, against other maxima: 2^-9 (bf16) or 2^-12 of the largest value
    # each; a query element whose fp32 value differs in its last bit may round the other way (a few in a million)
    u = 2.0 ** -9 if kv == "bf16" else 2.0 ** -12
    assert (err <= 2 * u).float().mean() >= 0.99
    assert err.max() <= 2 * u * max(4.0, sharp)
