"""Decode attention by clusters (pieces of an item merged through distributed shared memory, straight into the O projection's
blocks) through one layer, against separate kernels for the QK-norm, the pieces and their merge: empty pieces, one key, tile
and unit edges, one to eight blocks to an item, new rows in a piece of their own."""
import pytest
import torch

from helpers import to_cuda
from synthetic import SHAPES, make_weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dmtd():
    import paper_2510_11958_b200 as pkg
    pkg.load_library()
    return pkg


@pytest.mark.parametrize("kv", ["f16", "bf16"])
@pytest.mark.parametrize("nq,nkv,B,R,pos0", [
    (8, 2, 1, 1, 0),             # one key
    (8, 2, 1, 3, 63),            # the new rows lie in two units
    (8, 2, 2, 4, 64),            # ... in a unit of their own, 16 query rows
    (8, 2, 3, 15, 130),          # four row blocks
    (8, 2, 16, 1, 320),          # 32 items: fewer than eight blocks each; five units, empty pieces
    (8, 8, 9, 1, 1000),          # one query head per kv head
    (16, 1, 5, 2, 511),          # one position to a row block
    (8, 2, 70, 1, 200),          # 140 items
    (8, 2, 148, 1, 70),          # 296 items: a block each
    (8, 2, 150, 1, 70),          # 300 items: a few more than resident blocks
    (8, 2, 250, 1, 70),          # 500 items: a block each
    (8, 2, 300, 1, 70),          # 600 items: a few more than two waves
])
def test_layer(dmtd, kv, nq, nkv, B, R, pos0):
    shape = SHAPES["mid"].with_(n_layers=1, hidden=256, intermediate=256, n_q_heads=nq, n_kv_heads=nkv, vocab=64)
    w = to_cuda(make_weights(shape, seed=3, norm_jitter=0.1, std=0.05))
    g = torch.Generator().manual_seed(7)
    before = torch.randn(B, max(pos0, 1), shape.hidden, generator=g).cuda()
    rows = torch.randn(B, R, shape.hidden, generator=g).cuda()
    eng = dmtd.Dmtd(shape, w, L_d=1, tau=1, max_batch=B, max_seq=pos0 + R + 1, kv_dtype=kv)
    step = max(1, min(256, 1024 // B))
    for p in range(0, pos0, step):
        eng.step_layers(0, 1, before[:, p:min(p + step, pos0)].clone(memory_format=torch.contiguous_format), p)
    out = []
    for fused in (1, 0):
        eng.set_option("fused_qk_rope", fused)
        n0 = eng.launch_count()
        out.append(eng.step_layers(0, 1, rows.clone(), pos0).double())
        out.append(eng.launch_count() - n0)
    assert out[1] < out[3]
    # query and probabilities rounded to 16 bits on both sides, the latter against other maxima: 2^-9 (bf16) or 2^-12 each
    tol = 4e-3 if kv == "bf16" else 5e-4
    assert (out[0] - out[2]).abs().max() <= tol * max(1.0, out[2].abs().max().item())


def test_more_items_than_resident_blocks(dmtd):
    """A layer takes a block to an item, and no launch that merges, up to one wave, and for short items in a well filled
    second one; otherwise equal shares and a merge, which are faster there."""
    shape = SHAPES["mid"].with_(n_layers=1, hidden=256, intermediate=256, vocab=64)
    eng = dmtd.Dmtd(shape, to_cuda(make_weights(shape, seed=3)), L_d=1, tau=1, max_batch=600, max_seq=700, kv_dtype="f16")
    wave = 2 * torch.cuda.get_device_properties(0).multi_processor_count

    def launches(items, pos0):
        B = items // shape.n_kv_heads
        x = torch.zeros(B, 1, shape.hidden, device="cuda")
        n0 = eng.launch_count()
        eng.step_layers(0, 1, x, pos0)
        # more than 128 rows: gate+up and down run differently; the number of launches is the same up to there and from there
        return eng.launch_count() - n0

    one_launch = launches(wave, 600)
    assert launches(wave * 9 // 5, 200) == one_launch
    for items, pos0 in [(wave + 60, 200), (wave * 9 // 5, 600), (wave * 5 // 2, 200), (wave * 4, 64)]:
        assert launches(items, pos0) == one_launch + 1


def test_few_long_items(dmtd):
    """Where clusters leave places free, long items take equal shares and a merge; the passes of a context that grows past the
    line are captured for either side, and their tokens are those of passes launched one by one."""
    shape = SHAPES["mid"].with_(n_layers=2, hidden=256, intermediate=256, vocab=512)
    w = to_cuda(make_weights(shape, seed=3, norm_jitter=0.1))
    places = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    items, ranks = shape.n_kv_heads, 8
    # the first number of 64-key units that is more than 18 of them longer in a block of a cluster than in an equal share
    line = 18 * ranks * places // (places - items * ranks) + 1
    keys = (line - 1) * 64                                    # the last context of fewer units
    toks = []
    for graph in (1, 0):
        eng = dmtd.Dmtd(shape, w, L_d=1, tau=3, max_batch=1, max_seq=keys + 60, kv_dtype="f16")
        eng.set_option("fused_pass", 0)
        eng.set_option("cuda_graph", graph)
        g = torch.Generator(device="cuda").manual_seed(5)
        eng.prefill(torch.randint(0, shape.vocab, (1, keys - 20), generator=g, dtype=torch.int32, device="cuda"))
        while eng.state()["slot"]:
            eng.decode_cycle(3)
        counts, out = [], []
        for _ in range(12):
            before, n0 = eng.state()["n_known"], eng.launch_count()
            out.append(eng.decode_cycle(3)[2].clone())
            counts.append((before, eng.launch_count() - n0))
        assert eng.device_state() == eng.state()
        short = {n for p, n in counts if p + 2 <= keys}
        far = {n for p, n in counts if p > keys}
        # a merge in each of the cycle's four layers
        assert len(short) == 1 and far == {short.pop() + 4}
        toks.append(torch.cat(out, 1))
    assert torch.equal(*toks)
