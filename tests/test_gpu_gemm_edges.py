"""Projections on the tcgen05 GEMM at the sizes where its tiles, row counts and work shares end: the scoring pass
(its LM head takes all positions in one GEMM) and teacher-forced decoding against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from synthetic import SHAPES, make_prompts, make_weights

from helpers import check_logits, gpu_forced, oracle_forced, to_cuda

pytestmark = pytest.mark.gpu

# every K a multiple of 64, so that the tcgen05 GEMM runs; a vocabulary that no 4-value load divides
SHAPE = SHAPES["mid"].with_(n_layers=4, intermediate=1856, vocab=5001)


@pytest.fixture(scope="module")
def dmtd():
    import paper_2510_11958_b200 as pkg
    pkg.load_library()
    return pkg


@pytest.mark.parametrize("B,P,n", [
    (1, 1, 1),              # a single row
    (1, 3, 6),              # 4 rows: fewer than the mma.sync kernels' limit
    (2, 7, 71),             # rows of two sequences, in one segment each
    (1, 6, 133),            # 128 rows in the head, 133 in the layers: both forms of a column tile
    (1, 5, 133),            # 129 rows in the head
    (1, 2, 257),            # two column tiles
    (3, 40, 400),           # several chunks of the workspace, four column tiles each
    (70, 3, 17),            # 14 and 1 positions of two chunks: fewer than sequences, position by position
])
def test_scoring_pass(dmtd, B, P, n):
    w = make_weights(SHAPE, seed=0, norm_jitter=0.1)
    tokens = make_prompts(SHAPE.vocab, B, n, seed=5).numpy()
    eng = dmtd.Dmtd(SHAPE, to_cuda(w), L_d=2, tau=3, max_batch=B, max_seq=n + 2, kv_dtype="f32")
    got = eng.masked_forward(torch.from_numpy(tokens).cuda(), P).double().cpu().numpy()
    for b in range(B):
        ref = oracle.masked_parallel_forward(SHAPE, w, 2, 3, tokens[b], P)
        # fp32 cache and sums, bf16 hi + lo activations (2^-17): the bound of the other fp32-cache tests
        assert np.abs(got[b] - ref).max() < 1e-3


@pytest.mark.parametrize("B,tau", [(1, 1), (1, 3), (3, 1), (4, 1), (5, 3), (17, 4), (43, 3)])
def test_decode_rows(dmtd, B, tau):
    """1 to 129 rows a pass on the per-step kernels."""
    w = make_weights(SHAPE, seed=0, norm_jitter=0.1)
    prompts = make_prompts(SHAPE.vocab, B, 9, seed=1).numpy()
    forced = make_prompts(SHAPE.vocab, B, 2 * tau + 2, seed=2).numpy()
    ref_logits, ref_am, o = oracle_forced(SHAPE, w, 2, tau, prompts, forced)
    eng = dmtd.Dmtd(SHAPE, to_cuda(w), L_d=2, tau=tau, max_batch=B, max_seq=9 + forced.shape[1] + 1, kv_dtype="f32")
    eng.set_option("fused_pass", 0)
    got_logits, got_am = gpu_forced(eng, prompts, forced)
    err, _ = check_logits(got_logits, ref_logits, got_am, ref_am)
    assert err < 1e-3
    assert eng.device_state() == o.state()


@pytest.mark.parametrize("intermediate", [
    9472,       # 74 pairs of row tiles of gate+up: all dealt out whole on 148 SMs
    9536,       # one pair more, half of it padding
    9728,       # two pairs more
])
@pytest.mark.parametrize("n", [90, 129, 300])
def test_gated_epilogue(dmtd, intermediate, n):
    """Gate+up wide enough for whole tiles: below 129 rows a pass of its own gates, above the epilogue does."""
    shape = SHAPE.with_(n_layers=2, hidden=256, intermediate=intermediate, vocab=600)
    w = make_weights(shape, seed=4, norm_jitter=0.1)
    tokens = make_prompts(shape.vocab, 1, n, seed=6).numpy()
    ref = oracle.masked_parallel_forward(shape, w, 1, 2, tokens[0], 5)
    eng = dmtd.Dmtd(shape, to_cuda(w), L_d=1, tau=2, max_batch=1, max_seq=n + 2, kv_dtype="f32")
    got = eng.masked_forward(torch.from_numpy(tokens).cuda(), 5).double().cpu().numpy()
    assert np.abs(got[0] - ref).max() < 1e-3


@pytest.mark.parametrize("head_dim,B,tau,P", [
    (64, 1, 1, 1),          # one row
    (64, 4, 1, 130),        # full groups of 4 rows, key slices that end inside the new rows
    (64, 3, 5, 61),         # 15 rows in the lower layers, 3 in the upper ones
    (64, 16, 1, 9),         # the most rows
    (64, 17, 1, 9),         # one more: the separate kernels
    (64, 1, 15, 9),         # the most new positions of a sequence
    (64, 1, 16, 9),         # one more: step a3 as a launch of its own
    (128, 5, 3, 33),
])
def test_f32_decode_rows(dmtd, head_dim, B, tau, P):
    """fp32 weights: projections together with the step in front of them, and the separate kernels past their limits."""
    shape = SHAPES["tiny"].with_(head_dim=head_dim, hidden=260, intermediate=776, vocab=1003, n_layers=4)
    w = make_weights(shape, seed=0, norm_jitter=0.1)
    prompts = make_prompts(shape.vocab, B, P, seed=1).numpy()
    forced = make_prompts(shape.vocab, B, 2 * tau + 2, seed=2).numpy()
    ref_logits, ref_am, o = oracle_forced(shape, w, 2, tau, prompts, forced)
    eng = dmtd.Dmtd(shape, to_cuda(w), L_d=2, tau=tau, max_batch=B, max_seq=P + forced.shape[1] + 1, kv_dtype="f32")
    got_logits, got_am = gpu_forced(eng, prompts, forced)
    err, _ = check_logits(got_logits, ref_logits, got_am, ref_am)
    assert err < 1e-3       # as above; fp32 sums of fp32 products
    assert eng.device_state() == o.state()


@pytest.mark.parametrize("B", [1, 3, 5, 33])
def test_rows_from_unmerged_slices(dmtd, B):
    """Captured passes launch the key slices of the whole cache: more than the O projection's activation blocks merge
    on the way, so its rows come from a merge of their own (1 to 66 rows a pass)."""
    shape = SHAPE.with_(n_layers=2, hidden=256, n_q_heads=16, n_kv_heads=4, head_dim=64)
    w = make_weights(shape, seed=0, norm_jitter=0.1)
    prompts = make_prompts(shape.vocab, B, 9, seed=1).numpy()
    eng = dmtd.Dmtd(shape, to_cuda(w), L_d=1, tau=2, max_batch=B, max_seq=41 * 64, kv_dtype="f32")
    eng.set_option("fused_pass", 0)
    tokens = [eng.prefill(torch.from_numpy(prompts).cuda())[0][:, None]]
    for _ in range(3):
        rc, n, out = eng.decode_cycle(2)
        tokens.append(out[:, :n].clone())
    forced = torch.cat(tokens, 1).cpu().numpy()
    ref_logits, ref_am, _ = oracle_forced(shape, w, 1, 2, prompts, forced)
    srt = np.sort(ref_logits, -1)
    clear = srt[..., -1] - srt[..., -2] > 2e-3       # logits within 1e-3, as above: picks may differ below twice that
    assert clear.mean() > 0.8
    assert (forced.T == ref_am)[clear].all()


@pytest.mark.parametrize("n", [100, 128, 144, 208, 512])
def test_stage_counts(dmtd, n):
    """Every pipeline depth, with the prefill attention (16-bit cache) in front of the O projection: both hold tensor memory."""
    w = to_cuda(make_weights(SHAPE, seed=0, norm_jitter=0.1))
    prompt = torch.from_numpy(make_prompts(SHAPE.vocab, 1, n, seed=5).numpy()).cuda()
    eng = dmtd.Dmtd(SHAPE, w, L_d=2, tau=3, max_batch=1, max_seq=n + 2, kv_dtype="f16")
    logits = []
    for stages in (0, 2, 3, 4, 5, 6):
        eng.reset()
        eng.set_option("tcgen05_gemm_stages", stages)
        logits.append(eng.prefill(prompt, want_logits=True)[1].double())
        eng.device_state()                                  # raises if a wait gave up
    # the same products; the order of the reductions moves the last bit of single values of the fp16 cache (2^-11)
    for got in logits[1:]:
        assert (got - logits[0]).norm() <= 2 ** -11 * logits[0].norm()


@pytest.mark.parametrize("model", ["f32", "bf16"])
@pytest.mark.parametrize("B,R", [(1, 1), (2, 2), (3, 2), (2, 20)])
def test_step_layers_rows_off_a_16_byte_boundary(dmtd, model, B, R):
    shape = SHAPES["tiny"] if model == "f32" else SHAPE.with_(n_layers=2)
    eng = dmtd.Dmtd(shape, to_cuda(make_weights(shape, seed=0, norm_jitter=0.1)), L_d=1, tau=1, max_batch=B, max_seq=R + 1, kv_dtype="f32")
    rows = torch.randn(B, R, shape.hidden, generator=torch.Generator().manual_seed(3)).cuda()
    ref = eng.step_layers(0, 2, rows.clone(), 0)
    for off in (1, 2, 3):
        buf = torch.full((rows.numel() + 8,), 7.0, device="cuda")
        view = buf[off:off + rows.numel()].view(rows.shape)
        view.copy_(rows)
        got = eng.step_layers(0, 2, view, 0)
        # the same kernels on the same values: fp32 reductions in another order at most
        assert (got - ref).abs().max() <= 1e-5 * max(1.0, ref.abs().max().item())
        assert (buf[:off] == 7).all() and (buf[off + rows.numel():] == 7).all()


# projections of this size keep 74 block pairs busy with uncut tiles from 897 rows on
WIDE = SHAPE.with_(n_layers=2, hidden=2560, n_q_heads=32, n_kv_heads=8, intermediate=9728, vocab=20000)


@pytest.fixture(scope="module")
def wide_weights():
    return make_weights(WIDE, seed=0, device="cuda", norm_jitter=0.1)


@pytest.mark.parametrize("B,P,kv", [
    (1, 897, "f16"),
    (2, 512, "f16"),
    (3, 300, "f32"),        # 900 rows
    (8, 256, "bf16"),       # two chunks
])
def test_large_prefill_repeats(dmtd, wide_weights, B, P, kv):
    """Large chunks give the same bits again, cache and logits."""
    prompt = torch.from_numpy(make_prompts(WIDE.vocab, B, P, seed=5).numpy()).cuda()
    eng = dmtd.Dmtd(WIDE, wide_weights, L_d=1, tau=3, max_batch=B, max_seq=P + 1, kv_dtype=kv)
    first = None
    for _ in range(4):
        eng.reset()
        logits = eng.prefill(prompt, want_logits=True)[1]
        if first is None:
            first = logits.clone()
        assert torch.equal(logits, first)


@pytest.mark.parametrize("layers", [1, 2])
@pytest.mark.parametrize("R", [897, 950, 1000])
def test_large_chunk_against_small_ones(dmtd, wide_weights, layers, R):
    eng = dmtd.Dmtd(WIDE, wide_weights, L_d=1, tau=1, max_batch=1, max_seq=R + 1, kv_dtype="f32")
    rows = torch.randn(1, R, WIDE.hidden, generator=torch.Generator().manual_seed(3)).cuda()
    got = eng.step_layers(0, layers, rows.clone(), 0)
    ref = torch.cat([eng.step_layers(0, layers, rows[:, p:p + 200].clone(), p) for p in range(0, R, 200)], 1)
    # sums of at most 9728 products in another order, activations within 2^-17 on both sides
    assert (got - ref).abs().max() <= 1e-4 * max(1.0, ref.abs().max().item())


@pytest.mark.parametrize("intermediate", [
    6400,       # gate+up in 50 row-tile pairs: none dealt out whole, its tiles in two parts at most
    9472,       # 74: all dealt out whole
])
def test_large_chunk_repeats_at_other_widths(dmtd, intermediate):
    shape = WIDE.with_(n_layers=1, intermediate=intermediate, vocab=600)
    eng = dmtd.Dmtd(shape, make_weights(shape, seed=0, device="cuda", norm_jitter=0.1), L_d=1, tau=1, max_batch=1, max_seq=951, kv_dtype="f16")
    rows = torch.randn(1, 950, shape.hidden, generator=torch.Generator().manual_seed(3)).cuda()
    first = eng.step_layers(0, 1, rows.clone(), 0)
    for _ in range(3):
        assert torch.equal(eng.step_layers(0, 1, rows.clone(), 0), first)
    ref = torch.cat([eng.step_layers(0, 1, rows[:, p:p + 200].clone(), p) for p in range(0, 950, 200)], 1)
    # as above; the fp16 cache rounds K and V of sums in another order (2^-11), the query and the probabilities too
    assert (first - ref).abs().max() <= 2e-3 * max(1.0, ref.abs().max().item())


@pytest.mark.parametrize("P,B,tau", [
    (500, 1, 4),        # 4 rows x 4 heads x 64 x 8 slices: the most that the O projection merges itself
    (513, 1, 4),        # one slice more
    (130, 11, 1),       # 11 rows, 3 slices
])
def test_f32_slices_merged_apart(dmtd, P, B, tau):
    shape = SHAPES["tiny"].with_(n_layers=2, vocab=500)
    w = make_weights(shape, seed=0, norm_jitter=0.1)
    prompts = make_prompts(shape.vocab, B, P, seed=1).numpy()
    forced = make_prompts(shape.vocab, B, tau + 2, seed=2).numpy()
    ref_logits, ref_am, o = oracle_forced(shape, w, 1, tau, prompts, forced)
    eng = dmtd.Dmtd(shape, to_cuda(w), L_d=1, tau=tau, max_batch=B, max_seq=P + forced.shape[1] + 1, kv_dtype="f32")
    got_logits, got_am = gpu_forced(eng, prompts, forced)
    err, _ = check_logits(got_logits, ref_logits, got_am, ref_am)
    assert err < 1e-3       # fp32 sums of fp32 products, as above
