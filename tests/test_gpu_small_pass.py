"""Passes of small fp32 models as one launch of one cluster, against the kernels of one launch per step on the same
weights: logits of every pass, the cache, tokens and counters, where its key tiles (8 keys), slices and rows end."""
import pytest
import torch

from helpers import to_cuda
from synthetic import SHAPES, make_weights

pytestmark = pytest.mark.gpu

SHAPE = SHAPES["tiny"]
# fp32 sums in another order: K <= 768 products a sum, some 30 sums in a row (2^-24 sqrt(768) 30 = 5e-5 of the values' size)
RTOL = 5e-5


@pytest.fixture(scope="module")
def dmtd():
    import paper_2510_11958_b200 as pkg
    pkg.load_library()
    return pkg


@pytest.fixture(scope="module")
def weights():
    return {n: to_cuda(make_weights(s, seed=3, norm_jitter=0.1)) for n, s in _shapes().items()}


def _shapes():
    return {"tiny": SHAPE,
            "wide": SHAPE.with_(n_layers=3, hidden=512, intermediate=1024, vocab=1028),      # two gate-up sets, an odd vocabulary
            "mha": SHAPE.with_(n_layers=2, n_q_heads=8, n_kv_heads=8, vocab=4100)}


def _run(dmtd, name, weights, fused, L_d, tau, B, P, sample):
    eng = dmtd.Dmtd(_shapes()[name], weights[name], L_d=L_d, tau=tau, max_batch=B, max_seq=P + 3 * tau + 2, kv_dtype="f32")
    eng.set_option("fused_pass", fused)
    if sample:
        eng.set_sampling(0.7, 5)
    g = torch.Generator(device="cuda").manual_seed(P)
    eng.prefill(torch.randint(0, SHAPE.vocab, (B, P), generator=g, dtype=torch.int32, device="cuda"))
    forced = torch.randint(0, SHAPE.vocab, (B, 2 * tau), generator=g, dtype=torch.int32, device="cuda")
    n0 = eng.launch_count()
    logits, am = eng.decode_forced(forced)                 # starts inside the first cycle
    launches = eng.launch_count() - n0
    toks = []
    while eng.state()["slot"]:
        toks.append(eng.decode_cycle(1)[2].clone())        # one pass at a time
    rc, n, out = eng.decode_cycle(tau, allow_capacity=True)
    toks.append(out)
    assert eng.device_state() == eng.state()
    shape = _shapes()[name]
    kv = [torch.as_tensor(_View(p, (B, shape.n_kv_heads, P + 3 * tau + 2, 64)), device="cuda")[:, :, :eng.state()["up_len"]].clone()
          for p in eng.kv(shape.n_layers - 1)]
    return logits, am, torch.cat(toks, 1), kv, launches


class _View:
    def __init__(self, ptr, shape):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f4", "data": (int(ptr), False), "version": 2}


@pytest.mark.parametrize("name,L_d,tau,B,P,sample", [
    ("tiny", 2, 3, 1, 1, False),          # no slice but the last has keys
    ("tiny", 2, 3, 1, 8, False),
    ("tiny", 2, 3, 1, 63, True),
    ("tiny", 1, 4, 1, 64, False),         # eight query rows
    ("tiny", 2, 2, 1, 515, False),        # a warp's second tile
    ("tiny", 4, 3, 1, 1100, False),       # no lower layers
    ("tiny", 2, 1, 1, 9, False),
    ("tiny", 2, 2, 3, 40, True),          # six rows; slices that do not use every block
    ("tiny", 2, 2, 4, 77, False),         # eight rows
    ("tiny", 2, 3, 8, 33, False),         # full passes by the other kernels, short ones by the cluster
    ("wide", 1, 3, 2, 50, False),
    ("mha", 1, 4, 1, 130, True),
    ("mha", 1, 2, 2, 21, False),
])
def test_small_pass(dmtd, weights, name, L_d, tau, B, P, sample):
    logits, am, toks, kv, launches = _run(dmtd, name, weights, 1, L_d, tau, B, P, sample)
    ref, ref_am, ref_toks, ref_kv, ref_launches = _run(dmtd, name, weights, 0, L_d, tau, B, P, sample)
    assert launches < ref_launches
    for got, want in [(logits, ref)] + list(zip(kv, ref_kv)):
        assert (got - want).abs().max() <= RTOL * want.abs().max().clamp(min=1.0)
    if sample:
        # a draw goes the other way only where two perturbed logits lie within RTOL of each other: at these seeds none do
        assert torch.equal(am, ref_am) and torch.equal(toks, ref_toks)
        assert (am != ref.argmax(-1)).any()                 # and they are draws
        return
    srt = ref.sort(-1).values
    clear = srt[..., -1] - srt[..., -2] > 1e-3
    assert (am[clear] == ref_am[clear]).all()
    if clear.all():
        assert (toks == ref_toks).all()


def test_same_bits_every_time(dmtd, weights):
    """No buffer is written while a warp may still read it: repeated passes give the same logits, bit for bit."""
    g = torch.Generator(device="cuda").manual_seed(2)
    for B, tau, P in ((1, 3, 90), (1, 4, 500), (2, 4, 40)):
        eng = dmtd.Dmtd(SHAPE, weights["tiny"], L_d=2, tau=tau, max_batch=B, max_seq=P + 5 * tau, kv_dtype="f32")
        prompt = torch.randint(0, SHAPE.vocab, (B, P), generator=g, dtype=torch.int32, device="cuda")
        forced = torch.randint(0, SHAPE.vocab, (B, 4 * tau), generator=g, dtype=torch.int32, device="cuda")
        want = None
        for _ in range(40):
            eng.reset()
            eng.prefill(prompt)
            logits, _ = eng.decode_forced(forced)
            want = logits if want is None else want
            assert torch.equal(logits, want)
