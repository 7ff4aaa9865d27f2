"""Projections of fp32 models with more rows than the fused decode kernels take, at the edges of their tiles (16, 32 and 64
rows and weight rows, pieces of 32, 128 and 256 values), through one layer against the oracle."""
import pytest
import torch

import oracle
from synthetic import SHAPES, make_weights

from helpers import to_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dmtd():
    import paper_2510_11958_b200 as pkg
    pkg.load_library()
    return pkg


@pytest.mark.parametrize("hidden,intermediate,nq,nkv", [
    (256, 768, 4, 2),
    (100, 36, 1, 1),           # less than a piece, and no size a multiple of a tile
    (260, 1028, 3, 1),
])
@pytest.mark.parametrize("B,R", [(1, 17), (2, 32), (5, 13), (1, 161), (2, 300)])       # 17, 64, 65, 161 and 600 rows
def test_layer_rows(dmtd, hidden, intermediate, nq, nkv, B, R):
    shape = SHAPES["tiny"].with_(n_layers=1, hidden=hidden, intermediate=intermediate, n_q_heads=nq, n_kv_heads=nkv, vocab=64)
    w = make_weights(shape, seed=3, norm_jitter=0.1)
    h = torch.randn(B, R, hidden, generator=torch.Generator().manual_seed(5)) * 0.5
    ref = torch.from_numpy(oracle.Oracle(shape, w, L_d=1, tau=1, max_batch=B, max_seq=R + 1).step_layers(0, 1, h.double().numpy(), 0))
    eng = dmtd.Dmtd(shape, to_cuda(w), L_d=1, tau=1, max_batch=B, max_seq=R + 1)
    got = eng.step_layers(0, 1, h.cuda(), 0).double().cpu()
    # some ten fp32 sums in a row, 2^-24 sqrt(1028) of their terms' size each
    assert (got - ref).abs().max() <= 2e-5 * max(1.0, ref.abs().max().item())


def test_largest_tiles(dmtd):
    """Enough rows for the widest tiles, against the same rows in chunks that take the narrower ones."""
    shape = SHAPES["tiny"].with_(n_layers=1, hidden=1024, intermediate=3076, n_q_heads=16, n_kv_heads=8, vocab=64)
    w = to_cuda(make_weights(shape, seed=3, norm_jitter=0.1))
    eng = dmtd.Dmtd(shape, w, L_d=1, tau=1, max_batch=64, max_seq=16)
    h = torch.randn(64, 15, 1024, generator=torch.Generator().manual_seed(5)).cuda()
    got = eng.step_layers(0, 1, h.clone(), 0)
    ref = torch.cat([eng.step_layers(0, 1, h[i:i + 4].clone(), 0) for i in range(0, 64, 4)])
    assert (got - ref).abs().max() <= 2e-5 * ref.abs().max()
