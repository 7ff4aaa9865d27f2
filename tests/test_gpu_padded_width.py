"""bf16 models whose intermediate size is no multiple of 64 on the tcgen05 GEMM: gate+up and down are filled up to whole k
blocks.  Against the mma.sync kernels on the same context, at row counts where the GEMM's forms change."""
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


@pytest.mark.parametrize("intermediate", [32, 1824, 19552])       # less than a block; half a block left; more row tiles than SM pairs
@pytest.mark.parametrize("B,R", [(1, 1), (3, 2), (8, 16), (3, 43), (2, 450)])   # 1, 6, 128, 129 and 900 rows
def test_padded_intermediate(dmtd, intermediate, B, R):
    shape = SHAPES["mid"].with_(n_layers=2, intermediate=intermediate, vocab=1000)
    w = to_cuda(make_weights(shape, seed=4, norm_jitter=0.1))
    eng = dmtd.Dmtd(shape, w, L_d=1, tau=1, max_batch=B, max_seq=R + 8, kv_dtype="f32")
    g = torch.Generator(device="cuda").manual_seed(intermediate)
    x = torch.randn(B, R, shape.hidden, generator=g, device="cuda")
    out = []
    for tc in (1, 0):
        eng.set_option("tcgen05_gemm", tc)
        junk = torch.full((B, R, shape.hidden), 3e4, device="cuda")
        eng.step_layers(0, 2, junk, 0)                       # what the workspace held before must not matter
        eng.reset()
        h = x.clone()
        eng.step_layers(0, 2, h, 0)
        out.append(h)
    # both multiply the same hi and lo parts (2^-17 each), fp32 sums in another order: 2^-24 sqrt(K) per sum, ten in a row
    err = (out[0] - out[1]).norm() / out[1].norm()
    assert err < 1e-5
