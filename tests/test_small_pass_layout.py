"""Shared memory of the cluster pass for small fp32 models, as the library's own host code lays it out: buffers that are in use
at the same time lie apart; and where the warps' shares of a matrix lie.  Runs without a GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROBE = r"""
#include <cstdio>
#include <cstdlib>
#include "small_pass.cuh"
int main(int argc, char **argv) {
  int a[7];
  if (argc == 4) {
    dmtd::SmallParams P{};
    P.H = atoi(argv[1]); P.vocab = atoi(argv[2]);
    const dmtd::SmallWalk w = dmtd::sp_walk(P, dmtd::SP_HEAD, atoi(argv[3]));
    printf("%zu %d\n", (size_t)w.first, w.batches);
    return 0;
  }
  for (int i = 0; i < 7; ++i) a[i] = atoi(argv[i + 1]);
  const dmtd::SmallMap m = dmtd::small_pass_map(a[0], a[1], a[2], a[3], a[4], a[5], a[6]);
  printf("%d %d %d %d %d %d %d\n", m.xs, m.qkv, m.merged, m.wide, m.part_o, m.total, dmtd::SP_WARPS * dmtd::SP_MAX_ROWS * dmtd::SP_D);
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("probe")
    src, exe = d / "probe.cu", d / "probe"
    src.write_text(PROBE)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O0", "-I",
                    os.path.join(ROOT, "paper_2510_11958_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    return exe


@pytest.mark.parametrize("H,I,nq,nkv,L,B,R", [(256, 768, 4, 2, 4, 1, 1), (256, 768, 4, 2, 4, 1, 4), (512, 256, 16, 8, 3, 1, 2),
                                              (256, 256, 8, 8, 2, 2, 2), (256, 768, 4, 2, 4, 8, 1)])
def test_buffers_in_use_at_once_lie_apart(probe, H, I, nq, nkv, L, B, R):
    xs, qkv, merged, wide, part_o, total, warps_out = map(int, subprocess.run(
        [str(probe)] + [str(x) for x in (H, I, nq, nkv, L, B, R)], check=True, capture_output=True, text=True).stdout.split())
    M = B * R
    areas = {"residual": (xs, M * H), "merged": (merged, M * nq * 64), "warps' outputs": (wide, warps_out), "slices": (part_o, M * nq * 64)}
    spans = sorted((a, a + n, name) for name, (a, n) in areas.items())
    for (_, end, one), (start, _, other) in zip(spans, spans[1:]):
        assert end <= start, (one, other)
    # merged rows may take the place of the projection's rows, which no warp reads any more, but not reach past them
    assert not (qkv <= merged < wide) or merged + M * nq * 64 <= qkv + M * (nq + 2 * nkv) * 64
    assert spans[-1][1] <= total


@pytest.mark.parametrize("H,vocab", [(256, 1024), (256, 1028), (1024, 1 << 20), (1024, (1 << 21) + 4)])
def test_shares_of_the_head(probe, H, vocab):
    """Four-row batches of 128 warps, one share after the other, also past 4 GiB."""
    at = 0
    for share in range(128):
        first, batches = map(int, subprocess.run([str(probe), str(H), str(vocab), str(share)], check=True, capture_output=True,
                                                 text=True).stdout.split())
        assert batches == 0 or first == at
        at += batches * 4 * H * 4
    assert at == vocab * H * 4
