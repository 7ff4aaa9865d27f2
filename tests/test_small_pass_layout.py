"""Shared memory of the cluster pass for small fp32 models, as the library's own host code lays it out: buffers that are in use
at the same time lie apart; where the warps' shares of a matrix lie; for which models the form is chosen.  Runs without a GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROBE = r"""
#include <cstdio>
#include <cstdlib>
#include "small_pass.cuh"
int main(int argc, char **argv) {
  int a[10];
  if (argc == 11) {
    for (int i = 0; i < 10; ++i) a[i] = atoi(argv[i + 1]);
    printf("%f\n", dmtd::small_pass_gain(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9] != 0));
    return 0;
  }
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


# cycles as measured, us: one launch, captured launches per step
MEASURED = [
    # H, I, nq, nkv, vocab, layers, L_d, B, tau, the full pass by the cluster, times
    (256, 768, 4, 2, 1024, 4, 2, 1, 3, 1, 97, 163), (256, 768, 4, 2, 1024, 4, 4, 8, 1, 1, 95, 118), (256, 768, 4, 2, 1024, 12, 6, 2, 3, 0, 404, 457),
    (256, 768, 4, 2, 16384, 4, 2, 1, 3, 1, 145, 182), (256, 768, 4, 2, 65536, 4, 2, 1, 3, 1, 306, 241), (256, 768, 4, 2, 151936, 4, 4, 1, 1, 1, 200, 145),
    (256, 768, 4, 2, 151936, 4, 2, 2, 3, 1, 913, 412), (256, 768, 4, 2, 32768, 4, 4, 4, 1, 1, 116, 103), (256, 768, 4, 2, 32768, 4, 4, 8, 1, 1, 179, 151),
    (256, 768, 4, 2, 32768, 1, 1, 1, 1, 1, 52, 44), (256, 768, 4, 2, 8192, 1, 1, 1, 1, 1, 27, 34),
    (512, 1536, 8, 4, 1024, 4, 2, 1, 3, 1, 162, 192), (512, 1536, 8, 4, 1024, 4, 2, 2, 3, 0, 251, 233), (512, 1536, 8, 4, 32768, 4, 2, 1, 3, 1, 319, 301),
    (512, 512, 4, 2, 1024, 4, 2, 2, 3, 0, 172, 184), (512, 2048, 8, 8, 1024, 4, 2, 2, 3, 0, 304, 274),
    (1024, 3072, 16, 8, 1024, 4, 4, 1, 1, 1, 166, 175), (1024, 3072, 16, 8, 32768, 4, 4, 1, 1, 1, 246, 235), (1024, 1024, 4, 2, 1024, 4, 2, 2, 3, 0, 278, 243),
]


@pytest.mark.parametrize("case", MEASURED, ids=lambda c: "-".join(map(str, c[:10])))
def test_chosen_where_it_is_the_faster_form(probe, case):
    gain = float(subprocess.run([str(probe)] + [str(x) for x in case[:10]], check=True, capture_output=True, text=True).stdout)
    assert (gain > 0) == (case[10] < case[11]), gain
