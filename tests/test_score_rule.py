"""The rules of the score kernels, compiled for the host as they stand in the source, against measured times: how the general kernel's key blocks are split
over clusters, where two of its CTAs share an SM, and which scores take two kernels instead."""
import pathlib
import subprocess

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2409_12490_b200" / "csrc"

HARNESS = """
#include <cstddef>
#include <initializer_list>
#include <cstdio>
struct Dims { int B, Hkv, g, n1, n2, d, es; };
%s
int main() {
  Dims m{1};
  int U;
  while (std::scanf("%%d %%d %%d %%d %%d %%d", &m.Hkv, &m.g, &m.n1, &m.n2, &m.d, &m.es) == 6) {
    U = m.g %% 4 == 0 ? 4 : (m.g %% 2 == 0 ? 2 : 1);
    int nb = 0;
    const int CL = cluster_of(m, U, &nb);
    const size_t smem = 12 * 4 * size_t(U) * nb;
    std::printf("%%d %%d %%d\\n", CL, nb, int(two_per_sm(m, (long long)m.Hkv * (m.g / U) * m.n1 * CL, smem)));
  }
}
"""

# KV heads, group, segments, key blocks, channels, bytes; us with as few CTAs per row group as fit an SM (512 threads) and with twice as many
SPLIT = [
    (8, 4, 5, 600, 128, 2, 25.6, 16.4), (2, 4, 4, 800, 128, 2, 29.5, 19.0), (8, 4, 2, 1024, 128, 4, 71.5, 29.9), (8, 4, 7, 875, 64, 2, 27.3, 16.6),
    (2, 4, 15, 938, 64, 2, 29.3, 17.2), (8, 4, 15, 938, 128, 2, 33.2, 37.0), (8, 4, 15, 938, 64, 2, 29.4, 30.8), (8, 4, 34, 576, 128, 2, 46.0, 52.1),
    (8, 4, 34, 576, 128, 4, 65.8, 71.4), (8, 4, 34, 576, 64, 2, 40.5, 42.9), (8, 4, 34, 1108, 128, 2, 101.3, 107.5), (8, 4, 34, 1108, 64, 4, 91.7, 94.1),
    (8, 2, 30, 1132, 64, 2, 52.1, 48.1), (8, 2, 30, 1132, 64, 4, 59.4, 52.4), (12, 1, 25, 2268, 64, 2, 119.4, 95.2), (12, 1, 25, 2268, 128, 4, 280.1, 229.2)]
# the same; us with one CTA of 512 threads per SM and with two of 256
SHARED = [
    (8, 4, 34, 432, 128, 4, 51.9, 51.3), (8, 4, 34, 464, 128, 4, 55.1, 54.2), (8, 4, 32, 480, 128, 4, 55.4, 71.2), (8, 4, 34, 544, 128, 4, 64.2, 80.2),
    (8, 2, 30, 892, 128, 4, 85.9, 80.0), (8, 2, 30, 988, 128, 4, 93.0, 126.9), (12, 1, 25, 1884, 128, 4, 235.5, 223.5), (12, 1, 25, 1980, 128, 4, 246.2, 327.0),
    (8, 4, 33, 528, 64, 4, 42.4, 37.4), (8, 4, 33, 528, 128, 2, 47.5, 40.7), (8, 2, 30, 1084, 128, 2, 66.0, 58.8), (8, 4, 34, 1072, 128, 2, 101.4, 81.0)]

# 16 bit, 128 channels: query / KV heads, segment, block, tokens; us with the general kernel and with two (geometric mean of fused and not), of shapes
# drawn from some 500 that lie around the line; clustered keys, and keys of which many come near a row's maximum
PATHS_CLUSTERED = [
    (40, 8, 1024, 32, 15643, 62.0, 99.3), (12, 2, 128, 32, 20635, 123.5, 91.0), (32, 4, 1024, 32, 48507, 165.6, 127.9), (8, 8, 1024, 32, 28603, 42.9, 68.0),
    (28, 4, 1024, 32, 18715, 59.1, 71.3), (16, 4, 512, 32, 42299, 131.1, 117.6), (32, 4, 256, 128, 36475, 94.7, 84.4), (32, 4, 512, 64, 45243, 127.5, 134.9),
    (32, 8, 1024, 128, 72955, 93.7, 99.0), (8, 8, 1024, 32, 63995, 173.6, 124.2), (12, 2, 512, 64, 46715, 77.2, 74.3), (32, 4, 512, 32, 34299, 148.9, 116.4),
    (40, 8, 128, 32, 5531, 71.1, 58.7), (32, 32, 1024, 32, 17499, 57.2, 100.7), (32, 16, 1024, 32, 42907, 177.4, 193.5), (16, 8, 1024, 32, 45243, 102.3, 116.8),
    (16, 4, 1024, 128, 119675, 121.3, 107.6), (8, 2, 512, 32, 40443, 75.2, 94.7), (16, 8, 128, 32, 14299, 86.3, 81.2), (40, 8, 1024, 128, 25595, 50.5, 68.5),
    (32, 8, 1024, 128, 114427, 200.8, 133.1), (16, 8, 1024, 128, 121339, 165.8, 112.1), (16, 8, 256, 128, 55419, 146.2, 87.4), (16, 4, 1024, 32, 51579, 93.1, 123.0),
    (16, 4, 512, 64, 63995, 127.9, 97.6), (12, 2, 256, 128, 58363, 127.3, 107.7), (8, 8, 512, 64, 49531, 110.3, 82.7), (32, 4, 128, 32, 18555, 185.9, 128.7),
    (32, 16, 1024, 128, 71547, 121.6, 98.8), (8, 8, 128, 32, 22619, 167.8, 115.9), (32, 32, 128, 32, 6171, 75.2, 61.0), (16, 8, 512, 64, 35003, 62.1, 73.4),
    (16, 4, 128, 32, 21147, 124.7, 129.5), (16, 8, 512, 32, 47451, 209.5, 192.8), (28, 4, 256, 128, 21627, 96.0, 76.2), (16, 8, 1024, 32, 60699, 170.9, 137.5),]
PATHS_MANY_NEAR = [
    (32, 4, 256, 128, 33531, 102.0, 99.2), (12, 2, 128, 32, 14299, 76.8, 110.2), (32, 8, 512, 32, 37147, 241.3, 252.5), (12, 2, 512, 64, 58363, 137.4, 174.2),
    (12, 2, 256, 128, 70011, 198.6, 137.5), (32, 32, 128, 32, 7995, 104.2, 71.1), (16, 4, 1024, 32, 55419, 116.0, 211.5), (24, 8, 512, 64, 28603, 119.6, 116.2),
    (24, 8, 128, 32, 5819, 51.4, 46.0), (12, 2, 512, 64, 40443, 73.9, 84.0), (24, 8, 256, 128, 20219, 81.7, 63.0), (28, 4, 512, 64, 18683, 72.8, 61.2),
    (16, 4, 512, 64, 51579, 100.9, 118.1), (40, 8, 256, 128, 24699, 183.3, 106.5), (12, 2, 128, 32, 24763, 181.8, 164.1), (16, 8, 1024, 128, 110843, 146.9, 159.1),
    (32, 8, 256, 128, 57211, 222.0, 190.2), (32, 4, 128, 32, 12891, 103.3, 112.9), (32, 8, 1024, 32, 36475, 114.1, 168.3), (28, 4, 1024, 128, 59131, 149.0, 107.8),
    (16, 8, 1024, 32, 67099, 233.6, 234.4), (32, 32, 1024, 32, 14299, 49.2, 72.9), (28, 4, 256, 128, 15227, 56.6, 50.1), (32, 16, 128, 32, 11291, 114.9, 125.9),
    (8, 2, 1024, 32, 78363, 144.8, 237.7), (16, 4, 1024, 32, 59835, 150.9, 219.4), (32, 4, 512, 64, 45243, 149.1, 182.9), (24, 8, 512, 64, 26107, 107.0, 105.4),
    (40, 8, 512, 32, 12795, 85.9, 107.5), (24, 8, 1024, 32, 28603, 111.9, 158.1), (16, 8, 1024, 32, 40443, 102.6, 147.0), (16, 4, 256, 128, 47355, 92.2, 124.7),
    (32, 16, 1024, 32, 28603, 97.2, 119.0), (24, 8, 256, 128, 36859, 213.7, 104.6), (32, 16, 512, 32, 17499, 68.7, 94.0), (16, 4, 1024, 32, 74331, 259.7, 273.7),]
PATHS_HARNESS = """
#include <cstdio>
enum { CP_BF16 = 0, CP_F32 = 1, CP_F16 = 2, CP_FLAG_FORCE_SPLIT_SCORE = 16 };
struct cp_params { int dtype, flags; };
struct Dims { int B, Hq, Hkv, g, n1, n2, d; };
%s
%s
int main() {
  Dims m{1};
  cp_params p{CP_BF16, 0};
  while (std::scanf("%%d %%d %%d %%d %%d", &m.Hq, &m.Hkv, &m.n1, &m.n2, &m.d) == 5) {
    m.g = m.Hq / m.Hkv;
    std::printf("%%d\\n", int(score_is_split(p, m)));
  }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    text = (CSRC / "score.cu").read_text()
    a, b = text.index("constexpr size_t kSmemShared"), text.index("struct ScoreProblem")
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text(HARNESS % text[a:b])
    subprocess.run(["g++", "-std=c++17", "-O1", "-o", str(d / "rule"), str(d / "rule.cpp")], check=True)

    def ask(cases):
        out = subprocess.run([str(d / "rule")], input="\n".join(" ".join(map(str, c[:6])) for c in cases), capture_output=True, text=True, check=True)
        return [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    return ask


def test_the_faster_split_is_taken(rule):
    for c, (CL, nb, _) in zip(SPLIT, rule(SPLIT)):
        U = 4 if c[1] % 4 == 0 else 2 if c[1] % 2 == 0 else 1
        few = next(x for x in (1, 2, 4, 8) if 48 * U * ((-(-c[3] // x) + 7) // 8 * 8) <= 200 * 1024)
        assert CL == (few if c[6] < c[7] else 2 * few), c


def test_the_faster_share_of_an_sm_is_taken(rule):
    for c, (_, _, two) in zip(SHARED, rule(SHARED)):
        assert two == (c[7] < c[6]), c


def test_every_row_that_is_accepted_has_room(rule):
    cases = [(2, g, n1, n2, d, es) for g in (1, 2, 3, 4, 8) for n1 in (1, 9, 10, 37, 38, 400) for n2 in list(range(1, 8193, 37)) + [552, 553, 1064, 1065, 8192]
             for d, es in ((64, 2), (128, 4))]
    for (Hkv, g, n1, n2, _, _), (CL, nb, _) in zip(cases, rule(cases)):
        U = 4 if g % 4 == 0 else 2 if g % 2 == 0 else 1
        assert CL in (1, 2, 4, 8) and CL * nb >= n2 and nb % 8 == 0 and 48 * U * nb <= 200 * 1024


@pytest.fixture(scope="module")
def is_split(tmp_path_factory):
    common, fast = (CSRC / "cp_common.cuh").read_text(), (CSRC / "score_fast.cu").read_text()
    d = tmp_path_factory.mktemp("paths")
    (d / "rule.cpp").write_text(PATHS_HARNESS % (common[common.index("inline int score_heads"):common.index("// Device status block.")],
                                                 fast[fast.index("constexpr long long kFastMinScores"):fast.index("// K2 dispatcher.")]))
    subprocess.run(["g++", "-std=c++17", "-O1", "-o", str(d / "rule"), str(d / "rule.cpp")], check=True)

    def ask(cases):
        lines = "\n".join(f"{hq} {hkv} {-(-n // seg)} {-(-n // blk)} {d}" for hq, hkv, seg, blk, n, d in cases)
        return [x == "1" for x in subprocess.run([str(tmp / "rule")], input=lines, capture_output=True, text=True, check=True).stdout.split()]
    tmp = d
    return ask


@pytest.mark.parametrize("paths,mean,worst", [(PATHS_CLUSTERED, 1.02, 1.4), (PATHS_MANY_NEAR, 1.035, 1.4)])
def test_the_faster_path_is_taken_where_it_matters(is_split, paths, mean, worst):
    losses = [(c[6] if split else c[5]) / min(c[5:]) for c, split in zip(paths, is_split([c[:5] + (128,) for c in paths]))]
    assert sum(losses) / len(losses) <= mean and max(losses) <= worst, sorted(zip(losses, paths))[-5:]


def test_which_scores_may_take_two_kernels(is_split):
    assert is_split([(32, 8, 1024, 128, 131072, 128), (32, 8, 512, 32, 131072, 128), (32, 8, 512, 32, 131072, 64), (32, 8, 512, 64, 32768, 128),
                     (32, 8, 512, 32, 1, 128), (4, 1, 131072, 16, 131072, 128)]) == [True, True, False, False, False, False]
