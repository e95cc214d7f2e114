"""The rule that gives an attention launch to pairs of CTAs or to single ones, compiled for the host as it stands in the source, against
measured times of both kernels."""
import pathlib
import random
import subprocess

import pytest

SOURCE = pathlib.Path(__file__).resolve().parent.parent / "paper_2409_12490_b200" / "csrc" / "attention_sm100.cu"

# query / KV heads, tokens, segment, block, budget (0: dense), us on single CTAs and on pairs (graphs of ten launches in loops of 0.1 s)
MEASURED = [
    (1, 1, 18944, 256, 32, 256, 12.1, 10.8), (8, 2, 41600, 256, 32, 256, 70.3, 78.5), (32, 8, 16576, 256, 32, 256, 107.6, 121.8),
    (1, 1, 56832, 256, 32, 512, 26.3, 22.7), (8, 2, 1184, 256, 32, 512, 16.8, 13.9), (32, 8, 1776, 256, 32, 512, 26.2, 23.8),
    (1, 1, 9472, 512, 32, 1024, 22.5, 15.8), (8, 2, 7104, 512, 32, 1024, 37.6, 31.8), (32, 8, 1184, 512, 32, 1024, 29.7, 24.7),
    (32, 8, 2368, 512, 32, 1024, 45.7, 41.3), (1, 1, 56832, 512, 32, 1408, 47.9, 41.9), (32, 8, 1776, 512, 32, 1408, 39.0, 34.0),
    (1, 1, 75776, 512, 32, 1536, 57.3, 63.8), (8, 2, 2368, 512, 32, 1536, 29.6, 23.8), (32, 8, 1776, 1024, 32, 1024, 32.8, 27.6),
    (1, 1, 18944, 1024, 32, 2048, 36.7, 26.3), (1, 1, 28160, 1024, 32, 4096, 64.6, 73.6), (8, 2, 2368, 1024, 32, 4096, 40.3, 29.5),
    (8, 2, 14208, 1024, 32, 4096, 186.3, 208.5), (1, 1, 75776, 1024, 32, 8192, 269.5, 308.1), (8, 2, 4736, 1024, 32, 8192, 72.1, 64.0),
    (1, 1, 28160, 512, 32, 0, 383.1, 316.5), (8, 2, 14208, 512, 32, 0, 394.5, 444.8), (32, 8, 1776, 512, 32, 0, 44.7, 38.7),
    (32, 8, 4800, 512, 32, 0, 194.6, 219.7)]

HARNESS = """
#include <algorithm>
#include <cstdint>
#include <cstdio>
constexpr int kTile = 128;
struct Dims { int B, Hq, r, seg, blk, k; };
struct SeqSlot { int len; };
%s
int main() {
  Dims m;
  int n, dense, emul;
  SeqSlot s[16];
  while (std::scanf("%%d %%d %%d %%d %%d %%d %%d %%d", &m.B, &m.Hq, &m.seg, &m.blk, &m.k, &dense, &emul, &n) == 8) {
    for (int i = 0; i < n; ++i) std::scanf("%%d", &s[i].len);
    m.r = m.seg / m.blk;
    std::printf("%%d\\n", int(pairs_are_faster(m, s, n, dense, emul)));
  }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    text = SOURCE.read_text()
    a, b = text.index("long long count_units("), text.index("// (segment, pair)s that have query rows, by the tiles they stream")
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text(HARNESS % text[a:b])
    # an index out of the table's bounds traps
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=bounds", "-fsanitize-undefined-trap-on-error", "-o", str(d / "rule"), str(d / "rule.cpp")], check=True)

    def ask(cases):
        lines = "\n".join(" ".join(map(str, [B, Hq, seg, blk, budget // blk if budget else seg // blk, int(budget == 0), int(budget == 0 or budget >= 1536),
                                             len(lens), *lens])) for B, Hq, lens, seg, blk, budget in cases)
        out = subprocess.run([str(d / "rule")], input=lines, capture_output=True, text=True, check=True).stdout.split()
        return [x == "1" for x in out]
    return ask


def test_the_faster_kernel_is_taken(rule):
    for (Hq, Hkv, n, seg, blk, budget, single, pair), pairs in zip(MEASURED, rule([(1, c[0], [c[2]], c[3], c[4], c[5]) for c in MEASURED])):
        assert pairs == (pair < single), (Hq, n, seg, budget)


def test_any_shape_stays_within_the_table(rule):
    rng = random.Random(1)
    cases = []
    for _ in range(4000):
        seg = 256 * rng.randint(1, 8)
        blk = rng.choice([32, 64, 128])
        budget = rng.choice([0, max(seg, blk * rng.randint(1, 300)) // blk * blk])
        lens = [rng.randint(1, 10 ** rng.randint(1, 6)) for _ in range(1 if budget == 0 else rng.randint(1, 16))]
        cases.append((rng.randint(1, 4), rng.choice([1, 2, 3, 8, 32]), lens, seg, blk, budget))
    cases += [(1, 1, [256 * 444], 256, 32, 1024), (1, 1, [256 * 444 + 1], 256, 32, 1024), (1, 1, [2 ** 31 - 1 - 256], 512, 32, 0), (1, 1, [1], 256, 32, 256)]
    assert len(rule(cases)) == len(cases)
