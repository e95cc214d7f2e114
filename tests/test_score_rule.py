"""The rules that split the general score kernel's key blocks over clusters and put two of its CTAs on an SM, compiled for the host as they stand in
the source, against measured times."""
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


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    text = (CSRC / "score.cu").read_text()
    a, b = text.index("constexpr size_t kSmemShared"), text.index("// as many heads per CTA as divide the group")
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
