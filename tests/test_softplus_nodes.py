"""ln(1 + e^-x) of the visible-score kernel: its table of nodes, and its series in the kernel's own order of operations, compiled for the host as it stands in
the source, against long double."""
import pathlib
import random
import re
import subprocess

import numpy as np

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2409_12490_b200" / "csrc"

HARNESS = """
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#define __device__
#define __forceinline__ inline
struct double2 { double x, y; };
using std::fma;
static int __double2hiint(double x) { int64_t u; std::memcpy(&u, &x, 8); return int(u >> 32); }
static int __double2loint(double x) { int64_t u; std::memcpy(&u, &x, 8); return int(u); }
static const double2 nodes[] = {
#include "softplus_nodes.inc"
};
%s
int main() {
  double worst = 0, x;
  while (std::scanf("%%lf", &x) == 1) {
    double v[1] = {x};
    softplus_nodes(nodes, v);
    const double err = double(fabsl(v[0] - log1pl(expl(-(long double)x))));
    if (!(err <= worst)) worst = err;
  }
  std::printf("%%.3e\\n", worst);
}
"""


def test_nodes():
    rows = re.findall(r"\{(\S+), (\S+)\}", (CSRC / "softplus_nodes.inc").read_text())
    got = np.array([[float.fromhex(v) for v in r] for r in rows], dtype=np.longdouble)
    x = np.arange(40 * 32 + 1, dtype=np.longdouble) / 32
    assert got.shape == (len(x), 2)
    for column, value in ((0, np.log1p(np.exp(-x))), (1, 1 / (1 + np.exp(x)))):
        assert np.all(np.abs(got[:, column] - value) <= value * np.longdouble(2) ** -53 * 1.001)


def test_series(tmp_path):
    text = (CSRC / "score_fast.cu").read_text()
    a = text.index("template <int N>\n__device__ __forceinline__ void softplus_nodes(")
    (tmp_path / "s.cpp").write_text(HARNESS % text[a:text.index("// the same by fmax and fmin")])
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", str(CSRC), "-o", str(tmp_path / "s"), str(tmp_path / "s.cpp")], check=True)
    rng = random.Random(5)
    xs = [rng.uniform(0, 40) for _ in range(100000)] + [10.0 ** rng.uniform(-12, 1.6) for _ in range(20000)]
    xs += [i / 64 for i in range(2561)] + [i / 64 + s * 1e-9 for i in range(1, 2560) for s in (-1, 1)]       # nodes and the points between them
    xs += [0.0, 39.999999, 40.0, 40.0001, 41.0, 700.0, 1e300, float("inf")]
    out = subprocess.run([str(tmp_path / "s")], input="\n".join(map(repr, xs)), capture_output=True, text=True, check=True).stdout
    # half a unit in the last place of a result below 1 (1.1e-16), the tail of the series (2e-17), the rounding of its last product
    assert float(out) <= 1.7e-16
