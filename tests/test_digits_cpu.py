"""The integer joins of the digit products (csrc/blas_digits.cu) on the host, with undefined behaviour trapped:
the accumulators' bits (1.5 2^23 plus an integer, a Gram element's two added) become one integer."""
import random
import re
import subprocess
from pathlib import Path

CSRC = Path(__file__).resolve().parents[1] / "paper_0907_3261_gb300" / "csrc"

HARNESS = """
#include <algorithm>
#include <cstdint>
#include <cstdio>
#define WD_DEV inline
typedef long long i64;
typedef unsigned long long u64;
using std::min;
static int __clzll(long long v) { return v ? __builtin_clzll((u64)v) : 64; }
namespace fx {
inline u64 absbits(i64 v) { return (u64)(v ^ (v >> 63)); }
inline i64 shr_s(i64 v, int n) { return v >> n; }
}
%s
template <int ND> void run(const unsigned* j, unsigned b) {
  int k;
  const i64 s = product_sum<ND>(j, b, k);
  std::printf("%%lld %%lld %%d\\n", (long long)joined<ND, 0>(j, b), (long long)s, k);
}
int main() {
  unsigned j[8], b;
  int nd;
  while (std::scanf("%%d %%u", &nd, &b) == 2) {
    for (int i = 0; i < nd; ++i) if (std::scanf("%%u", j + i) != 1) return 1;
    nd == 7 ? run<7>(j, b) : run<8>(j, b);
  }
}
"""


def function(src, head):
    m = re.search(r"template <[^>]*>\nWD_DEV i64 " + head + r"\(.*?\n}\n", src, re.S)
    assert m
    return m.group(0)


def test_joins_are_exact_and_defined(tmp_path):
    src = (CSRC / "blas_digits.cu").read_text()
    (tmp_path / "j.cpp").write_text(HARNESS % (function(src, "joined") + function(src, "product_sum")))
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-o",
                    tmp_path / "j", tmp_path / "j.cpp"], check=True)
    rng = random.Random(1)
    magic, lines, sums = 0x4B400000, [], []
    for _ in range(2000):
        nd, two = rng.choice([7, 8]), rng.random() < 0.5
        top = 1 << rng.randint(4, 19)
        v = [rng.randint(-top, top) for _ in range(nd)]
        if rng.random() < 0.3:
            v[:rng.randint(1, nd - 1)] = [0] * nd
            v = v[:nd]
        b = 2 * magic if two else magic
        lines.append(" ".join(str(x) for x in [nd, b] + [(b + x) % 2 ** 32 for x in v]))
        sums.append((nd, sum(x << 8 * (nd - 1 - i) for i, x in enumerate(v))))
    run = subprocess.run([tmp_path / "j"], input="\n".join(lines), capture_output=True, text=True)
    assert run.returncode == 0, run.stderr
    out = run.stdout
    for (nd, want), line in zip(sums, out.splitlines(), strict=True):
        one, s, k = map(int, line.split())
        # `joined` counts the order 0 in units of 2^40, product_sum in units of 2^(43 - k): exact but for one rounding
        unit = 8 * (nd - 1)
        assert abs(one * 2 ** (unit - 40) - want) <= 2 ** (unit - 40) // 2
        scaled = s * 2 ** k * 2 ** (unit - 43) if k + unit >= 43 else s / 2 ** (43 - k - unit)
        if nd == 8:
            assert abs(scaled - want) <= max(2 ** (unit - 43 + k) // 2, 0) and (k == 19 - 32 or abs(s) >= 2 ** 60)
        else:
            assert abs(scaled - want) <= 2 ** (unit - 43) // 2
