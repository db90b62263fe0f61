"""The exchange of sums between the two threads of a (site, right-hand side) in the fixed-point stencil
(csrc/fixed.cuh), on the host: the function's own text is compiled for two host threads whose warp
barrier is a real one, and each lane in turn is held back before it writes its sums.  Whatever the order,
the lanes must end with the sums that both wrote."""
import re
import subprocess
from pathlib import Path


CSRC = Path(__file__).resolve().parents[1] / "paper_0907_3261_gb300" / "csrc"

HARNESS = """
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <thread>
constexpr int TPB = 2;
struct Lane { unsigned x; };
static thread_local Lane threadIdx;
static std::mutex mx;
static std::condition_variable cv;
static int waiting = 0, phase = 0;
static void __syncwarp() {
  std::unique_lock<std::mutex> l(mx);
  const int mine = phase;
  if (++waiting == 2) { waiting = 0; ++phase; cv.notify_all(); }
  else cv.wait(l, [&] { return phase != mine; });
}
#define WD_DEV inline
%s
static long long acc[2][6][TPB];
static long long hs[2][12];
static void lane(int t, int late) {
  threadIdx.x = t;
  if (t == late) std::this_thread::sleep_for(std::chrono::milliseconds(200));
  long long au[6];
  for (int q = 0; q < 6; ++q) {
    au[q] = 1000 * (t + 1) + q;
    acc[0][q][t] = 10000 * (t + 1) + q;
    acc[1][q][t] = 100000 * (t + 1) + q;
  }
  exchange(acc, au, t, hs[t]);
}
int main() {
  for (int late = 0; late < 2; ++late) {
    for (auto& a : acc) for (auto& b : a) for (auto& c : b) c = -1;
    std::thread a(lane, 0, late), b(lane, 1, late);
    a.join(); b.join();
    for (int t = 0; t < 2; ++t) { for (long long v : hs[t]) std::printf("%%lld ", v); std::puts(""); }
  }
}
"""


def test_lanes_see_each_others_sums_in_any_order(tmp_path):
    src = (CSRC / "fixed.cuh").read_text()
    m = re.search(r"template <typename T>\nWD_DEV void exchange\(.*?\n}\n", src, re.S)
    assert m
    body = re.sub(r"#pragma unroll.*", "", m.group(0))
    (tmp_path / "x.cpp").write_text(HARNESS % body)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-o", tmp_path / "x", tmp_path / "x.cpp"], check=True)
    out = subprocess.run([tmp_path / "x"], capture_output=True, text=True, check=True, timeout=60).stdout.split("\n")
    q = range(6)
    # even lane: both upper spins; odd lane: spin 2 (own mu 0, 1 and the other's mu 2, 3), spin 3 (the reverse)
    even = [1000 + i for i in q] + [2000 + i for i in q]
    odd = [20000 + i + 100000 + i for i in q] + [200000 + i + 10000 + i for i in q]
    for late in range(2):
        assert [int(v) for v in out[2 * late].split()] == even
        assert [int(v) for v in out[2 * late + 1].split()] == odd
