"""Host rules of the launches, compiled from their headers with the host
compiler: heights of the units of work, the once-per-device setup that they
depend on, and the sharing out of the ring sums."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_16659_gb300", "csrc")


def run_cpp(tmp_path, source, *args, timeout=20):
    """Compiles and runs a C++ program that includes the library's headers;
    its output lines."""
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True, timeout=120)
    r = subprocess.run([str(exe), *map(str, args)], check=True, timeout=timeout,
                       capture_output=True, text=True)
    return r.stdout.split()


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
def test_unit_heights_end_for_any_number_of_slots(tmp_path, n):
    """Also for none, which an unset occupancy gives: every height lies in
    1..64."""
    out = run_cpp(tmp_path, """
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#include "unit_rows.h"
int main(int, char** a) {
  for (bool heavy : {false, true})
  for (int slots : {0, 1, 152, 1824})
    for (int ny : {1, 2, 7, 64, 1024, 5000})
      for (int strips : {1, 2, 19, 1000})
        printf("%d %d ", mlsw::march_rows(atoi(a[1]), heavy, ny, strips, 152, slots),
               mlsw::solo_rows(heavy, ny, strips, 152, slots));
}""", n)
    assert len(out) == 2 * 2 * 4 * 6 * 4 and all(1 <= int(v) <= 64 for v in out)


def test_device_setup_is_seen_whole_by_every_thread(tmp_path):
    """Sixteen threads start together: each finds the value that the setup of
    its device stored, the setup runs once per device, and one that failed is
    tried again."""
    out = run_cpp(tmp_path, """
#include <cstdio>
#include <thread>
#include <vector>
#include "device_once.h"
int main() {
  int wrong = 0, runs = 0;
  for (int trial = 0; trial < 300; ++trial) {
    mlsw::DeviceOnce once;
    int value[64] = {};
    std::atomic<int> count{0}, bad{0}, go{0};
    std::vector<std::thread> t;
    for (int k = 0; k < 16; ++k)
      t.emplace_back([&, k] {
        const int dev = k % 2 ? 63 : 0;
        ++go;
        while (go < 16) {}
        if (once(dev, [&] { value[dev] = 7; ++count; return 0; }) != 0 || value[dev] != 7) ++bad;
      });
    for (auto& x : t) x.join();
    wrong += bad;
    runs += count;
  }
  mlsw::DeviceOnce once;
  int a = once(3, [] { return 5; }), b = once(3, [] { return 0; }), c = once(3, [] { return 9; });
  printf("%d %d %d %d %d", wrong, runs, a, b, c);
}""")
    assert out == ["0", "600", "5", "0", "0"]


@pytest.mark.parametrize("nx,ny", [(1, 1), (8, 100000), (9, 33), (255, 7), (256, 1), (257, 5),
                                   (1024, 1024), (5000, 3), (100000, 8), (1000000, 1), (1, 4099)])
def test_ring_sums_are_shared_out_whole_and_evenly(tmp_path, nx, ny):
    """Every cell belongs to one thread of one block; a block has turns of 256
    threads, and no block has more than twice the turns that an even split
    over all of them leaves, rounded up."""
    out = run_cpp(tmp_path, """
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "ring_plan.h"
int main(int, char** a) {
  const int nx = atoi(a[1]), ny = atoi(a[2]);
  const mlsw::RingPlan p = mlsw::ring_plan(nx, ny);
  const int tx = 1 << p.lgx;
  std::vector<unsigned char> seen((size_t)nx * ny);
  long twice = 0, most = 0;
  for (int b = 0; b < p.blocks; ++b) {
    long turns = 0;
    for (int item = b; item < p.groups * p.segs; item += p.blocks) {
      const int g = item / p.segs, first = (item - g * p.segs) * p.seg;
      const int last = first + p.seg < nx ? first + p.seg : nx;
      turns += (last - first + tx - 1) / tx;
      for (int t = 0; t < 256; ++t) {
        const int y = g * p.tr + (t >> p.lgx);
        if (y >= ny) continue;
        for (int x = first + (t & (tx - 1)); x < last; x += tx) twice += seen[(size_t)y * nx + x]++;
      }
    }
    if (turns > most) most = turns;
  }
  long missing = 0;
  for (unsigned char c : seen) missing += c == 0;
  printf("%ld %ld %ld %d", twice, missing, most, tx * p.tr);
}""", nx, ny)
    twice, missing, most, threads = map(int, out)
    assert (twice, missing, threads) == (0, 0, 256)
    turns = -(-ny // max(1, 256 // max(8, 1 << (min(nx, 256) - 1).bit_length()))) * -(-nx // 256)
    assert most <= 2 * -(-turns // 608)


def test_nominal_heights_of_a_batch_differ(tmp_path):
    """Units of nominal 8 rows are half as high as those of 16, from two rows on,
    for every kind and duration; heights lie in 1..64 and grow with the
    duration; a table in several waves costs no less than its longest unit."""
    out = run_cpp(tmp_path, """
#include <cstdio>
#include <initializer_list>
#include "unit_rows.h"
int main() {
  int bad = 0, seen = 0;
  for (int n = 1; n <= 5; ++n)
    for (int mode = 0; mode < 3; ++mode)
      for (int sub = 0; sub < 2; ++sub) {
        int last = 0;
        for (double t = 1.0; t < 1000.0; t *= 1.02, ++seen) {
          const int rows = mlsw::batch_rows(mlsw::batch_weight(n, mode, sub), t);
          bad += rows < 1 || rows > 64 || rows < last;
          bad += mlsw::half_rows(rows) < 1 || (rows > 1 && mlsw::half_rows(rows) >= rows);
          bad += mlsw::half_rows(rows) != (rows + 1) / 2;
          for (double units : {1.0, 500.0, 1216.0, 1217.0, 1e5})
            bad += !(mlsw::batch_cost(units, units * t, t, 152, 1216) >= t);
          last = rows;
        }
        bad += last != 64;
      }
  printf("%d %d", bad, seen);
}""")
    assert out[0] == "0" and int(out[1]) > 5000
