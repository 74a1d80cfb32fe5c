"""What the library remembers about devices on the host (csrc/device_state.h) and
its staging of uploads (csrc/staging.h), with the CUDA calls played by the test."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_12350_gb300",
                    "csrc")

PRELUDE = r"""
#include <cstdio>
#include <cstdlib>
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); std::exit(1); } } while (0)
"""


def _run(tmp_path, body, header="device_state.h"):
    src, exe = str(tmp_path / "t.cpp"), str(tmp_path / "t")
    with open(src, "w") as f:
        f.write(f'#include "{header}"\n' + PRELUDE + body)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-pthread", "-I", CSRC, src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_occupancy_is_kept_by_device_and_not_after_a_failure(tmp_path):
    _run(tmp_path, r"""
int main() {
  mamute::OccupancyMemo memo;
  int asked = 0;
  auto answer = [&](int n) { return [&asked, n] { ++asked; return n; }; };
  CHECK(memo.get({0, 64, 16, 0, 0, 0, 100}, answer(-1)) == -1);  // a failed query
  CHECK(memo.get({0, 64, 16, 0, 0, 0, 100}, answer(2)) == 2);    // is asked again
  CHECK(memo.get({0, 64, 16, 0, 0, 0, 100}, answer(7)) == 2 && asked == 2);
  CHECK(memo.get({1, 64, 16, 0, 0, 0, 100}, answer(3)) == 3);    // another device has its own
  CHECK(memo.get({0, 64, 16, 0, 0, 0, 101}, answer(0)) == 0);    // a variant that does not fit
  CHECK(memo.get({0, 64, 16, 0, 0, 0, 101}, answer(5)) == 0 && asked == 4);
  for (int k = 0; k < 5000; ++k) memo.get({0, 0, 0, 0, 0, 0, k}, answer(1));
  CHECK(memo.get({0, 0, 0, 0, 0, 0, 4999}, answer(9)) == 1);     // bounded, the latest kept
}
""")


def test_shared_memory_allowance_is_per_device_and_never_lowered(tmp_path):
    _run(tmp_path, r"""
#include <thread>
#include <vector>
int main() {
  mamute::SmemLimit lim;
  std::vector<size_t> on[70];
  auto set = [&](int dev, int rc = 0) { return [&on, dev, rc](size_t b) { on[dev].push_back(b); return rc; }; };
  CHECK(lim.raise(0, 100, set(0)) == 0 && lim.raise(0, 60, set(0)) == 0);
  CHECK(on[0] == std::vector<size_t>{100});                    // smaller: nothing to do
  CHECK(lim.raise(1, 60, set(1)) == 0 && on[1].size() == 1);    // a second device is set too
  CHECK(lim.raise(1, 80, set(1, 5)) == 5);                      // a failure is reported
  CHECK(lim.raise(1, 80, set(1)) == 0 && on[1].size() == 3);    // and tried again
  CHECK(lim.raise(68, 90, set(68)) == 0 && lim.raise(69, 10, set(69)) == 0);
  CHECK(on[69] == std::vector<size_t>{90});                     // devices without an entry of their own
  // threads with different needs: the attribute only grows
  mamute::SmemLimit many;
  std::atomic<size_t> attr{0};
  std::atomic<bool> fell{false}, early{false};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] {
      for (size_t k = 1; k <= 2000; ++k) {
        const size_t need = k * 8 + t;
        many.raise(0, need, [&](size_t b) {
          if (attr.exchange(b) > b) fell = true;
          return 0;
        });
        if (attr.load() < need) early = true;
      }
    });
  for (auto& t : ts) t.join();
  CHECK(!fell && !early);
}
""")


def test_staging_area_is_bounded(tmp_path):
    _run(tmp_path, r"""
int main() {
  mamute::Staging st;
  int waits = 0, allocs = 0, frees = 0;
  bool refuse = false;
  auto begin = [&] {
    return st.begin([&] { return ++waits, 0; },
                    [&](size_t n) -> void* { return ++allocs, refuse ? nullptr : std::malloc(n); },
                    [&](void* p) { ++frees, std::free(p); });
  };
  CHECK(begin() == 0 && allocs == 0 && waits == 0);
  CHECK(!st.take(1000) && !st.take(10));                     // the first call copies and waits
  begin();
  CHECK(st.bytes() == 1280 && allocs == 1 && waits == 0);
  char* a = static_cast<char*>(st.take(1000));
  char* b = static_cast<char*>(st.take(10));
  CHECK(a && b == a + 1024 && !st.take(1));                  // as much as the call before
  begin();
  CHECK(waits == 1 && st.bytes() == 1536 && frees == 1);
  CHECK(!st.take(10 * mamute::Staging::kMax) && st.take(256));  // a table beyond the bound
  begin();
  CHECK(st.bytes() == mamute::Staging::kMax);                // never more than the bound
  CHECK(!st.take(mamute::Staging::kMax + 1) && st.take(4096));
  begin();
  CHECK(st.bytes() == mamute::Staging::kMax && allocs == 3);
  st.release([&](void* p) { ++frees, std::free(p); });
  CHECK(frees == 3 && st.bytes() == 0 && !st.take(1));
  refuse = true;
  begin();
  CHECK(st.bytes() == 0 && !st.take(1));                     // none to be had: the copies wait
}
""", "staging.h")
