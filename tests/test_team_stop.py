"""The end of a team's tile loop in the tensor-core corrector (csrc/dg_team.h), run on the CPU: the workers, the
copy warp and the MMA warp as threads with the kernel's sequence of barriers, for every choice of the barriers
after which a warp is late, that is, reads its stop number only when the workers have come as far as they can.
Every run has to end with all three out of their loops."""
import itertools
import os
import subprocess

import pytest

import paper_2502_09714_gb300  # noqa: F401

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <thread>
#include "dg_team.h"

#ifdef FLAG                       // a plain flag in place of the numbers: the mistake that the runs have to show
struct Stop {
  volatile int flag;
  void init() { flag = 0; }
  void set(int, int) { flag = 1; }
  bool copy_stops(int) const { return flag; }
  bool mma_stops(int) const { return flag; }
};
#else
using Stop = dg::TeamStop;
#endif

static std::mutex m;
static std::condition_variable cv;
// barrier between the workers and one warp.  A late warp (bit n of `late`: after barrier n) reads its number when
// the workers wait for it again or are out of the loop; for any other the workers wait until it has.
struct Barrier {
  unsigned late = 0;
  int workers = 0, warp = 0, read = 0;
  bool gone = false;
};
static Barrier copy_bar, mma_bar;
static const Barrier* waiting = nullptr;         // where the workers wait, if they do
static bool workers_done = false, hung = false;

static void worker_sync(Barrier& b) {
  std::unique_lock<std::mutex> l(m);
  const int n = ++b.workers;
  waiting = &b;
  cv.notify_all();
  cv.wait(l, [&] { return b.warp >= n || b.gone || hung; });
  if (b.warp < n) hung = true;                   // the warp has left: nobody will come
  waiting = nullptr;
  cv.notify_all();
  if (!(b.late >> (n - 1) & 1)) cv.wait(l, [&] { return b.read >= n || b.gone || hung; });
}
static void warp_sync(Barrier& b) {
  std::unique_lock<std::mutex> l(m);
  const int n = ++b.warp;
  cv.notify_all();
  cv.wait(l, [&] { return b.workers >= n || hung || workers_done; });
  if (b.workers < n) hung = true;                // the workers are through without this barrier
  if (b.late >> (n - 1) & 1) cv.wait(l, [&] { return (waiting == &b && b.workers > n) || workers_done || hung; });
}

static void has_read(Barrier& b, bool gone) {
  std::lock_guard<std::mutex> l(m);
  ++b.read;
  b.gone = gone;
  cv.notify_all();
}

int main(int, char** argv) {
  const int tiles = std::atoi(argv[1]), fail_tile = std::atoi(argv[2]), fail_phase = std::atoi(argv[3]);
  copy_bar.late = std::atoi(argv[4]);
  mma_bar.late = std::atoi(argv[5]);
  static Stop stop;
  stop.init();
  std::thread copy([&] {
    for (int it = 0;; ++it) {
      warp_sync(copy_bar);
      const bool last = hung || stop.copy_stops(it);
      has_read(copy_bar, last);
      if (last) break;
    }
  });
  std::thread mma([&] {
    for (int n = 0;; ++n) {
      warp_sync(mma_bar);
      const bool last = hung || stop.mma_stops(n);
      has_read(mma_bar, last);
      if (last) break;
    }
  });
  // the workers of the kernel
  int it = 0, failed = 0;
  for (; it < tiles; ++it) {
    worker_sync(copy_bar);
    worker_sync(mma_bar);
    if (it == fail_tile && fail_phase == 1) { failed = 1; break; }
    worker_sync(mma_bar);
    if (it == fail_tile && fail_phase == 2) { failed = 2; break; }
  }
  stop.set(it, failed);
  worker_sync(mma_bar);
  worker_sync(copy_bar);
  {
    std::lock_guard<std::mutex> l(m);
    workers_done = true;
    cv.notify_all();
  }
  copy.join();
  mma.join();
  return hung ? 3 : 0;
}
"""

# (tiles, tile and phase of a wait that runs out): whole runs, and every place of a failure
RUNS = [(t, -1, 0) for t in range(4)] + [(t, k, p) for t in (1, 3) for k in range(t) for p in (1, 2)]


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("team")
    src = d / "team.cpp"
    src.write_text(HARNESS)
    out = {}
    for name, flags in (("numbers", []), ("flag", ["-DFLAG"])):
        out[name] = str(d / name)
        subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", *flags, "-I",
                        os.path.join(ROOT, "paper_2502_09714_gb300", "csrc"), str(src), "-o", out[name]], check=True)
    return out


def _run(exe, run, late_copy, late_mma):
    return subprocess.run([exe, *map(str, run), str(late_copy), str(late_mma)], timeout=60).returncode


@pytest.mark.parametrize("run", RUNS)
def test_every_role_ends(harness, run):
    tiles, k, phase = run
    n_copy = tiles + 1 if phase == 0 else k + 2
    n_mma = 2 * tiles + 1 if phase == 0 else 2 * k + phase + 1
    for late_copy in range(1 << n_copy):
        assert _run(harness["numbers"], run, late_copy, 0) == 0
    for late_mma in range(1 << n_mma):
        assert _run(harness["numbers"], run, 0, late_mma) == 0
    for late_copy, late_mma in itertools.product((0, (1 << n_copy) - 1), (0, (1 << n_mma) - 1)):
        assert _run(harness["numbers"], run, late_copy, late_mma) == 0


def test_a_plain_flag_is_found_out(harness):
    """A copy warp late after the last tile's barrier sees the flag one barrier early; likewise an MMA warp late
    after the barrier whose wait ran out."""
    assert _run(harness["flag"], (2, -1, 0), 0, 0) == 0
    assert _run(harness["flag"], (2, -1, 0), 1 << 1, 0) == 3
    assert _run(harness["flag"], (2, 1, 1), 0, 1 << 2) == 3
