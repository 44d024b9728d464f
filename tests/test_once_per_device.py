"""Kernel attributes set once per device while several threads make their first call: no call goes on before the attributes are
set.  The header is host code, compiled and run here."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_04732_b200", "csrc")

PROGRAM = r"""
#include "per_device.cuh"
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <thread>
int main() {
  flop::OncePerDevice once;
  // the first thread's setting takes until the second thread's call has returned
  std::mutex mu;
  std::condition_variable cv;
  bool started = false, second_returned = false, first_set = false, second_set = false;
  std::thread first([&] {
    once(3, [&] {
      std::unique_lock<std::mutex> lk(mu);
      started = true;
      cv.notify_all();
      cv.wait(lk, [&] { return second_returned; });
      first_set = true;
      return 0;
    });
  });
  bool covered;
  {
    std::unique_lock<std::mutex> lk(mu);
    cv.wait(lk, [&] { return started; });
  }
  once(3, [&] { second_set = true; return 0; });
  {
    std::unique_lock<std::mutex> lk(mu);
    covered = first_set || second_set;
    second_returned = true;
    cv.notify_all();
  }
  first.join();
  int again = 0, other = 0, failed = 0, unknown = 0;
  once(3, [&] { ++again; return 0; });
  once(4, [&] { ++other; return 0; });
  const int rc = once(5, [&] { ++failed; return 7; });
  once(5, [&] { ++failed; return 0; });
  once(5, [&] { ++failed; return 0; });
  for (int dev : {-1, -1, 64, 64}) once(dev, [&] { ++unknown; return 0; });
  printf("%d %d %d %d %d %d\n", (int)covered, again, other, rc, failed, unknown);
}
"""


def test_attributes_are_set_before_any_call_goes_on(tmp_path):
    (tmp_path / "main.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "main")
    subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-pthread", "-fsanitize=thread", "-x", "c++", "-I" + CSRC, "-o", exe, str(tmp_path / "main.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr[-2000:]
    assert [int(v) for v in r.stdout.split()] == [1, 0, 1, 7, 2, 4]
