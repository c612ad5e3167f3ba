"""The host entry point's order of copies, launches and waits (csrc/host_copies.h), compiled for the CPU with calls that are
recorded and made to fail one after the other: whatever fails, nothing that reads or writes the caller's buffers is still
under way when the call returns."""
import os
import subprocess


ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "host_copies.h"
#include <cstdio>
#include <cstdlib>
#include <vector>
using namespace psd;
// Stand-ins for two streams: the caller's buffers are in use while a stream has copies on it that nobody has waited for.
struct Fake {
  int fail_at, calls = 0;
  int pending[2] = {0, 0};               // copies on the stream since it was last waited for
  bool event_set[3] = {false, false, false};
  bool main_has[3] = {false, false, false};   // events the main stream is behind
  std::vector<int> in;
  bool overlap, ran = false, out = false;
  bool ok() { return calls++ != fail_at; }
  bool record(int e, int) { if (!ok()) return false; event_set[e] = true; return true; }
  bool wait(int s, int e) { if (!ok()) return false; if (!event_set[e]) std::abort(); if (s == kHostMain) main_has[e] = true; return true; }
  bool copy_in(int i, int s) { if (!ok()) return false; ++pending[s]; in.push_back(i); return true; }
  int run() {
    if (!ok()) return -7;
    if (in.size() != 4 || (overlap && !(main_has[1] && event_set[2]))) std::abort();
    main_has[2] = true;
    ran = true;
    return 0;
  }
  bool copy_out() { if (!ok()) return false; if (!ran) std::abort(); ++pending[kHostMain]; out = true; return true; }
  bool sync(int s) {
    const bool good = ok();
    pending[s] = 0;                        // a wait that reports an error has waited all the same
    if (s == kHostMain && main_has[2]) pending[kHostCopy] = 0;
    return good;
  }
};
int main() {
  for (int overlap = 0; overlap < 2; ++overlap) {
    int n = 0;
    for (int fail = 0;; ++fail) {
      Fake f{fail};
      f.overlap = overlap != 0;
      const int rc = host_pipeline(f, overlap != 0, 0, -4);
      if (f.pending[0] || f.pending[1]) { std::printf("overlap %d, call %d fails: copies under way on return\n", overlap, fail); return 1; }
      if (rc == 0) {
        if (!f.out || f.calls <= fail - 1) { std::printf("incomplete\n"); return 1; }
        n = fail;
        break;
      }
      if (rc != -4 && rc != -7) { std::printf("status %d\n", rc); return 1; }
    }
    if (n < 6) { std::printf("%d calls only\n", n); return 1; }
  }
  std::printf("ok\n");
  return 0;
}
"""


def test_no_copy_is_under_way_when_the_call_returns(tmp_path):
    src, exe = tmp_path / "copies.cpp", tmp_path / "copies"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_2510_12966_b200", "csrc"), str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
