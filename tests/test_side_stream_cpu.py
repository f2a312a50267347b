"""Streams and function attributes that belong to a device follow their user to another one:
side_stream.h with a fake of the runtime calls (the machine needs no GPU)."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_16094_gb300", "csrc")
PROGRAM = r"""
#include <cstdio>
#include <set>
#include "side_stream.h"
struct Fake {
  using Stream = int *;
  using Event = long *;
  static inline int device = 0, made = 0, fail_at = -1;
  static inline bool no_events = false;
  static inline std::set<const void *> live;
  static inline int stream_device[64];
  static bool current_device(int &d) { d = device; return true; }
  static bool create(bool, Stream &s) {
    if (made == fail_at) return false;
    stream_device[made] = device;
    s = &stream_device[made++];
    live.insert(s);
    return true;
  }
  static bool create(Event &e) {
    if (no_events) return false;
    e = new long;
    live.insert(e);
    return true;
  }
  static void destroy(Stream s) { live.erase(s); }
  static void destroy(Event e) { live.erase(e); delete e; }
};
#define NEED(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
  {
    gipm::SideStreamOf<Fake> a;
    NEED(a.create(false) && Fake::made == 1 && *a.s == 0);
    NEED(a.create(false) && Fake::made == 1);  // kept on its device
    Fake::device = 1;
    NEED(a.create(false) && Fake::made == 2 && *a.s == 1 && Fake::live.size() == 3);
    Fake::device = 0;
    Fake::fail_at = 2;
    NEED(!a.create(true) && !a.s && Fake::live.empty());  // reported, nothing left behind
    Fake::fail_at = -1;
    Fake::no_events = true;
    NEED(!a.create(true) && !a.s && Fake::live.empty());
    Fake::no_events = false;
    NEED(a.create(true) && *a.s == 0 && Fake::live.size() == 3);
  }
  NEED(Fake::live.empty());
  gipm::DeviceOnce once;
  NEED(once.needed(0) && once.needed(1));
  once.done(0);
  NEED(!once.needed(0) && once.needed(1));
  once.done(1);
  NEED(!once.needed(1) && once.needed(2) && once.needed(63));
  return 0;
}
"""


def test_state_follows_the_device(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_other_device_state():
    """Every stream the library makes is a SideStream, and no function attribute hangs on a flag
    of the whole process."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        if name != "launch.h":
            assert "cudaStreamCreate" not in text, name
        assert not re.search(r"static bool \w+ *=", text), name
