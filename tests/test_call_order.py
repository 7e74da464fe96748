"""When a decode call may read ahead of the kernel in front of it: the bookkeeping of the library's calls per stream, on the
host alone (the header is compiled by itself)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_05527_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include "gear_call_order.h"
using gear::CallOrder;
static int failures = 0;
#define EXPECT(cond) do { if (!(cond)) { ++failures; std::printf("line %d: %s\n", __LINE__, #cond); } } while (0)
static void call(CallOrder& o, const CallOrder::Key& k) { const uint64_t n = o.begin(); o.queued(k, n); }
static CallOrder::Write write(CallOrder& o, const CallOrder::Key& k) { call(o, k); return o.written(k); }
int main() {
  const CallOrder::Key s = {0x7000, 0, 0, true}, other = {0x7100, 0, 0, true};
  {  // directly behind the write; behind another call; a call on another stream does not count
    CallOrder o;
    EXPECT(!o.another_since(s, CallOrder::Write()));
    const CallOrder::Write w = write(o, s);
    EXPECT(!o.another_since(s, w));
    call(o, other);
    EXPECT(!o.another_since(s, w) && !o.another_since(other, w));
    call(o, s);
    EXPECT(o.another_since(s, w));
    EXPECT(!o.another_since(s, write(o, s)));
  }
  {  // a call that failed has queued nothing
    CallOrder o;
    const CallOrder::Write w = write(o, s);
    o.begin();
    EXPECT(!o.another_since(s, w));
  }
  {  // the default stream has one handle on every device
    CallOrder o;
    const CallOrder::Key d0 = {0, 0, 0, true}, d1 = {0, 0, 1, true};
    const CallOrder::Write w = write(o, d0);
    call(o, d1);
    EXPECT(!o.another_since(d0, w) && !o.another_since(d1, w));
  }
  {  // a handle that names a stream per thread
    CallOrder o;
    const CallOrder::Key t = {2, 0, 0, false};
    const CallOrder::Write w = write(o, t);
    call(o, t);
    EXPECT(!o.another_since(t, w));
  }
  {  // another thread draws its number before the write and launches behind it, or the other way round: not known to lie behind
    CallOrder o;
    const uint64_t early = o.begin();
    const CallOrder::Write w = write(o, s);
    o.queued(s, early);
    EXPECT(!o.another_since(s, w));
    const uint64_t late = o.begin();                // began behind the write, not launched yet
    EXPECT(!o.another_since(s, w));
    o.queued(s, late);
    EXPECT(o.another_since(s, w));
    o.queued(s, early);                             // a late report takes nothing back
    EXPECT(o.another_since(s, w));
  }
  {  // captured calls: a discarded capture has launched nothing, a write in a graph may be repeated at any time
    CallOrder o;
    const CallOrder::Key g = {0x7000, 41, 0, true}, h = {0x7000, 42, 0, true};
    const CallOrder::Write w = write(o, s);
    call(o, g);
    EXPECT(!o.another_since(s, w) && o.another_since(g, w) && !o.another_since(h, w));
    const CallOrder::Write wg = write(o, g);
    call(o, s);
    EXPECT(!o.another_since(s, wg) && !o.another_since(g, wg));
    call(o, g);
    EXPECT(!o.another_since(s, wg) && o.another_since(g, wg));
  }
  {  // streams come and go: what is kept is bounded, and forgetting a stream only makes its calls wait
    CallOrder o;
    const CallOrder::Write w = write(o, s);
    call(o, s);
    for (uint64_t i = 1; i < 5000; ++i) call(o, CallOrder::Key{0x10000 + 16 * i, 0, 0, true});
    EXPECT(!o.another_since(s, w));
    call(o, s);
    EXPECT(o.another_since(s, w));
  }
  {  // two threads on one stream
    CallOrder o;
    std::thread t([&] { for (int i = 0; i < 100000; ++i) call(o, s); });
    bool behind_itself = false;
    for (int i = 0; i < 1000; ++i) behind_itself = behind_itself || o.another_since(other, write(o, other));
    t.join();
    EXPECT(!behind_itself);
  }
  return failures != 0;
}
"""


def test_calls_that_are_known_to_lie_behind_a_write(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "order.cc", tmp_path / "order"
    src.write_text(PROGRAM)
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread", "-I", CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
