"""The table of streams whose last library call was an expansion (csrc/pipe_marks.h): host logic, compiled on its own."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_15806_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "pipe_marks.h"
using namespace pipe;
static int failed = 0;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); failed = 1; } } while (0)
static StreamKey key(int device, uint64_t handle) { return stream_key(device, handle); }

int main() {
  for (uint64_t h : {0ull, 4096ull}) {  // a mark on one device outlives calls on another device's stream of the same handle
    ExpansionMarks t;
    CHECK(t.none() && !t.marked(key(0, h)));
    t.mark(key(0, h));
    CHECK(!t.none() && t.marked(key(0, h)) && !t.marked(key(1, h)) && !t.marked(key(0, 8192)));
    CHECK(!t.take(key(1, h)) && !t.take(key(0, 8192)));
    CHECK(t.marked(key(0, h)));
    t.mark(key(0, h));   // (once is enough)
    CHECK(t.take(key(0, h)) && !t.take(key(0, h)) && t.none());
  }
  {  // the two handles of the default stream are one stream, the per-thread default stream is another in every thread
    ExpansionMarks t;
    t.mark(key(0, 0));
    CHECK(t.marked(key(0, 1)) && !t.marked(key(0, 2)));
    t.mark(key(0, 2));
    std::thread([&t] {
      if (t.take(key(0, 2)) || t.marked(key(0, 2)) || !t.marked(key(0, 0))) failed = 1;
    }).join();
    CHECK(t.take(key(0, 2)) && t.take(key(0, 1)) && t.none());
  }
  {  // no device known: treated as marked while any mark stands, and marking it marks all
    ExpansionMarks t;
    CHECK(!t.marked(StreamKey()));
    t.mark(key(0, 7));
    CHECK(t.marked(StreamKey()) && t.take(StreamKey()) && t.marked(key(0, 7)));
    t.mark(StreamKey());
    CHECK(t.take(key(0, 7)) && t.marked(key(0, 7)) && t.marked(key(3, 9)) && !t.none());
  }
  {  // more streams than the table holds: every call waits, none is taken for settled
    ExpansionMarks t;
    for (int i = 0; i <= ExpansionMarks::kMax; ++i) t.mark(key(0, 64 + i));
    for (int i = 0; i <= ExpansionMarks::kMax + 1; ++i) CHECK(t.take(key(0, 64 + i)) && t.marked(key(0, 64 + i)));
    CHECK(!t.none());
  }
  {  // threads on streams of their own do not disturb one another
    ExpansionMarks t;
    std::vector<std::thread> th;
    for (int d = 0; d < 8; ++d)
      th.emplace_back([&t, d] {
        for (int i = 0; i < 20000; ++i) {
          t.mark(key(d, 0));
          if (!t.marked(key(d, 1)) || !t.take(key(d, 0)) || t.marked(key(d, 0))) failed = 1;
        }
      });
    for (auto& x : th) x.join();
    CHECK(t.none());
  }
  return failed;
}
"""


def test_marks_tell_streams_of_different_devices_apart(tmp_path):
    src, exe = tmp_path / "marks.cpp", tmp_path / "marks"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


def test_the_library_asks_for_the_device_of_a_stream():
    text = open(os.path.join(CSRC, "pipe_layout.cu")).read()
    body = text[text.index("key_of("):text.index("void mark_expansion(")]
    assert "cudaGetDevice(&dev)" in body and "stream_key(dev," in body


def test_calls_inside_a_capture_leave_the_marks_alone():
    text = open(os.path.join(CSRC, "pipe_layout.cu")).read()
    assert "g_marks.marked(key_of(stream)) && !capturing(stream); }" in text[text.index("bool expansion_marked(cudaStream_t stream) {"):]
    assert "bool take_expansion_mark(cudaStream_t stream) { return expansion_marked(stream) && g_marks.take(" in text
    text = open(os.path.join(CSRC, "pipe_expand.cu")).read()
    assert re.findall(r"[^\n]*mark_expansion\(s\)", text) == ["  if (!captured) mark_expansion(s)"]
