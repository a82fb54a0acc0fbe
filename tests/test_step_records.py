"""Which forces steps are recorded (csrc/step_records.h, host bookkeeping): first run eager, second
recorded, then replayed; several keys side by side; the one used longest ago makes room; a recording
that did not complete is not tried again; everything is released."""
import os
import subprocess

import paper_2506_04055_gb300 as eng

SRC = os.path.join(os.path.dirname(os.path.abspath(eng.__file__)), "csrc")

PROGRAM = r"""
#include <cstdio>
#include <set>
#include "step_records.h"
static std::set<int*> live;
struct Drop { void operator()(int* p) const { if (!live.erase(p)) std::puts("released twice"); delete p; } };
using Records = ctd::StepRecords<int*, Drop>;
using Act = Records::Act;
// a step of the key: e eager, r recorded and replayed, p replayed, x the recording failed and it ran eagerly
static char step(Records& rec, uint64_t key, bool capture_works = true) {
  switch (rec.next(key)) {
    case Act::kReplay: return *rec.replay(key) == (int)key ? 'p' : '!';
    case Act::kRecord:
      if (capture_works) {
        int* e = new int((int)key);
        live.insert(e);
        rec.recorded(key, e);
        return *rec.replay(key) == (int)key ? 'r' : '!';
      }
      rec.refused(key);
      rec.ran(key);
      return 'x';
    default: rec.ran(key); return 'e';
  }
}
static void show(const char* what, Records& rec, const char* keys, bool works = true) {
  std::printf("%s ", what);
  for (const char* k = keys; *k; ++k) std::putchar(step(rec, (uint64_t)*k, works));
  std::printf(" %zu\n", live.size());
}
int main() {
  {
    Records rec;
    show("one", rec, "AAAA");
    show("alternating", rec, "ABABAB");
    rec.clear();
    show("cleared", rec, "AAA");
    rec.clear();
    show("refused", rec, "AAAAAA", false);
    rec.clear();
    show("four", rec, "ABCDABCDABCD");
    show("fifth", rec, "EEABCD");
    rec.clear();
    show("pairs", rec, "AABBCCDDEEFF");
  }
  std::printf("left %zu\n", live.size());
}
"""


def test_records(tmp_path):
    src, exe = tmp_path / "records.cpp", tmp_path / "records"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-I", SRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    assert out[:8] == [
        "one erpp 1",
        "alternating peprpp 2",
        "cleared erp 1",
        "refused exeeee 0",
        "four eeeerrrrpppp 4",
        "fifth ereeee 0",
        "pairs erererererer 4",
        "left 0",
    ]
