"""The bounded map that holds a slot's executable graphs (csrc/lru.h), compiled for the host:
it never holds more than its bound, gives back what leaves, and that is the entry used
longest ago."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_16022_gb300", "csrc")

SRC = r"""
#include "lru.h"
#include <cassert>
#include <cstdio>
int main() {
  dotpe::LruMap<int> m(3);
  int out = -1, seen = 0;
  assert(!m.find("a"));
  assert(!m.put("a", 1, &out) && !m.put("b", 2, &out) && !m.put("c", 3, &out));
  assert(m.size() == 3 && *m.find("a") == 1);          // order of use: b, c, a
  assert(m.put("d", 4, &out) && out == 2);             // c, a, d
  assert(!m.find("b") && *m.find("c") == 3);           // a, d, c
  assert(m.put("e", 5, &out) && out == 1);             // d, c, e
  m.erase("c");
  assert(m.size() == 2 && !m.find("c") && !m.put("f", 6, &out));
  m.for_each([&](int v) { seen += v; });
  assert(seen == 4 + 5 + 6);
  for (int k = 0; k < 1000; ++k) {                     // a pattern per call: bounded, each given back once
    out = -1;
    assert(m.put("k" + std::to_string(k), 100 + k, &out) && m.size() == 3);
    assert(k < 3 || out == 100 + k - 3);
  }
  puts("ok");
}
"""


def test_bounded_map(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=address,undefined", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stderr
