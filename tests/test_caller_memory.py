"""The rule for working on the caller's buffers in place (csrc/caller_mem.h): only where
kernels of the handle's device reach all of the buffer, in one allocation, aligned.
Compiled and run on the host: memory of another device, which the runtime can copy but
a kernel without peer access cannot touch, must go through a copy."""
import os
import shutil
import subprocess

import pytest

from paper_2510_24543_gb300 import build as B

SRC = r"""
#include <cstdio>
#include "caller_mem.h"
using egpe::PtrFacts;
static int bad = 0;
static void expect(const char* what, bool got, bool want) {
  if (got != want) { std::printf("%s: %d\n", what, got); ++bad; }
}
int main() {
  const uint64_t base = 0x7f0000000000ull, p = base + 4096;
  const size_t bytes = 1 << 20;
  auto facts = [](uint64_t d, uint64_t s, size_t n) { PtrFacts f; f.device_ptr = d; f.range_start = s; f.range_size = n; return f; };
  expect("own device", egpe::in_place(facts(p, base, 4096 + bytes), p, bytes, 16), true);
  expect("not reachable by kernels", egpe::in_place(facts(0, base, 4096 + bytes), p, bytes, 16), false);
  expect("reachable elsewhere", egpe::in_place(facts(p + 64, base, 4096 + bytes), p, bytes, 16), false);
  expect("unknown pointer", egpe::in_place(PtrFacts(), p, bytes, 16), false);
  expect("no range known", egpe::in_place(facts(p, 0, 0), p, bytes, 16), false);
  expect("one byte short", egpe::in_place(facts(p, base, 4095 + bytes), p, bytes, 16), false);
  expect("smaller than the field", egpe::in_place(facts(p, p, bytes - 1), p, bytes, 16), false);
  expect("before the range", egpe::in_place(facts(p, p + 16, bytes * 2), p, bytes, 16), false);
  expect("misaligned", egpe::in_place(facts(p + 8, base, 8192 + bytes), p + 8, bytes, 16), false);
  expect("aligned for FP32", egpe::in_place(facts(p + 8, base, 8192 + bytes), p + 8, bytes, 8), true);
  expect("null", egpe::in_place(facts(0, 0, 0), 0, bytes, 16), false);
  return bad;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_rule(tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-I", B.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.skipif(not os.path.isdir(B.CSRC), reason="sources not installed")
def test_every_in_place_use_asks():
    """The standalone evaluations decide by the rule, not by alignment alone."""
    with open(os.path.join(B.CSRC, "engine_impl.cuh")) as f:
        src = f.read()
    for fn in ("param_grad(const C* psi", "enq_evaluation(const C* psi", "precondition(int mode"):
        body = src[src.index("Engine<R>::" + fn):]
        assert "usable(" in body[:body.index("\n}\n")], fn
