"""CPU: which calls of a plan launch, capture and replay (csrc/scw_replay.h). Only a key's second call in a row may
capture: outputs used in turn never pay for a graph, whether one of them has been captured before or not."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include "scw_replay.h"
int main(int, char** argv) {
  static int keys[256];
  scw::ReplayRule r;
  for (const char* c = argv[1]; *c; ++c) {
    if (*c == '-') { r.drop(); continue; }  // another solution
    const void* k = &keys[(int)*c];
    const scw::ReplayRule::Step s = r.next(k);
    std::putchar(s == scw::ReplayRule::LAUNCH ? 'l' : s == scw::ReplayRule::CAPTURE ? 'c' : 'r');
    r.done(s, k);
  }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("replay")
    (d / "t.cpp").write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2404_07293_gb300", "csrc"), "-o", str(d / "t"),
                    str(d / "t.cpp")], check=True)
    return lambda calls: subprocess.run([str(d / "t"), calls], check=True, capture_output=True, text=True).stdout


@pytest.mark.parametrize("calls,steps", [
    ("a", "l"), ("aaaa", "lcrr"),
    ("abababab", "llllllll"),            # in turn, nothing captured
    ("aabababab", "lclrlrlrl"),          # in turn after one was captured: that one replays, the other launches
    ("aabbab", "lclclr"), ("aabbb", "lclcr"), ("aba", "lll"), ("abb", "llc"),
    ("aa-aaa-a", "lclcrl"), ("a-a-a", "lll"),
])
def test_sequences(rule, calls, steps):
    assert rule(calls) == steps
