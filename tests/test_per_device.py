"""Limits that the CUDA runtime keeps per device are set on each device: the
flag that remembers it, compiled alone, and no process-wide flag in its place
in the sources."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1101_1427_gb300", "csrc")

PROGRAM = r"""
#include "per_device.h"
int main() {
  static spin::OncePerDevice once;
  for (int dev = -1; dev <= 64; ++dev) if (once.done(dev)) return 1;
  once.mark(0);
  if (!once.done(0) || once.done(1) || once.done(63)) return 2;
  once.mark(63);
  if (!once.done(63) || once.done(1) || once.done(62)) return 3;
  once.mark(64);
  once.mark(-1);
  if (once.done(64) || once.done(-1) || !once.done(0) || once.done(1)) return 4;
  return 0;
}
"""


def test_the_flag_is_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_no_process_wide_flag_guards_a_limit():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = open(path).read()
        assert not re.search(r"static\s+(?:std::atomic<)?bool>?\s+\w+\s*(?:=|;|\{)", text), path
