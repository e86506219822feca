"""Buffers that the field kernels must not dereference (another GPU's, the host's) go
through the copy engine: the rule, compiled from the library's header and run here."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_01035_gb300", "csrc")
PROGRAM = """
#include "ms_pointer.h"
using namespace msgb;
int main() {
  bool ok = kernel_reaches(kMemDevice, 0, 0) && kernel_reaches(kMemDevice, 3, 3);   // its own memory
  ok = ok && !kernel_reaches(kMemDevice, 1, 0) && !kernel_reaches(kMemDevice, 0, 1);   // another GPU's
  ok = ok && kernel_reaches(kMemManaged, 1, 0);
  ok = ok && !kernel_reaches(kMemHost, 0, 0) && !kernel_reaches(kMemUnregistered, 0, 0);
  return ok ? 0 : 1;
}
"""


def test_the_rule(tmp_path):
    src, exe = tmp_path / "rule.cpp", str(tmp_path / "rule")
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
