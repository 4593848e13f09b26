"""What the integer functions' callers and loads rely on beyond their values
(csrc/fxmath.cuh), compiled for the host."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1607_02904_gb300", "csrc")


def run(tmp_path, body, text=""):
    (tmp_path / "t.cpp").write_text(body)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-o", str(tmp_path / "t"), str(tmp_path / "t.cpp")], check=True)
    return subprocess.run([str(tmp_path / "t")], input=text, capture_output=True, text=True, check=True).stdout


def test_logarithm_table_is_declared_for_its_16_byte_loads(tmp_path):
    # the declaration's alignment, not where a linker happened to put the table
    out = run(tmp_path, '#include "fxmath.cuh"\n#include <cstdio>\nint main() { printf("%zu", __alignof__(tgb::fx::kLog2)); }')
    assert int(out) % 16 == 0
