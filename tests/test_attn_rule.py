"""Which extend rows share a pass over their keys (csrc/sizes.h, compiled here as plain C++): both sides of the line, at
sizes where one side was measured well ahead."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09338_gb300", "csrc")

# query heads, KV heads, sequences, rows a sequence, keys
ROW_BY_ROW = [(16, 8, 8, 8, 256), (16, 8, 6, 8, 1024), (16, 8, 32, 2, 16384), (16, 4, 12, 4, 1024), (32, 8, 4, 8, 1024),
              (16, 8, 96, 1, 16384)]
SHARED = [(16, 8, 96, 8, 4096), (16, 8, 24, 8, 2048), (16, 8, 3, 8, 16384), (16, 4, 16, 6, 8192), (32, 8, 16, 4, 2048)]


def test_line_between_the_kernels(tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    calls = "".join(f"printf(\"%d\", attn_rows_pays({B * m}, {hq}, {hkv}, {m}, {k}));" for hq, hkv, B, m, k in ROW_BY_ROW + SHARED)
    src.write_text("#include <cstdio>\n#include \"sizes.h\"\nusing namespace osp;\nint main() {" + calls + "}")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60).stdout
    assert got == "0" * len(ROW_BY_ROW) + "1" * len(SHARED)
