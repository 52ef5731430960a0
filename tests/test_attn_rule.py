"""Which extend rows share a pass over their keys, and how many blocks walk a tree (csrc/sizes.h, compiled here as plain
C++): both sides of each line, at sizes where one side was measured well ahead."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09338_gb300", "csrc")

# query heads, KV heads, sequences, rows a sequence, keys
ROW_BY_ROW = [(16, 8, 8, 8, 256), (16, 8, 6, 8, 1024), (16, 8, 32, 2, 16384), (16, 4, 12, 4, 1024), (32, 8, 4, 8, 1024),
              (16, 8, 96, 1, 16384)]
SHARED = [(16, 8, 96, 8, 4096), (16, 8, 24, 8, 2048), (16, 8, 3, 8, 16384), (16, 4, 16, 6, 8192), (32, 8, 16, 4, 2048)]


def results(tmp_path, calls):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text("#include <cstdio>\n#include \"sizes.h\"\nusing namespace osp;\nint main() {" +
                   "".join(f"printf(\"%d \", {c});" for c in calls) + "}")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return [int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True, timeout=60).stdout.split()]


def test_line_between_the_kernels(tmp_path):
    got = results(tmp_path, [f"attn_rows_pays({B * m}, {hq}, {hkv}, {m}, {k})" for hq, hkv, B, m, k in ROW_BY_ROW + SHARED])
    assert got == [0] * len(ROW_BY_ROW) + [1] * len(SHARED)


# sequences, KB a row, greedy, which sizes keep their slices, clusters of 8, 4, 2, 1 blocks at once, blocks a cluster
LARGE, SMALL = ((1, 0, 0, 0), (15, 72, 152, 304)), ((1, 1, 1, 1), (30, 72, 152, 304))
WALKS = [(1, 593.5, 0, *LARGE, 8), (8, 593.5, 0, *LARGE, 8), (16, 593.5, 0, *LARGE, 8), (64, 593.5, 0, *LARGE, 4),
         (128, 593.5, 0, *LARGE, 2), (256, 593.5, 0, *LARGE, 1), (32, 16, 0, *SMALL, 2), (128, 16, 0, *SMALL, 2),
         (512, 16, 0, *SMALL, 1), (8, 593.5, 1, (0,) * 4, (30, 72, 152, 304), 8), (512, 62.5, 1, (0,) * 4, (45, 108, 228, 456), 1)]


def test_blocks_of_a_walk(tmp_path):
    of = lambda v: "{" + ", ".join(map(str, v)) + "}"
    got = results(tmp_path, [f"8 >> tree_cluster({B}, {kb}, {g}, {of(bool(x) * 1 for x in fit)}, {of(at)})"
                             for B, kb, g, fit, at, _ in WALKS])
    assert got == [w[-1] for w in WALKS]
