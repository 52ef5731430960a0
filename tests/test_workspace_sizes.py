"""A draft workspace serves every call of fewer sequences: the sizes in csrc/sizes.h never fall as the rows grow, and
cover what any smaller call takes (compiled here as plain C++)."""
import os
import subprocess

from paper_2609_09338_gb300.workloads import TINY, WORKLOADS

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09338_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include "sizes.h"
using namespace osp;
#define CHECK(x) do { if (!(x)) { printf("%s: nout %d K %d rows %lld sms %d\n", #x, nout, K, r, sms); return 1; } } while (0)
int main(int argc, char **argv) {
    for (int sms : {152, 148, 132}) {
        long long planes = 0, lm = 0;
        int nout = 0, K = 0;
        for (long long r = 1; r <= TC_MAX_ROWS; ++r) {
            CHECK(tc_plane_rows(r) >= planes && tc_tiles_lm(r).rows() >= lm && tc_plane_rows(r) >= r);
            CHECK(tc_tiles(r, 64).npad <= TC_TILE_ROWS && tc_tiles(r, TC_BIG_K).npad <= TC_BIG_ROWS);
            planes = tc_plane_rows(r);
            lm = tc_tiles_lm(r).rows();
        }
        for (int i = 1; i + 1 < argc; i += 2)
            for (int mode = 0; mode < 4; ++mode) {   // block drafting, one range too
                nout = atoi(argv[i]);
                K = atoi(argv[i + 1]);
                const bool block = mode & 1, always = mode & 2;
                long long taken = 0, before = 0;
                for (long long r = 1; r <= TC_MAX_ROWS; ++r) {
                    const int ns = tc_nsplit(nout, K, block ? TC_BLOCK_SPLITS : tc_tiles(r, K), sms);
                    if (ns > 1 || always) taken = std::max(taken, ns * r * nout);
                    const long long got = tc_part_floats(nout, K, r, sms, block, always);
                    CHECK(got >= taken && got >= before);
                    before = got;
                }
            }
        for (int hkv : {1, 2, 4, 8, 16, 32})
            for (int max_ctx : {16, 64, 112, 1008, 2048, 16384, 131072}) {
                nout = hkv;
                K = max_ctx;
                long long taken = 0, before = 0;
                for (long long r = 1; r <= 5000; ++r) {
                    taken = std::max(taken, r * attn_splits((int)r, hkv, max_ctx, sms));
                    const long long got = attn_ranges(r, hkv, max_ctx, sms);
                    CHECK(got >= taken && got >= before);
                    before = got;
                }
                // extend rows: their own ranges, those of rows taken 16 queries together, those of groups of a block call
                for (long long B = 1; B <= 300; ++B)
                    for (int m : {1, 2, 3, 8, 15, 64}) {
                        const long long r = B * m, have = m * attn_ranges(B, hkv, max_ctx, sms);
                        CHECK(have >= r * attn_splits((int)r, hkv, max_ctx, sms));
                        for (int g : {1, 2, 4, 8}) CHECK(have >= r * attn_splits((int)(B * ((m * g + 15) / 16)), hkv, max_ctx, sms));
                        for (long long n = 1; n <= B && n * m <= TC_TILE_ROWS; ++n)
                            CHECK(have >= n * m * attn_splits((int)(n * m), hkv, max_ctx, sms));
                    }
            }
    }
    puts("sizes ok");
}
"""


def test_sizes_never_fall(tmp_path):
    args = []
    for s in [TINY] + [w.shape for w in WORKLOADS.values()]:
        d, a = s.d_model, s.n_q_heads * s.head_dim
        for pair in ((d, s.feat_dim), (s.qkv_rows, 2 * d), (d, a), (2 * s.ffn_dim, d), (d, s.ffn_dim)):
            if pair not in args:
                args.append(pair)
    src, exe = tmp_path / "sizes.cpp", tmp_path / "sizes"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe), *(str(x) for p in args for x in p)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "sizes ok" in r.stdout, r.stdout
