"""The counts that a traversal depth's tiles pass on (msp_hostdev.cuh), at
sizes no test allocates: past 2^31 children the running numbers stay exact, so
that a depth whose children exceed the pair table is always seen to."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# tiles of 256 pairs, all split into 64 children each: 2^14 children a tile, 2^33
# in all (2^19 tiles: 2^27 pairs); then a mix whose counts end at 2^31 - 1 pairs
SOURCE = r"""
#include <cstdio>
#include "msp_hostdev.cuh"
template <int W>
static bool run(const int (*tile)(long long, int), long long tiles) {
    const unsigned long long mask = (1ull << 62) - 1;    // a status word's value
    unsigned long long sum[W] = {};
    long long want[4] = {};
    for (long long t = 0; t < tiles; ++t) {
        long long w[W], ex[4];
        for (int k = 0; k < W; ++k) w[k] = (long long)(sum[k] & mask);
        msp::trav_unpack(w, ex);
        for (int k = 0; k < 4; ++k)
            if (ex[k] != want[k]) {
                std::printf("tile %lld count %d: %lld, not %lld\n", t, k, ex[k], want[k]);
                return false;
            }
        int tot[4];
        for (int k = 0; k < 4; ++k) want[k] += tot[k] = tile(t, k);
        msp::trav_pack(tot, w);
        for (int k = 0; k < W; ++k) sum[k] = (sum[k] + (unsigned long long)w[k]) & mask;
    }
    return true;
}
static const int all_split(long long, int k) { return k == 0 ? 256 * 64 : (k == 1 ? 256 : 0); }
static const int mixed(long long t, int k) {
    const int split = (int)(t % 200), near = (256 - split) / 2;
    return k == 0 ? 64 * split : (k == 1 ? split : (k == 2 ? near : 256 - split - near));
}
static const int no_far(long long t, int k) { return k < 3 ? mixed(t, k) : 0; }
static const int near_only(long long, int k) { return k == 2 ? 256 : 0; }
static const int far_only(long long, int k) { return k == 3 ? 256 : 0; }
int main() {
    const long long most = ((1ll << 31) - 1) / 256;      // tiles of the largest table
    return run<3>(all_split, 1ll << 19) && run<3>(mixed, most) && run<3>(near_only, most) &&
           run<3>(far_only, most) && run<2>(all_split, 1ll << 19) && run<2>(no_far, most) &&
           run<2>(near_only, most) ? 0 : 1;
}
"""


def test_running_counts_are_exact_beyond_the_pair_table(tmp_path):
    src, exe = tmp_path / "counts.cpp", tmp_path / "counts"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-x", "c++", "-I",
                           os.path.join(ROOT, "paper_2301_10570_gb300", "csrc"), str(src), "-o",
                           str(exe)])
    done = subprocess.run([str(exe)], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout
