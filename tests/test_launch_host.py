"""What the any-shape kernels ask of a device (csrc/simt_layout.h), with devices that grant less."""
import pathlib
import subprocess

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2608_21308_b200" / "csrc"

GRANTS = r"""
#include "simt_layout.h"
using namespace e2ttt;
int main() {
    int asked = 0;
    auto grants = [&](int clusters) { return [&asked, clusters](int cl) { ++asked; return cl == 16 ? clusters : 1000; }; };
    for (int N = 1; N <= 300; ++N)
        for (int io = 0; io < 2; ++io) {
            const int cl = simt_cluster_size(N, io);
            if (cl != (io == 0 && N <= 7 ? 16 : cl) || cl > 16) return 1;
            if (simt_granted_cluster(cl, grants(7)) != cl) return 2;        // a GPU that runs them
            const int less = simt_granted_cluster(cl, grants(0));           // one that does not, or whose calculator reports an error
            if (less != (cl > 8 ? 8 : cl)) return 3;
        }
    return asked == 2 * 7 ? 0 : 4;                                          // portable sizes are not asked for
}
"""


def test_a_device_without_clusters_of_16_still_runs_the_fp64_kernels(tmp_path):
    (tmp_path / "grants.cpp").write_text(GRANTS)
    subprocess.run(["g++", "-std=c++17", "-I", str(CSRC), str(tmp_path / "grants.cpp"), "-o", str(tmp_path / "grants")], check=True)
    assert subprocess.run([str(tmp_path / "grants")]).returncode == 0

SHARE = r"""
#include "simt_layout.h"
using namespace e2ttt;
int main() {
    for (int d : {1, 16, 64, 128, 1024})
        for (int h : {1, 16, 256, 8192})
            for (int C = 1; C <= 512; ++C)
                if (f64_fwd_two(149, d, h, C) && 2 * (f64_fwd_small(d, h, C) + 1024) > 228 * 1024) return 1;
    if (!f64_fwd_two(149, 16, 16, 446) || f64_fwd_two(149, 16, 16, 447)) return 2;      // the longest chunks, narrow and wide tiles
    if (!f64_fwd_two(300, 64, 256, 215) || f64_fwd_two(300, 64, 256, 216)) return 3;
    return f64_fwd_two(148, 16, 16, 1) ? 4 : 0;                                         // an SM for each
}
"""


def test_more_fp32_sequences_than_sms_share_them(tmp_path):
    (tmp_path / "share.cpp").write_text("#include <initializer_list>\n" + SHARE)
    subprocess.run(["g++", "-std=c++17", "-I", str(CSRC), str(tmp_path / "share.cpp"), "-o", str(tmp_path / "share")], check=True)
    assert subprocess.run([str(tmp_path / "share")]).returncode == 0
