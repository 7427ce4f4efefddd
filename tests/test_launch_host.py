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
