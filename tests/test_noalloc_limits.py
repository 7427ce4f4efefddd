"""What e2ttt_chunk_fwd_noalloc's scratch must hold of a call in fp64 that it accepts (csrc/noalloc.cu, simt_layout.h)."""
import pathlib
import subprocess

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2608_21308_b200" / "csrc"

FITS = r"""
#include "simt_layout.h"
#include <initializer_list>
using namespace e2ttt;
int main() {
    const size_t limit = (size_t)8 << 20, room = limit / 2 * 5 - 256;
    for (int d = 1; d <= 1024; d += d < 64 ? 7 : 48)
        for (int h : {1, 3, 16, 40, 64, 256, 1024, 8192})
            for (int C = 1; C <= 512; C += C < 64 ? 9 : 32)
                for (int nmat : {2, 3}) {
                    const size_t counted = simt_layout(d, h, C, nmat, 4, false, false).per_seq * 8, kept = simt_layout(d, h, C, nmat, 4, false, false, 0, 0, 1, 1).per_seq * 8;
                    const size_t n = (limit - 256) / counted;  // sequences that are accepted
                    if (n * kept > room) return 1;
                }
    return 0;
}
"""


def test_every_accepted_fp32_call_fits(tmp_path):
    (tmp_path / "fits.cpp").write_text(FITS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", str(CSRC), str(tmp_path / "fits.cpp"), "-o", str(tmp_path / "fits")], check=True)
    assert subprocess.run([str(tmp_path / "fits")]).returncode == 0
