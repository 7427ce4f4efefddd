"""What e2ttt_chunk_fwd_noalloc accepts of fp32 calls (csrc/api.cu, simt_layout.h): those whose e2ttt_workspace_bytes fits its scratch."""
import ctypes
import pathlib
import subprocess

import pytest

from paper_2608_21308_b200 import binding as E

ROOT = pathlib.Path(__file__).resolve().parent.parent
CSRC = ROOT / "paper_2608_21308_b200" / "csrc"

# A forward without saved states asks for twice the bytes of a bf16 call on the SIMT kernels, whatever the fp64 kernels make of them: what a
# caller of the fixed scratch counts by does not move with the kernels
FITS = r"""
#include "simt_layout.h"
#include <initializer_list>
using namespace e2ttt;
int main() {
    int compact = 0;
    for (int d = 1; d <= 1024; d += d < 64 ? 7 : 48)
        for (int h : {1, 3, 16, 40, 64, 256, 1024, 8192})
            for (int C = 1; C <= 512; C += C < 64 ? 9 : 5)
                for (int nmat : {2, 3}) {
                    const SimtLayout l = simt_layout(d, h, C, nmat, 4, false, false, 0, 0, 1, 1);
                    if (l.per_seq != simt_layout(d, h, C, nmat, 4, false, false).per_seq) return 1;
                    F64Layout f{};
                    if (f64_layout(f, l.M[2] + (nmat == 3 ? ((size_t)d * h + 31) / 32 * 32 : 0), 1, d, h, C, nmat, false, 4) > l.per_seq) return 2;
                    if (l.fl.compact && f64_parts(C, d, h) != 1) return 3;
                    compact += l.fl.compact;
                    if (simt_layout(d, h, C, nmat, 4, true, true, 0, 0, 1, 1).fl.compact) return 4;  // training calls keep the keys apart
                }
    return compact > 1000 ? 0 : 5;
}
"""


def test_the_fp64_kernels_need_no_more_than_callers_count_by(tmp_path):
    (tmp_path / "fits.cpp").write_text(FITS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", str(CSRC), str(tmp_path / "fits.cpp"), "-o", str(tmp_path / "fits")], check=True)
    assert subprocess.run([str(tmp_path / "fits")]).returncode == 0


@pytest.mark.parametrize("kind", [E.E2TTT_MLP_GELU, E.E2TTT_SWIGLU])
@pytest.mark.parametrize("N,d,h,C", [(1, 64, 256, 16), (4, 64, 256, 16), (40, 64, 256, 16), (1, 828, 1, 365), (1, 832, 1, 512), (2, 828, 1, 365),
                                     (1, 1024, 1, 300), (1, 1024, 2048, 64), (7, 24, 40, 8)])
def test_accepted_is_what_fits_by_the_size_that_callers_can_ask_for(N, d, h, C, kind):
    """Null tensors: a refused call says so (-5), any other ends before a launch with another error."""
    import re

    limit = re.search(r"#define E2TTT_NOALLOC_SCRATCH_BYTES \((\d+)u << (\d+)\)", (ROOT / "include" / "e2ttt.h").read_text())
    limit = int(limit[1]) << int(limit[2])
    assert limit == E.E2TTT_NOALLOC_SCRATCH_BYTES
    p = E.make_params(N, 1, C, d, h, C, kind)
    rc = E.lib().e2ttt_chunk_fwd_noalloc(ctypes.byref(p), *[None] * 12)
    assert rc != 0 and (rc == -5) == (E.e2ttt_workspace_bytes(p, 0) > limit)
    assert E.e2ttt_workspace_bytes(E.make_params(1, 1, 365, 828, 1, 365, kind), 0) < limit
    # the array is as large as the limit, not more
    assert "g_static_scratch[E2TTT_NOALLOC_SCRATCH_BYTES]" in (CSRC / "noalloc.cu").read_text()
