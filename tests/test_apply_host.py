"""What the decode kernels (csrc/apply.cu) rest on and a CPU can check."""
import pathlib
import re
import subprocess

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2608_21308_b200" / "csrc"


def kernel(name):
    text = (CSRC / "apply.cu").read_text()
    body = text[text.index(f" {name}(const ApplyArgs a) {{"):]
    return body[:body.index("\n}\n")]


@pytest.mark.parametrize("name", ["apply_kernel", "apply_stream_kernel"])
def test_the_cluster_has_started_before_its_shared_memory_is_written(name):
    """A CTA without hidden units reaches the store of its partial sums at once; the first CTA need not run by then unless a cluster
    barrier says so."""
    body = kernel(name)
    store = re.search(r"\bslot0\[[^\]]*\] = ", body).start()
    arrive, wait = body.find("cluster_arrive();"), body.find("cluster_wait();")
    assert 0 <= arrive < wait < store


def test_a_wait_that_gives_up_shows_in_the_outputs():
    """The decode step has no status word.  The flag that such a wait leaves is looked at before the partial sums are handed over, and
    again before the CTA gives up its shared memory to copies that may still be under way."""
    body = kernel("apply_stream_kernel")
    flag, store, drain = body.find("dead = *(volatile int*)&sh.dead"), body.find("= dead ? __int_as_float"), body.rfind("if (dead)")
    assert 0 <= body.find("*dead = 1") < flag < store < drain


SIZES = r"""
#include "apply.h"
#include <cstdio>
#include <initializer_list>
using namespace e2ttt;
int main() {
    int bad = 0;
    for (int N : {1, 33, 34, 37, 45, 56, 71, 93, 94, 128, 148, 149, 296, 297, 5000})
        for (int d = 4; d <= kDsCols; d += 4)
            for (int h = 4; h <= kDsMaxHidden; h += 4) {
                const StreamGeometry g = apply_stream_geometry(N, d, h);
                const int cols = g.per < kDsCols ? g.per : kDsCols;
                if (g.smem > kDsMaxSmem || g.nslots < 1 || g.per * g.cl < h || g.slot_bytes < 32u * (d > cols ? d : cols) || g.ring_at % 128 ||
                    g.slot_bytes % 16 || g.ring_at < kDsFixedBytes + 4u * g.per)
                    if (bad++ < 5) std::printf("N=%d d=%d h=%d: %zu bytes\n", N, d, h, g.smem);
            }
    return bad != 0;
}
"""


def test_no_call_takes_more_shared_memory_than_the_limit_set_for_all(tmp_path):
    """The limit is a kernel attribute, set once: a larger call later would be refused at its launch."""
    (tmp_path / "sizes.cpp").write_text(SIZES)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", str(CSRC), str(tmp_path / "sizes.cpp"), "-o", str(tmp_path / "sizes")], check=True)
    out = subprocess.run([str(tmp_path / "sizes")], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
