"""What the decode kernels (csrc/apply.cu) rest on and a CPU can check."""
import pathlib
import re

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
