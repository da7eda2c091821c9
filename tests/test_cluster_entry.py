"""Kernels whose CTAs write one another's shared memory: a CTA may be written only after
it has started, so a cluster-wide barrier comes before the first such store.  Read from
the source: on a GPU the unordered store mostly goes unnoticed."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_19075_gb300", "csrc")


def _body(text, kernel):
    """The kernel's body with the bodies of its lambdas (declarations, not yet calls) left out."""
    start = text.index("{", text.index(")", re.search(r"\n\s+" + kernel + r"\(", text).end()))
    body = text[start:text.index("\n}\n", start)]
    return re.sub(r"\n    auto \w+ = \[&\].*?\n    };", "", body, flags=re.S)


@pytest.mark.parametrize("source,kernel", [("ring_cluster.cu", "ring_cluster_kernel"),
                                           ("ring_dp_cluster.cu", "ring_dp_cluster_kernel")])
def test_cluster_barrier_before_the_first_remote_store(source, kernel):
    body = _body(open(os.path.join(CSRC, source)).read(), kernel)
    first_store = re.search(r"\bpublish(_y)?\(", body)
    arrive, wait = body.find("cluster.barrier_arrive();"), body.find("cluster.barrier_wait();")
    assert first_store and 0 <= arrive < wait < first_store.start()
    # every thread of the CTA passes both: no return in between
    assert not re.search(r"\breturn\b", body[arrive:wait])
