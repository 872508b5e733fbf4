"""Ordering rules of the kernels that a run cannot show (what breaks them shows by timing alone),
checked on the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_05061_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name", sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh"))))
def test_step_slots_is_read_and_written_as_one_word(name):
    """The attention reads step_slots while the ingest before it may write it: in device code only
    put_step_slots and get_step_slots touch it, each with one 64-bit scalar access."""
    text = source(name)
    if name == "kvpop_internal.cuh":
        for f, op in (("put_step_slots", "st.relaxed.gpu.global.u64"), ("get_step_slots", "ld.relaxed.gpu.global.u64")):
            body = text[text.index(f + "("):]
            assert op in body[:body.index("\n}")]
        return
    assert not re.search(r"step_slots\s*\[", text)
    assert not re.search(r"ld\w*\(\s*(a\.|st\.|a\.st\.)?step_slots", text)


def test_cluster_ingest_writes_no_peer_before_all_have_started():
    """A CTA's shared memory may be written by its cluster only once it runs: each CTA arrives at a
    cluster barrier at its start and waits for it before the first remote store."""
    text = source("kvpop_ingest_cluster.cu")
    body = text[text.index("ingest_cluster_kernel(ClArgs"):]
    at = [body.index(x) for x in ("cluster_started_arrive();", "griddepcontrol.wait", "cluster_started_wait();",
                                  "st_cluster_v4(")]
    assert at == sorted(at)
    assert "cluster_sync();" not in body[:at[2]]
