"""The way out of the thread-block clusters after a timed-out wait, read from the
kernel sources (a timeout is not provoked on a GPU: what it would show is a store
into the shared memory of a CTA that has ended).

A CTA of a step kernel is the target of its peers' st.async stores.  When one of
its waits gives up it must not end before they have stopped (a cluster barrier,
which ended CTAs count as arrived at), must not re-arm a barrier whose phase it
has not seen end."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_04235_gb300", "csrc")


def _body(text, head):
    """The brace-matched body after the first occurrence of `head`."""
    i = text.index("{", text.index(head))
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i + 1:j]
    raise AssertionError(head)


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


STEPS = [("decode_rows.cu", "decode_rows_kernel(", "dr_leave"), ("decode_cluster.cu", "decode_cluster_kernel(", "dc_leave")]


@pytest.mark.parametrize("name,kernel,leave", STEPS)
def test_timed_out_cta_waits_for_its_cluster(name, kernel, leave):
    text = _source(name)
    out = _body(text, leave + "(")
    assert "barrier.cluster.arrive" in out and "barrier.cluster.wait" in out
    # every way out of the kernel after the set-up barrier passes the abort flag to it
    body = _body(text, kernel)
    body = body[body.index("barrier.cluster.wait"):]
    ends = [m.start() for m in re.finditer(r"\breturn;\n    \}\n\n", body)] + [len(body)]
    assert ends
    at = 0
    for e in ends:
        assert re.search(r"if \((\*abort_flag|dc_fate\(P\)->abort)\)( \{[^}]*?| )" + leave + r"\(", body[at:e]), body[at:e][-300:]
        at = e


def test_exchange_barriers_are_armed_only_after_a_seen_phase():
    """The batched step arms its two exchange barriers in turn, after a wait that
    has seen their phase end; the single-cluster step has one per phase, armed
    before the cluster's set-up barrier."""
    arms = [line for line in _source("decode_rows.cu").split("\n") if re.search(r"mbar_expect_tx\(bar, ", line)]
    assert len(arms) >= 2 and all(re.search(r"\bok\b", line) for line in arms)
    body = _body(_source("decode_cluster.cu"), "decode_cluster_kernel(")
    assert "mbar_expect_tx" in body[:body.index("barrier.cluster.arrive")]
    assert "mbar_expect_tx" not in body[body.index("barrier.cluster.arrive"):]


def test_batched_step_sends_nothing_after_a_timed_out_wait():
    """Barriers that are not armed again would take the bytes of a whole step, which
    may pass the 2^20 that a barrier counts: a thread that has given up sends to
    no CTA, and the peers that miss its bytes give up too."""
    text = _source("decode_rows.cu")
    lines = text.split("\n")
    sends = [i for i, line in enumerate(lines) if re.search(r"\bdr_send[24]\(", line) and "void " not in line]
    assert len(sends) >= 5
    for i in sends:
        if "k < nc; k++" in lines[i - 1] + lines[i]:  # dr_attention: nc is its parameter
            assert re.search(r"xbar, live\);", text)
            continue
        assert re.search(r"\blive\b", "\n".join(lines[max(0, i - 6):i + 1])), lines[i]
