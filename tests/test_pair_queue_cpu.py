"""The tile queue of a CTA pair: the home CTA overwrites a description in the
other CTA's shared memory, so that CTA's reads of it must be ordered before the
store: by a barrier of their own CTA after every lane has read, then by one
arrival with cluster-scope release that the home's wait acquires."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_22541_gb300", "csrc")


def _body(text, head):
    start = text.index("{", text.index(head))
    depth, end = 1, start + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
    return text[start:end]


def _text(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_descriptions_are_handed_back_with_cluster_scope():
    text = _text("pair.cuh")
    queue = _body(text, "struct PairQueue")
    assert "mbar_arrive_pair(" not in queue  # CTA scope
    release = _body(queue, "void release(")
    assert release.index("__syncwarp()") < release.index("mbar_arrive(")
    assert "mbar_wait_acquire_pair(empty" in _body(queue, "bool push(")
    assert ".acquire.cluster." in _body(text, "bool mbar_wait_acquire_pair(")
    assert ".release.cluster." in _body(text, "void mbar_arrive_release_pair(")
    forward = _body(text, "bool pair_forward(")
    assert forward.index("mbar_wait(PairQueue::read") < forward.index("mbar_arrive_release_pair(PairQueue::empty")


def test_every_role_releases_as_a_warp():
    for name in ("gemm_pair.cu", "gemm_fp8.cu"):
        text = _text(name)
        assert not re.search(r"if \([^)]*\) tq\.release", text), name
        assert len(re.findall(r"tq\.release\((?:issuer|lane == 0)\)", text)) >= 3, name
