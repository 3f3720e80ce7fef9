"""Orderings of the pair scheduler that no run can be made to miss: the source
of each function must hold them, in the order given."""
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1511_07658_gb300", "csrc")


def body(name, function):
    """A function's text, comments taken out, from its name to the closing brace in column 0."""
    with open(os.path.join(CSRC, name)) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    at = re.search(rf"^[^\n;]*\b{function}\([^;{{]*\{{", src, re.M).start()
    return src[at:src.index("\n}\n", at)]


@pytest.mark.parametrize(
    "name,function,pattern",
    [
        # The peer CTA's reads of an item before the leader's control warp overwrites its slot:
        # released to the peer's own barrier, and from there to the cluster.
        ("gvm_sched.cu", "pair_item_release", r"mbar_arrive\(&sh\.item_empty"),
        ("gvm_sched.cu", "pair_relay", r"mbar_wait\(&sh\.item_empty.*mbar_arrive_release_cta\(&sh\.item_empty"),
        # One lane's reading of the abort word decides for the warp that claims together.
        ("gvm_sched.cu", "pair_control", r"seen = bcast\(seen\);(?!.*sh\.abort \?).*\(seen & 2u\) \? 0 : acquire<true>"),
        # Every lane's reads of a landing before lane 0 frees it for the next copies.
        ("gvm_pair.cuh", "pr_convert_aligned", r"read_b\(3\);.*__syncwarp\(\);\s*if \([^)]*\) mbar_arrive\(&ps->land_free"),
        ("gvm_pair.cuh", "pr_convert_packed", r"__syncwarp\(\);\s*if \([^)]*\) \{\s*mbar_arrive\(&ps->land_free"),
        ("gvm_pair.cuh", "pr_vec_convert", r"__syncwarp\(\);\s*if \([^)]*\) mbar_arrive\(&ps->land_free"),
    ],
)
def test_ordering_is_in_the_source(name, function, pattern):
    assert re.search(pattern, body(name, function), re.S)
