"""The tensor-core kernels' sources: lanes of a warp that meet again at a warp-wide instruction do not
part before it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1511_04552_gb300", "csrc")


def _source(name):
    """The file without comments."""
    src = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)


def _block(src, start):
    """The brace block that opens at or after start, and where it ends."""
    a = src.index("{", start)
    depth = 0
    for i in range(a, len(src)):
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        if depth == 0:
            return src[a:i + 1], i + 1
    raise AssertionError("unbalanced braces")


@pytest.mark.parametrize("name", ["net_conv.cu", "net_gemm.cu"])
def test_waits_before_a_vote_are_voted_on(name):
    """In a role whose lanes vote, or load tensor memory, after a bounded wait, the wait's result is
    voted on first: a lane that gave up alone would leave the others in the vote for ever."""
    src = _source(name)
    seen = 0
    # the branches of the roles: if (warp ...) { } else if (warp ...) { }
    for m in re.finditer(r"if \(warp[^;{]*\) \{", src):
        role, _ = _block(src, m.end() - 1)
        collective = "__all_sync(0xffffffffu, mask" in role or "tmem_ld" in role
        if not collective or "_wait(" not in role:
            continue
        for w in re.finditer(r"(\w+) =[^;]*?(?:role|cluster)_wait\([^;]*;(.{0,80})", role, flags=re.S):
            seen += 1
            assert "__all_sync(0xffffffffu, %s)" % w.group(1) in w.group(2), role[w.start():w.end()]
        alone = re.search(r"if \([^;{]*!(?:role|cluster)_wait\(", role)
        assert not alone, role[alone.start():alone.end() + 80]
    assert seen >= 2


@pytest.mark.parametrize("name", ["net_conv.cu", "net_gemm.cu"])
def test_lanes_meet_before_tensor_memory_loads(name):
    """tcgen05.ld is undefined unless all 32 lanes execute it together: in a loop around one no lane
    goes on alone, and the lanes meet before the load (tmem_ld16 does that itself)."""
    src = _source(name)
    helper, _ = _block(_source("net_tc.cuh"), _source("net_tc.cuh").index("void tmem_ld16("))
    assert helper.index("__syncwarp();") < helper.index("tcgen05.ld")
    seen = 0
    for m in re.finditer(r"\bfor \([^{}]*?\) \{", src):
        body, _ = _block(src, m.end() - 1)
        inner = min((body.find(t) for t in ("tmem_ld16(", "tmem_ld8_async(") if t in body), default=-1)
        if inner < 0 or "role_wait(" in body or "cluster_wait(" in body or "bar_wait(" in body:
            continue  # none, or a loop over tiles, whose waits are voted on
        seen += 1
        assert "continue;" not in body, body[:200]
        if "tmem_ld8_async(" in body:
            assert 0 <= body.find("__syncwarp();") < inner, body[:200]
    assert seen >= 2
