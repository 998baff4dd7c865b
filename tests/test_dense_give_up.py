"""How the roles of the dense (tcgen05) kernels end after a wait that ran out, from their source: no GPU is made to let one run out."""
import os
import re

import pytest

import paper_2505_11157_b200

SOURCE = os.path.join(os.path.dirname(paper_2505_11157_b200.__file__), "csrc", "sna_kernels_dense2.cu")
# the barriers that report the copies of a stage, and the MMAs of each issuing role
COPIES = {"forward": ["B_KFULL", "B_VFULL"], "backward_dq": ["Q_KFULL", "Q_VFULL"], "backward_dkdv": ["K_QFULL", "K_YFULL"]}
MMAS = {"forward": ["B_SFULL", "B_PVDONE"], "backward_dq": ["Q_STFULL", "Q_G2DONE"], "backward_dkdv": ["K_STFULL", "K_G2DONE"]}


def block(text, start):
    """(what stands between the brace that opens at or after `start` and its partner, what follows)"""
    at = text.index("{", start) + 1
    begin, depth = at, 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[at], 0)
        at += 1
    return text[begin:at - 1], text[at:]


@pytest.fixture(params=COPIES)
def kernel(request):
    """(name, the loops over a tile's blocks with what follows each)"""
    text = re.sub(r"//[^\n]*", "", open(SOURCE).read())
    body = block(text, text.index(f"\n{request.param}_dense2_kernel("))[0]
    return request.param, [block(body, m.end()) for m in re.finditer(r"for \([^;]*; it <=? total && ok; \+\+it[^{]*", body)]


def waited_for(after):
    """The barrier of the full-length wait for block it - 1 that directly follows a loop."""
    m = re.match(r"\s*(?:if \(total > 0 && ok\) fold\(total - 1\);\s*else )?if \(it > 0\) (?:ok = )?mb_wait_polls\(s32\(&bars\[(\w+)"
                 r"[^;]*\(it - 1\) & 1\)\]\), \(\(it - 1\) >> 1\) & 1, WAIT2\)", after)
    return m and m[1]


def test_no_copy_is_left_under_way(kernel):
    """The producer starts no copy into a stage that has not become free, and waits, with a limit, for its last ones."""
    name, loops = kernel
    (loop, after), = [x for x in loops if "tma_tile(" in x[0]]
    assert re.search(r"if \(!ok\) break;", loop[loop.rindex("mb_wait("):loop.index("mb_expect(")])
    assert re.findall(r"tma_tile\([^;]*bars\[(\w+) \+ s\]", loop) == COPIES[name]
    waits = block(after, after.index("for (int j = max(0, it - "))[0]
    assert re.findall(r"mb_wait_polls\(s32\(&bars\[(\w+) \+ j[^;]*WAIT2\)", waits) == COPIES[name]


def test_no_mma_is_left_under_way(kernel):
    """After a role that issues MMAs, or the one that releases them, comes a wait, with a limit, for the last ones."""
    name, loops = kernel
    first, second = MMAS[name]
    issuers = [x for x in loops if "mma_commit(" in x[0]]
    assert len(issuers) == 2 and f"bars[{first}" in issuers[0][0] and f"bars[{second}" in issuers[1][0]
    assert waited_for(issuers[0][1]) == first
    released = [x for x in loops if "tm_st16(" in x[0]]
    assert second in (waited_for(issuers[1][1]), *(waited_for(after) for _, after in released))
