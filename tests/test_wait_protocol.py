"""The bounded waits of the kernels, read from their source (no GPU: the path
on which a wait gives up runs only when a copy or a product never completes).

* A wait whose outcome steers a warp is the warp form, one answer for all 32
  lanes: shuffles, votes and tensor-memory loads follow it.  The per-thread
  form appears in code that one lane runs, inside a vote, or as a statement
  (its outcome unused).
* A kernel frees its tensor memory only past a wait for its products that the
  abort flag does not cut short.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_19331_gb300", "csrc")


def _source(name):
    s = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", s, flags=re.S))


def _waits(s):
    """(statement up to the call, headers of the enclosing blocks) of every
    per-thread wait outside the helpers that define one."""
    heads, start = [], 0
    for m in re.finditer(r"[{};]|\b(?:wait_phase|mbar_wait|mbar_try_wait)\(", s):
        tok = m.group()
        if tok == "{":
            heads.append(s[start:m.start()].strip())
        elif tok == "}":
            heads.pop()
        if tok in "{};":
            start = m.end()
        elif heads and not any(re.search(r"\bbool (wait_phase|mbar_wait|mbar_try_wait)", h) for h in heads):
            if not s[start:m.start()].strip().endswith("bool"):      # the helper's own head
                yield s[start:m.start()].strip(), heads


def test_waits_that_steer_a_warp_are_uniform():
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        for stmt, heads in _waits(_source(name)):
            seen += 1
            one_lane = any("lane == 0" in h for h in heads)
            vote = "__all_sync(" in stmt
            unused = stmt == "" or re.fullmatch(r"\+\+\w+\)", stmt)
            assert one_lane or vote or unused, (name, stmt)
    assert seen >= 8


def test_tensor_memory_is_freed_past_the_products():
    s = _source("iso_gemm.cu")
    kernels = re.split(r"__global__", s)[1:]
    freeing = [k for k in kernels if "tcgen05.dealloc" in k]
    assert len(freeing) == 3
    for k in freeing:
        before = k[:k.index("tcgen05.dealloc")]
        assert re.search(r"\n\s+mbar_wait\((accum_bar|empty_bar\()", before), k[:120]
        assert before.rindex("__syncthreads") > max(m.start() for m in re.finditer(r"mbar_wait\(", before))
