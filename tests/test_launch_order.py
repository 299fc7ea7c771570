"""Kernels launched while their predecessor still runs (programmatic dependent
launch) may not touch global memory before they have waited for it: not even
data of an earlier kernel, which need not have finished either.  Read off the
sources: ahead of the wait, no load, copy, prefetch or store and no subscript of
a pointer argument."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_01372_gb300", "csrc")
ACCESS = re.compile(r"\b(cp_async|prefetch_l2|__ld\w+|__st\w+|ld_\w+|bulk_g2s)\s*[<(]")


def kernels():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__.*?\b(k_\w+)\(([^{;]*)\)\s*\{", text, re.S):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            body = text[m.end():end]
            if "pdl_wait()" in body or "pdl_start_next()" in body:
                found.append((m.group(1), m.group(2), body))
    return found


def test_there_are_such_kernels():
    assert {"k_fa", "k_fb", "k_fc"} <= {name for name, _, _ in kernels()}


@pytest.mark.parametrize("name,args,body", kernels(), ids=lambda v: v if len(v) < 12 else "")
def test_nothing_is_touched_before_the_wait(name, args, body):
    assert "pdl_wait()" in body
    head = body[:body.index("pdl_wait()")]
    assert not ACCESS.search(head), name
    for a in args.split(","):
        if "*" in a:
            p = re.search(r"(\w+)\s*$", a).group(1)
            assert not re.search(r"\b%s\s*\[" % p, head), (name, p)
