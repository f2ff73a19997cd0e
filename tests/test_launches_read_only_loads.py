"""Loads through the read-only path (`__ldg`, `ld.global.nc`, a `const __restrict__` parameter) ask that nothing writes the memory while
the kernel runs. A kernel that may begin while the one ahead of it in the stream still runs (`launch_after` with anything but
`false` first) runs beside that one's writes, so it has no such load."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_07114_b200", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _functions(text):
    """(head, head and body) of every function: from a blank line or the start of a declaration to the brace that closes it."""
    for m in re.finditer(r"^[^\s#}/][^;{}]*\)\s*(?:const\s*)?\{", text, flags=re.M):
        depth, at = 1, m.end()
        while depth and at < len(text):
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        yield m.group(0), text[m.start():at]


def test_kernels_that_begin_early_have_no_read_only_loads():
    read_only = set()
    for name in os.listdir(CSRC):
        if name.endswith((".cuh", ".cu")):
            for head, body in _functions(_source(name)):
                kernel = re.search(r"__global__.*?\b(\w+)\s*\(const", head, flags=re.S)
                if kernel and re.search(r"__ldg|ld\.global\.nc|__restrict__", body):
                    read_only.add(kernel.group(1))
    assert {"drift_pairwise_kernel", "drift_finalize_kernel"} <= read_only            # (the two that have them today: the search finds them)
    early = 0
    for head, body in _functions(_source("lossy_api.cu")):
        for m in re.finditer(r"launch_after\(\s*([^,]+),", body):
            if m.group(1).strip() in ("false", "bool early"):
                continue
            early += 1
            rest = body if "auto kern" in body else body[m.start():m.start() + 600]
            assert not [k for k in read_only if re.search(r"\b%s\b" % k, rest)], (head, m.group(1))
    assert early >= 4
