"""Rules for the kernels that may be scheduled while their predecessor still runs, read from the sources (no GPU needed).

A kernel that waits for its predecessor (chain, chain_wait) begins before the data it reads is complete.  The read-only
load path requires data that is constant while the kernel runs, and the compiler may hoist a load through a restrict
pointer over the wait: neither is allowed there.  A kernel launched with the overlap attribute has to wait.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1511_08486_b200", "csrc")


def _sources():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        yield os.path.basename(f), re.sub(r"//[^\n]*", "", open(f).read())


def _kernels(text):
    """(name, parameters, body) of every kernel definition."""
    def close(at, pair):
        depth = 0
        while True:
            depth += (text[at] == pair[0]) - (text[at] == pair[1])
            at += 1
            if depth == 0:
                return at

    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", text):
        end = close(m.end() - 1, "()")
        start = text.index("{", end)
        yield m.group(1), text[m.end():end - 1], text[start:close(start, "{}")]


def test_chained_kernels_read_through_ordinary_loads():
    seen = 0
    for f, text in _sources():
        for name, params, body in _kernels(text):
            if re.search(r"\bchain(_wait)?\(\)", body):
                seen += 1
                assert "__restrict__" not in params + body, f"{f}: {name}"
                assert "__ldg" not in body and ".nc" not in body, f"{f}: {name}"
    assert seen >= 20


def test_kernels_launched_with_the_overlap_wait():
    waits, names, launched = set(), set(), set()
    for _, text in _sources():
        found = list(_kernels(text))
        names |= {n for n, _, _ in found}
        waits |= {n for n, _, b in found if re.search(r"\bchain(_wait)?\(\)", b)}
        # named in the launch itself, or handed to it as `kernel`
        launched |= set(re.findall(r"(?:launch_chained|\bgo)\((\w+)", text))
        launched |= set(re.findall(r"cudaLaunchKernelEx\(&\w+, (\w+)", text)) | set(re.findall(r"auto kernel = (\w+)", text))
    launched &= names
    assert len(launched) >= 20 and launched <= waits, launched - waits
