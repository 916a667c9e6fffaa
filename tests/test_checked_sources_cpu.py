"""Every function of the device core that reads populations has its check in
the bounds-checked build: the sources are read as text, function by function."""
import os
import re

CORE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2103_01444_gb300", "csrc", "lbm_core.cuh")

# loads of a population buffer, of the row ring and of the tile
READ = re.compile(r"\b(?:ldp<CG>|ldq<CG>|ld_s|ldq_s)\((?:src\.)?[pd]\b|copy_async<")
WRAPPERS = {"ld_r", "ld_cg", "ld_s", "ldp", "ldq", "ldq_s", "copy_async", "take_interior"}


def functions(text):
    """(name, body) of every device function defined in the text."""
    for m in re.finditer(r"__device__ (?:__forceinline__ )?[^;{}()]*?\b(\w+)\(", text):
        start = text.find("{", m.end())
        end = text.find(";", m.end())
        if start < 0 or 0 <= end < start:
            continue
        depth, k = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            if depth == 0:
                break
            k += 1
        yield m.group(1), text[start:k + 1]


def test_population_reads_are_checked():
    readers = {}
    for name, body in functions(open(CORE).read()):
        if name not in WRAPPERS and READ.search(body):
            readers.setdefault(name, []).append("in_bounds(" in body)
    assert {"at", "group", "load_interior", "request_interior", "load_shared", "load_own"} <= set(readers)
    assert all(all(v) for v in readers.values()), readers
