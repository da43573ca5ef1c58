"""Kernels launched as programmatic dependents read with coherent loads (by
reading the sources; no GPU).  Such a kernel may be resident while the kernels
before it still write: neither ``__restrict__`` parameters, which let the compiler
use the non-coherent path and move accesses across the wait, nor ld.global.nc."""
import glob
import os
import re

import paper_2404_07183_gb300 as P

CSRC = os.path.join(os.path.dirname(P.__file__), "csrc")


def _code(path):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)


def _kernels(code):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s+)?(\w+)\s*\(", code):
        at, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(code[at], 0)
            at += 1
        params = code[m.end():at - 1]
        start = at = code.index("{", at)
        depth = 0
        while True:
            depth += {"{": 1, "}": -1}.get(code[at], 0)
            at += 1
            if not depth:
                break
        yield m.group(1), params, code[start:at]


def test_chained_kernels_read_coherently():
    chained, bad = set(), []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = _code(path)
        found = [(n, p) for n, p, body in _kernels(code) if re.search(r"\bchain_(start|wait)\(", body)]
        chained.update(n for n, _ in found)
        bad += [f"{os.path.basename(path)}: {n} takes a __restrict__ parameter"
                for n, p in found if "__restrict__" in p]
        if found and re.search(r"global\.nc|__ldg\(", code):
            bad.append(f"{os.path.basename(path)}: non-coherent load")
    assert {"walk_kernel", "validate_kernel", "pack_keyed_kernel", "radix_pass_kernel",
            "rank_write_kernel", "sort_small_kernel", "init_header_kernel"} <= chained
    assert not bad, bad
