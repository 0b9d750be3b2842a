"""The rules of pdl.cuh for kernels that may start before the kernel before them has ended, kept by the sources.

Such a kernel (its body calls pdl_wait) is alive while others still write, so a vector of the running solve may
not be read as constant data: not through __ldg and not through a const __restrict__ parameter.  And it may be
launched so only directly behind a kernel, not behind a copy, a memset or an event wait."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1201_5991_gb300", "csrc")
# pointers to what only the set-up writes: index lists, weights, factors, the explicit coarse inverse
SETUP_PARAMS = {"crow_sub", "rows", "row_sub", "W", "loc2glob", "v32_pos", "part_off", "tasks"}
SETUP_LOADS = {"t", "L.val", "L.col", "L.iface_occ4"}   # t: a factor tile


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        s = _source(os.path.basename(path))
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(([^{]*)\)\s*\{", s):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(s[i], 0)
                i += 1
            yield m.group(1), m.group(2), s[m.end():i]


def test_early_kernels_read_running_vectors_with_ordinary_loads():
    early = [k for k in _kernels() if "pdl_wait()" in k[2]]
    assert len(early) > 12
    for name, params, body in early:
        const = set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params))
        assert const <= SETUP_PARAMS, (name, const - SETUP_PARAMS)
        for load in re.findall(r"__ldg\(\s*(?:\(const \w+\*\))?\s*\(?\s*([\w.]+)", body):
            assert load in SETUP_LOADS, (name, load)


def test_early_launches_follow_kernels():
    s = _source("capi.cpp")
    breaks = ("cudaMemcpyAsync", "cudaMemsetAsync", "cudaStreamWaitEvent")
    stmts = [t for t in re.split(r"[;{}]", s)]
    early = 0
    for i, t in enumerate(stmts):
        if "kAfterKernel" not in t or "launch_" not in t:
            continue
        early += 1
        before = next(b for b in reversed(stmts[:i]) if re.search(r"\w+(<[^()]*>)?\s*\(", b) and "ProfScope" not in b)
        assert not any(b in before for b in breaks), (before, t)
    assert early > 8
    # helpers that are called behind copies and memsets launch plainly unless their caller says otherwise
    v = _source("vector.cu")
    for helper in ("gather_iface", "spmv", "convert", "add_to_double", "axpy"):
        assert not re.search(r"launch_pdl\(k_" + helper + r"\b", v), helper
