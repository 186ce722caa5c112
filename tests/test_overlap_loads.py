"""Read-only loads in kernels that overlap the launch ahead of them.

A kernel that calls pdl_wait is resident while the kernel before it on the
stream still writes.  ld.global.nc (__ldg, and ld_store, which uses it) is for
memory that nobody writes during the kernel's lifetime, so in such kernels it
may read only what was complete before the launch ahead of them began.  A
stale line would be a wrong field now and then that parity tests can miss, so
the sources are checked: every read-only load in a kernel that waits, or in a
function it calls, is of one of the operands below.  (The iteration kernels'
field loads take their form from a template flag, which a static_assert in
walk_tile ties to the overlapped launch.)
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_25924_gb300", "csrc")

# (function, start of the operand): why it is complete
COMPLETE = {
    ("k_prefilter", "a.w25"): "pre-filter weights",
    ("sample_level", "r"): "level images, once an iteration has run (the first one starts from V0 = 0)",
    ("ldp", "P"): "level images",
    ("bw_samples_walk", "t1"): "level images",
    ("bw_samples_walk", "t2"): "level images",
    ("ld_field", "p"): "the form without COH, see walk_tile",
}
READ_ONLY = re.compile(r"\b(?:__ldg|ld_store|ld_in|ld_raw)\s*\(\s*([^;]*)")
NOT_CALLS = {"if", "constexpr", "for", "while", "switch", "return", "sizeof", "defined"}


def functions():
    """name -> list of bodies, for every function defined in the CUDA sources."""
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            src = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", f.read(), flags=re.S))
        for m in re.finditer(r"\b(\w+)\s*\(", src):
            # a definition: the matching parenthesis is followed by a brace
            i, depth = m.end(), 1
            while i < len(src) and depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            tail = re.match(r"\s*(?:const\s*)?\{", src[i:])
            line = src[src.rfind("\n", 0, m.start()) + 1:m.start()]
            if not tail or m.group(1) in NOT_CALLS or not re.search(r"__global__|__device__|\w[\w:<>,\s\*&]*\s[\*&]?$", line + " "):
                continue
            j, depth = i + tail.end(), 1
            while j < len(src) and depth:
                depth += {"{": 1, "}": -1}.get(src[j], 0)
                j += 1
            out.setdefault(m.group(1), []).append((os.path.basename(path), src[i:j]))
    return out


def test_overlapping_kernels_load_coherently():
    fn = functions()
    kernels = {n for n, bodies in fn.items() if any("pdl_wait()" in b for _, b in bodies)}
    assert {"k_reduce", "k_prefilter", "k_bw_solve", "k_bw_box_tile", "k_bw_samples_walk", "walk_tile"} <= kernels
    reach, todo = set(), set(kernels)
    while todo:
        n = todo.pop()
        reach.add(n)
        for _, body in fn[n]:
            called = set(re.findall(r"\b(\w+)\s*(?:<[^<>;()]*>)?\s*\(", body))
            todo |= {c for c in called & fn.keys() if c not in NOT_CALLS} - reach
    assert {"load7", "bw_samples_walk", "sample_level", "ld_field", "walk_products"} <= reach
    bad = []
    for n in sorted(reach - {"ld_store", "ld_in", "ld_raw"}):
        for path, body in fn[n]:
            for m in READ_ONLY.finditer(body):
                if not any(n == f and m.group(1).startswith(op) for f, op in COMPLETE):
                    bad.append(f"{path} {n}: {m.group(0)[:60]}")
    assert not bad, "\n".join(bad)


def test_chained_iterations_read_fields_past_the_read_only_cache():
    with open(os.path.join(CSRC, "k_walk.cuh")) as f:
        assert "static_assert(COH != LD_READ_ONLY || !CHAIN" in f.read()
