"""Kernels launched so that they start before the kernel in front of them has ended
must not read its output through the read-only path (__ldg, or const T*
__restrict__ parameters): that path takes the memory as constant while the kernel
runs.  Checked on the sources; a race would show only now and then."""
import glob
import os
import re

# parameters that no kernel writes: uploaded by the host before any launch
CONSTANT = {"steps", "leaf_store", "leaves", "store", "descs", "perm"}


def _sources():
    from paper_2110_14502_gb300 import build as B
    for path in sorted(glob.glob(os.path.join(B.CSRC, "*.cu")) + glob.glob(os.path.join(B.CSRC, "*.h"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*", "", f.read())


def _span(text, at, left, right):
    """Index past the bracket that closes the first `left` at or after `at`."""
    i = text.index(left, at)
    depth = 0
    while True:
        depth += (text[i] == left) - (text[i] == right)
        i += 1
        if depth == 0:
            return i


def _kernels(text):
    """(name, parameter list, whole definition) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\b", text):
        at = m.end()
        while True:  # attributes such as __launch_bounds__(...) come before the name
            n = re.compile(r"\s*(\w+)").match(text, at)
            end = _span(text, n.end(), "(", ")")
            if not n.group(1).startswith("__"):
                break
            at = end
        yield n.group(1), text[n.end():end], text[m.start():_span(text, end, "{", "}")]


def test_no_read_only_loads_of_earlier_kernels_output():
    sources = dict(_sources())
    launched = set()
    for text in sources.values():
        launched |= set(re.findall(r"launch_overlapped\(\s*(\w+)", text))
    launched -= {"void"}  # its own declaration
    assert {"chain_kernel", "split_kernel", "gemm_simt_kernel", "vector_tile_kernel", "gemm_direct"} <= launched, launched
    seen, bad = set(), []
    for name, text in sources.items():
        if not any(k in launched for k, _, _ in _kernels(text)):
            continue
        rest = text
        for kernel, params, body in _kernels(text):
            if kernel not in launched:
                rest = rest.replace(body, "")
                continue
            seen.add(kernel)
            for p in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params):
                if p not in CONSTANT:
                    bad.append(f"{name}: {kernel}: parameter {p}")
        bad += [f"{name}: __ldg"] * rest.count("__ldg(")
        bad += [f"{name}: helper parameter {p}" for p in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", rest)
                if p not in CONSTANT and not any(f": parameter {p}" in b for b in bad)]
    assert seen == launched, launched - seen
    assert not bad, bad
