"""What overlapped launches demand of the kernel sources: a kernel may be
resident while the kernel before it still writes, so it reads such data neither
through the read-only path nor before its wait."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_22541_gb300", "csrc")
# written before a handle is returned and not again: router weights, its bias, FP8 block scales
CONSTANT = {"wr", "bias", "bs_lo", "bs_hi"}


def _sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*", "", f.read())


def _kernels():
    """(file, name, parameters and body) of every __global__ function."""
    for name, text in _sources():
        for m in re.finditer(r"__global__", text):
            start = text.index("{", m.start())
            depth, end = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            head = re.sub(r"__(launch_bounds|cluster_dims)__\((?:[^()]|\([^()]*\))*\)", "", text[m.start():start])
            yield name, re.search(r"(\w+)\s*\(", head).group(1), head, text[start:end]


def test_read_only_loads_are_of_constant_data():
    bad = []
    for name, text in _sources():
        for m in re.finditer(r"__ldg\(\s*([\w.\->]+)", text):
            if m.group(1) not in CONSTANT:
                bad.append((name, m.group(0)))
    assert not bad, bad


def test_no_restricted_input_of_a_dependent_kernel():
    bad = []
    for name, kernel, head, body in _kernels():
        if "pdl_wait" in body:
            bad += [(name, kernel, p) for p in re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", head + body)
                    if p not in CONSTANT]
    for name, text in _sources():  # the device functions they call
        bad += [(name, f, p) for f, args in re.findall(r"__device__ __forceinline__ \w+ (\w+)\(([^)]*)\)", text)
                for p in re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", args)]
    assert not bad, bad


def test_every_dependent_kernel_waits_before_it_leaves():
    """A kernel that left without its wait would let the next one start before
    the kernel in front of both has completed."""
    launched = set()
    for _, text in _sources():
        launched |= set(re.findall(r"launch_pdl\((\w+)", text))
    seen = set()
    for name, kernel, _, body in _kernels():
        if kernel not in launched:
            assert "pdl_wait" not in body, (name, kernel)
            continue
        seen.add(kernel)
        assert "pdl_wait()" in body, (name, kernel)
        first = re.search(r"\breturn\b", re.sub(r"\[&\]\([^)]*\)[^{]*\{[^}]*\}", "", body))
        stripped = re.sub(r"\[&\]\([^)]*\)[^{]*\{[^}]*\}", "", body)
        assert first is None or stripped.index("pdl_wait()") < first.start(), (name, kernel)
    assert seen == launched and len(seen) >= 12, (seen, launched)
