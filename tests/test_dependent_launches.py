"""Every kernel that may be launched as a dependent of the one before it waits for
that one first: a forgotten dependency_sync is a race on all earlier output that
no run has to show. Read from the sources: a kernel either begins with the wait,
or is launched by <<< >>> wherever it is named."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_19140_gb300", "csrc")
KERNEL = re.compile(r"__global__\s+void\s*(?:__launch_bounds__\s*(\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\))\s*)?(k_\w+)\s*\(")


def _sources():
    out = {}
    for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        s = re.sub(r"/\*.*?\*/", "", open(p).read(), flags=re.S)
        out[os.path.basename(p)] = re.sub(r"//[^\n]*", "", s)
    return out


def _first_statement(src, at):
    """The first statement of the body of the function whose parameter list starts at `at`."""
    depth = 0
    while True:
        depth += {"(": 1, ")": -1}.get(src[at], 0)
        at += 1
        if depth == 0:
            break
    assert src[at:].lstrip().startswith("{")
    return src[at:].lstrip()[1:].lstrip().split(";")[0]


def _offenders(sources):
    kernels, bad = 0, []
    for name, src in sources.items():
        for m in KERNEL.finditer(src):
            kernels += 1
            if _first_statement(src, m.end() - 1).startswith("dependency_sync("):
                continue
            k = m.group(2)
            for use in re.finditer(r"\b%s\b" % k, src):
                if use.start() == m.start(2):
                    continue
                rest = re.sub(r"^<[^<>]*>", "", src[use.end():].lstrip())
                if not rest.lstrip().startswith("<<<"):
                    bad.append("%s: %s" % (name, k))
    return kernels, bad


def test_every_dependent_kernel_waits_first():
    sources = _sources()
    kernels, bad = _offenders(sources)
    assert kernels == sum(s.count("__global__") for s in sources.values()) and kernels > 20
    assert not bad, bad


def test_a_forgotten_wait_is_found():
    for name, kernel in (("dup.cu", "k_ranges_search"), ("dup.cu", "k_dup_write"), ("sort.cu", "k_sweep"),
                         ("blend_fwd.cu", "k_blend_fwd_gauss"), ("project.cu", "k_project")):
        src = _sources()[name]
        at = src.index("dependency_sync(", src.index("%s(" % kernel))
        _, bad = _offenders({name: src[:at] + src[src.index(";", at) + 1:]})
        assert "%s: %s" % (name, kernel) in bad
