"""Kernels that may be set up while their predecessor still runs: what their source has to keep to (CPU)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_04123_b200", "csrc")


def sources():
    return {os.path.basename(p): open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}


def chained_kernels():
    """{kernel: (parameters, body)} of every kernel that can be launched through launch_chained."""
    text = "\n".join(sources().values())
    names = set(re.findall(r"launch_(?:chained\(|kernel\([^,()]*,)\s*(\w+_kernel)\b", text))
    found = {}
    for name in names:
        m = re.search(r"__global__[^;{]*?\b" + name + r"\s*\(([^)]*)\)\s*\{(.*?)\n\}", text, re.S)
        assert m, name
        found[name] = m.groups()
    return found


def test_every_chained_kernel_waits_before_anything_else():
    kernels = chained_kernels()
    assert len(kernels) >= 18
    for name, (_, body) in kernels.items():
        assert body.split(";")[0].strip() == "await_predecessor()", name


def test_chained_kernels_read_nothing_but_the_points_as_read_only():
    """A `const __restrict__` pointer lets loads move ahead of the wait: only the points, an input of the call, may be one."""
    for name, (params, _) in chained_kernels().items():
        for p in params.split(","):
            if "__restrict__" in p:
                assert p.split()[-1] == "pts", (name, p.strip())
