"""Kernels that may start before their predecessor on the stream has finished
(launch_chained) are resident while it still writes fields, so only data that
nothing writes, the links, goes through the read-only path (__ldg,
ld.global.nc, a const __restrict__ parameter).  Checked on the source text."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1103_5103_gb300", "csrc")


def _sources():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        yield os.path.basename(f), re.sub(r"//[^\n]*", "", open(f).read())


def test_read_only_loads_are_links():
    seen = 0
    for name, src in _sources():
        scope = ""
        for line in src.splitlines():
            m = re.search(r"struct (\w+)|__device__ __forceinline__ \S+ (\w+)\(", line)
            if m:
                # a member function of LinkIO stays in its scope
                scope = m.group(1) or (scope if scope == "LinkIO" and line.startswith("    ") else m.group(2))
            if "__ldg(" in line or "ld.global.nc" in line:
                seen += 1
                assert "link" in (scope + line).lower(), f"{name}: {line.strip()}"
    assert seen > 5


def test_chained_kernels_have_no_restrict_inputs():
    text = "\n".join(src for _, src in _sources())
    chained = set(re.findall(r"launch_chained\(\s*(\w+)", text))
    assert len(chained) > 20
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\(([^)]*)\)", text):
        if m.group(1) in chained:
            assert not re.search(r"const [^,]*__restrict__", m.group(2)), m.group(1)
