"""Which global loads of the kernels may be non-coherent.

A kernel of a programmatic-dependent-launch chain is resident while the previous
one still writes the fields it will read. __ldg (ld.global.nc) is specified only
for memory that nobody writes during the kernel's lifetime, so it may load what an
upload wrote (geometry, connectivity, operators), never a field: fields are read
by plain or L2 loads, which griddepcontrol.wait makes coherent."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1211_0582_gb300", "csrc")
# written by uploads and material updates only, which are complete before a stage is launched
STATIC = r"(ops|geo|g|a\.geo|a\.fgeo|a\.fconn|a\.fmat|a\.LF|a\.Dn|a\.DT|a\.LT)\s*(\+|\))"
# kernels that are never launched into a chain: the launch waits for everything before it
UNCHAINED = {"energy.cu", "geometry.cu"}
FILES = sorted(f for ext in ("*.cu", "*.cuh") for f in glob.glob(os.path.join(CSRC, ext))
               if os.path.basename(f) not in UNCHAINED)


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_noncoherent_loads_are_of_static_data(path):
    src = re.sub(r"//[^\n]*", "", open(path).read())
    bad = []
    for m in re.finditer(r"\b(__ldg|ldg4)\s*\(", src):
        arg = src[m.end():]
        if re.match(r"const float \*p\)", arg) or re.match(r"reinterpret_cast<const float4 \*>\(p\)\)", arg):
            continue  # the helper ldg4 itself
        if not re.match(STATIC, arg):
            bad.append(src[m.start():m.end() + 60].split("\n")[0])
    assert not bad, bad
    assert "ld.global.nc" not in src


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_no_restrict_on_fields(path):
    # a const __restrict__ pointer lets the compiler choose the non-coherent load by itself
    src = re.sub(r"//[^\n]*", "", open(path).read())
    for m in re.finditer(r"const (\w+) \*__restrict__ (\w+)", src):
        assert m.group(2) in ("ops", "stream", "w", "geo", "fgeo", "fconn"), m.group(0)
