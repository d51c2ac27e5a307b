"""Non-coherent loads (ld.global.nc: __ldg, const __restrict__ parameters) are
defined only for memory that nothing writes while the kernel is resident. A
kernel launched with programmatic dependent launch is resident while its
predecessors still write, so in the sources of such kernels only the plan's
constant tables may be read that way."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_28183_gb300", "csrc")
CODE = {os.path.basename(f): re.sub(r"//[^\n]*", "", open(f).read())
        for f in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))}
# files whose functions run inside chained kernels (they wait for the kernel
# before, or are included by files that do)
CHAINED = sorted(n for n, t in CODE.items() if "pdl_wait()" in t or n.endswith(".cuh"))
# plan tables: twiddles (whole table, a pass's part of it) and band weights
TABLES = re.compile(r"^(tw_src|tp|tl|w|p\.w)\b")
# `g`: the shared spectrum, read by pf_band_spectrum_kernel alone, which is
# launched plainly (after its producer has ended)
PLAIN = {("pf_kernels.cu", "g + l")}


@pytest.mark.parametrize("name", CHAINED)
def test_noncoherent_loads_read_plan_tables_only(name):
    for m in re.finditer(r"__ldg\s*\(([^;]*?)\)", CODE[name]):
        arg = m.group(1).strip()
        assert TABLES.match(arg) or (name, arg) in PLAIN, f"{name}: __ldg({arg})"
    assert "__restrict__" not in CODE[name]
    assert "ld.global.nc" not in CODE[name]


def test_shared_spectrum_kernel_is_launched_plainly():
    text = CODE["pf_kernels.cu"]
    body = text[text.index("static cudaError_t launch_spec_one"):]
    body = body[:body.index("\n}\n")]
    assert "<<<" in body and "launch_kernel" not in body
