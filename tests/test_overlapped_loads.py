"""A step's blocks may be resident while the step before still writes the
records they will read, so those are not read-only for the life of the
kernel, as __ldg (ld.global.nc) asks.  Read from the sources: the only such
loads of the 2-D step kernels are of the network's weights, which no step
writes."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2302_09883_gb300", "csrc")


def test_records_are_not_read_by_non_coherent_loads():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "patch2d.cuh")).read())
    loads = re.findall(r"(?:__ldg|ldg_u32)\(([^;]*)\);", text)
    assert loads and all("src4" in e or "mlp_wt" in e for e in loads), loads
    assert re.search(r"src4 = reinterpret_cast<const float4\*>\(a\.mlp_wt\)", text)
    assert "ld.global.nc" not in text
