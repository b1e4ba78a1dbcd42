"""The sources that retire a kernel's committed ncu counters (bench.KERNEL_SOURCES):
every header that a listed source includes is listed too, so that a change of any of
them retires the counters.  (individual.cuh is included by the units hydro_f32.cu and
hydro_f64.cu only to be compiled there; no profiled kernel is in it.)"""
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_included_headers_are_listed():
    sys.path.insert(0, ROOT)
    import bench
    d = os.path.join(ROOT, "paper_0901_4107_gb300", "csrc")
    for kernel, sources in bench.KERNEL_SOURCES.items():
        names = {os.path.basename(s) for s in sources}
        for s in sources:
            with open(os.path.join(d, s), encoding="utf-8") as f:
                inc = set(re.findall(r'(?m)^#include "([^"]+)"', f.read())) - {"individual.cuh"}
            assert inc <= names, (kernel, s, inc - names)
