"""Kernels launched with programmatic stream serialisation start before their
predecessor has ended, so what that writes is not constant over their lifetime:
read-only loads (__ldg, const __restrict__ parameters) are for tables filled at
setup alone.  Checked on the sources that hold or are included by such kernels."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15253_gb300", "csrc")
SOURCES = ["common.cuh", "conv_lane.cuh", "demag.cu", "fft_ct.cuh", "fft_direct.cuh", "fft_lane.cuh", "fft_rt.cuh",
           "field.cu", "field_cells.cuh", "field_dev.cuh", "field_fine_d.cu", "field_x.cuh", "integrate.cu", "lane_x.cuh"]
# twiddles, tensor spectrum, per-region tables, the per-cell strain
TABLES = re.compile(r"^&?\(?(a\.)?(tw|khat|K[012]?|cpair|lut|strain_cell)\b")


def _kernels(text):
    """(name, parameters, body) of the kernels of a source."""
    text = re.sub(r"__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)", "", text)
    for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\(", text):
        i = m.end()
        j = text.index(")", i)
        yield m.group(1), text[i:j], text[j:text.find("\n}", j)]


def test_every_source_with_a_waiting_kernel_is_listed():
    have = {f for f in os.listdir(CSRC) if "dep_wait()" in open(os.path.join(CSRC, f)).read()}
    assert have - {"launch.h"} <= set(SOURCES)


def test_read_only_loads_are_for_tables():
    bad = []
    for f in SOURCES:
        text = open(os.path.join(CSRC, f)).read()
        bad += [(f, a) for a in re.findall(r"__ldg\(([^;]{0,40})", text) if not TABLES.match(a)]
    assert not bad


def test_waiting_kernels_have_no_read_only_parameters():
    seen = 0
    for f in SOURCES:
        for name, params, body in _kernels(open(os.path.join(CSRC, f)).read()):
            if "dep_wait()" in body:
                seen += 1
                assert "__restrict__" not in params, (f, name)
    assert seen >= 20
