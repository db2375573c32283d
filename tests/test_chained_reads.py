"""Kernels of a chain (programmatic dependent launch) start while the launch before them still
writes their inputs. What that launch writes (z, d, the partial u) may be read only by
ordinary loads or TMA after the wait: the read-only path (__ldg, ld.global.nc) and
`const ... __restrict__` promise data that nothing writes during the kernel. Checked on the
source, since a violation shows as a rare wrong value at most.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2401_12890_gb300", "csrc")
STATE = r"(?:Zin|Din|Uin|Pin|zrow|zr|din|pt)"       # pointers to the previous launch's output


def _chained_sources():
    out = []
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(f).read())
        if "pdl_wait();" in text:
            out.append((os.path.basename(f), text))
    return out


def test_chained_kernels_read_state_by_ordinary_loads():
    sources = _chained_sources()
    assert {"ssm_tc.cu", "ssm_lowrank.cuh", "ssm_lowrank_tc.cu", "ssm_table.cu"} <= \
        {name for name, _ in sources}
    for name, text in sources:
        text = text.replace("a.labels", "").replace("P.labels", "")
        bad = re.findall(rf"__ldg\(\s*(?:a\.|P\.)?{STATE}\b[^;]*;", text)
        bad += re.findall(rf"const float\s*\*\s*__restrict__\s+{STATE}\b[^;]*;", text)
        assert not bad, (name, bad)
