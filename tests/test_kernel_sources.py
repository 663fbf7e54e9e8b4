"""Rules that every kernel source keeps and that no run can show to be broken."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_04904_gb300", "csrc")


def _sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh", ".h"))}


def test_aligned_barriers_are_reached_by_whole_warps():
    """Cluster barriers and bar.sync are `.aligned`: undefined unless all lanes of a
    warp execute them together.  They stand in tc_common.cuh alone, each behind the
    __syncwarp() that brings together a warp whose lanes left a branch or a polling
    loop one by one."""
    raw = re.compile(r'asm volatile\(\s*"(?:barrier\.cluster|bar\.sync|barrier\.sync)')
    behind = re.compile(r'__syncwarp\(\);\s*asm volatile\(\s*"(?:barrier\.cluster|bar\.sync|barrier\.sync)')
    for name, text in _sources().items():
        if name == "tc_common.cuh":
            assert len(raw.findall(text)) == len(behind.findall(text)) == 3
        else:
            assert not raw.search(text), name
