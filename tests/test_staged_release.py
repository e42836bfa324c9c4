"""Orderings that no test could provoke reliably, read from the sources (no GPU).

The consumer warps of the staged kernels read a ring stage and then arrive on
its "empty" barrier, after which a bulk copy may overwrite it.  The arrival,
made by one lane, releases that lane's reads; the other lanes' are ordered
before it by __syncwarp() alone.  Reading the sources is the only way to check
this without provoking the race: every arrival of a warp must go through
mbar_arrive_warp(), and that function must order the lanes first."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1309_1894_gb300", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*", "", f.read())


def test_warps_arrive_through_the_ordered_form_only():
    plain = {name: len(re.findall(r"\bmbar_arrive\(", text)) for name, text in sources()}
    # its definition, and the one call of mbar_arrive_warp()
    assert {n: c for n, c in plain.items() if c} == {"bulk.cuh": 2}


def test_the_ordered_form_synchronises_the_warp_before_it_arrives():
    text = dict(sources())["bulk.cuh"]
    body = re.search(r"void mbar_arrive_warp\([^)]*\)\s*{(.*?)\n}", text, re.S).group(1)
    assert re.fullmatch(r"\s*__syncwarp\(\);\s*if \(lane == 0\) mbar_arrive\(bar\);\s*", body)


def test_every_consumed_stage_is_released():
    used = {name: re.findall(r"mbar_arrive_warp\(smem_addr\(&(\w+)\[", text) for name, text in sources()}
    assert {n: sorted(u) for n, u in used.items() if u} == {
        "vecops.cu": ["empty"], "reduce.cu": ["empty", "xempty", "xfull"]}


def test_cluster_barriers_bring_the_warp_together_first():
    """The aligned cluster barrier is undefined for a warp that is not converged;
    one thread of a block stores its value just before it."""
    plain = {name: len(re.findall(r"barrier\.cluster\.", text)) for name, text in sources()}
    assert {n: c for n, c in plain.items() if c} == {"cluster.cuh": 2}
    text = dict(sources())["cluster.cuh"]
    assert len(re.findall(r'__syncwarp\(\);\s*asm volatile\("barrier\.cluster\.', text)) == 2
