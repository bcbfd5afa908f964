"""Rules of the kernels' synchronisation that no run breaks visibly: shown on the source."""
import os
import re

from paper_2609_36938_b200 import build


def code(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_aligned_cluster_barriers_follow_a_reconvergence():
    """barrier.cluster.*.aligned is executed by a whole warp: the wrappers bring its lanes together, whatever branch precedes the call."""
    aligned = re.compile(r"barrier\.cluster\.\w+[\w.]*\.aligned")
    wrappers = 0
    for name in sorted(os.listdir(build.CSRC)):
        text = code(name)
        if name != "sm100_ptx.cuh":
            assert not aligned.search(text), name
            continue
        for body in re.findall(r"__forceinline__ void \w+\([^)]*\)\s*\{(.*?)\n?\}\n", text, re.S):
            m = aligned.search(body)
            if m:
                wrappers += 1
                assert "__syncwarp();" in body[:m.start()], body
    assert wrappers == len(re.findall(r"void cluster_(?:sync_all|arrive|arrive_release|wait)\(", code("sm100_ptx.cuh"))) == 4
