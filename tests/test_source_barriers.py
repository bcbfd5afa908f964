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


def test_copies_in_flight_are_waited_for():
    """cp.async.wait_group waits for committed groups only; copies that are counted on an mbarrier belong to none.  Who issues copies that way
    ends with cp.async.wait_all."""
    everything = {name: code(name) for name in os.listdir(build.CSRC)}
    commits = any("cp.async.commit_group" in text for text in everything.values())
    assert commits or not any("cp.async.wait_group" in text for text in everything.values())
    for name, text in everything.items():
        if "cp_async_arrive(" in text and name != "sm100_ptx.cuh":
            assert text.rindex("cp_async_wait_all()") > text.rindex("cp_async_arrive("), name
