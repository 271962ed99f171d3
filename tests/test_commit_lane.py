"""tcgen05.commit follows the MMAs of the thread that issues it, so a kernel's last commit (`drain`, which the
teardown waits for before tensor and shared memory are released) must come from the lane that issued its MMAs: where
those are issued under elect_one(), by lane 0 it would complete at once. Checked in the sources (the lane that
elect.sync names is the hardware's choice, so running a kernel does not show the difference)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_19528_gb300", "csrc")


def issuers(text):
    """The conditions under which MMAs are issued and under which `drain` is committed: the nearest choice of a lane
    before each."""
    text = re.sub(r"//[^\n]*", "", text)

    def lane(pos):
        return [m.group(0) for m in re.finditer(r"elect_one\(\)|lane == 0", text[:pos])][-1]

    mmas = {lane(m.start()) for m in re.finditer(r"\bumma_bf16(_pair)?\(", text)}
    drains = {lane(m.start()) for m in re.finditer(r"\bumma_commit\w*\(smem_u32\(&ctl->drain\)", text)}
    return mmas, drains


def test_the_lane_that_issues_the_mmas_commits_the_drain():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        with open(path) as f:
            mmas, drains = issuers(f.read())
        if mmas:
            seen += 1
            assert len(mmas) == 1 and drains == mmas, (os.path.basename(path), mmas, drains)
    assert seen >= 4
