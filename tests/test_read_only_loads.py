"""The read-only load path is for arrays that no thread of a launch writes.  Batches in persistent mode run all kernel bodies of
a stage in one launch, so the bodies take it for the setup's arrays only, and for the stage's through ld_stage."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_04514_gb300", "csrc")


def test_stage_arrays_are_not_read_as_constants():
    setup = {"col", "mu", "MKinv"}  # members of Dev that kernel bodies read so
    for path in sorted(glob.glob(os.path.join(CSRC, "kernels_*.cu"))):
        src = open(path).read()
        local = {m[0]: m[1] for m in re.findall(r"const \w+(?: \w+)?\* (\w+) = D\.(\w+)", src)}  # pointers into such an array
        for arg in re.findall(r"__ldg\(([^;]*?)\)", src):
            name = re.match(r"(D\.)?(\w+)", arg)
            assert (name[2] if name[1] else local.get(name[2])) in setup, (os.path.basename(path), arg)


def test_every_source_says_whether_the_launch_writes_the_stage():
    internal = open(os.path.join(CSRC, "gdg_internal.cuh")).read()
    persistent = open(os.path.join(CSRC, "persistent.cu")).read()
    assert re.search(r"struct One \{[^}]*kSameLaunch = false", internal) and re.search(r"struct Many \{[^}]*kSameLaunch = false", internal)
    assert re.search(r"struct Virt \{[^}]*kSameLaunch = true", persistent)
