"""Every device function of csrc/gdg_internal.cuh is reached by a kernel body, so that what the self-tests run is what the sweeps
run."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_04514_gb300", "csrc")


def test_no_helper_is_left_over():
    src = {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read())
           for p in glob.glob(os.path.join(CSRC, "*.cu*")) if "selftest" not in p}
    names = set(re.findall(r"__device__ (?:__forceinline__|__noinline__)[^;{(]*?\b(\w+)\((?=[^)]*\)\s*(?:const )?\{)",
                           src["gdg_internal.cuh"]))
    assert len(names) > 40
    text = "\n".join(src.values())
    assert not [n for n in sorted(names) if len(re.findall(r"\b%s\b" % n, text)) < 2]
