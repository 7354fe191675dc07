"""Named barriers of the kernels, read from the source: bar.sync and bar.red are the .aligned forms, whose
behaviour is undefined where the lanes of a warp have not reconverged; every one here follows per-lane code."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1609_06634_gb300", "csrc")


def test_named_barriers_do_not_assume_converged_warps():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"\bbar\.(cta\.)?(sync|red|arrive)\b", code), path
        assert not re.search(r"\bbarrier\.(cta\.)?(sync|red|arrive)\S*\.aligned", code), path
        found += len(re.findall(r"\bbarrier\.(?:sync|red)\b", code))
    assert found >= 3   # the scoring groups' barrier and the two of the tensor-core epilogue
