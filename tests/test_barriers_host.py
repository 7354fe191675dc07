"""Named barriers of the kernels, read from the source: bar.sync and bar.red are the .aligned forms, whose
behaviour is undefined where the lanes of a warp have not reconverged; every one here follows per-lane code, so
each has to come directly after a __syncwarp() (or be the form without .aligned)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1609_06634_gb300", "csrc")


def test_named_barriers_do_not_assume_converged_warps():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\bbar\.(cta\.)?(sync|red|arrive)\b|\bbarrier\.(cta\.)?(sync|red|arrive)\S*\.aligned", code):
            before = code[:code.rindex("asm volatile", 0, m.start())].rstrip()
            assert before.endswith("__syncwarp();"), (path, m.group(0))
            found += 1
    assert found == 3   # the scoring groups' barrier and the two of the tensor-core epilogue
