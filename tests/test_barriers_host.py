"""Barriers written as inline PTX (csrc): none but those of the tensor instructions asks for a converged warp.

The `.aligned` forms of the barrier instructions are defined only when all lanes of a warp execute them
together.  The compiler does not know that of an asm statement, and the kernels reach their barriers
after code that lanes leave apart (one lane's finalisation, a grid-stride loop's last round), where a warp
that has not come together again would wait for ever."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1311_5029_gb300", "csrc")


def test_inline_barriers_do_not_need_a_converged_warp():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        for op in re.findall(r"\b(?:barrier\.cluster\.\w+|barrier\.sync|barrier\.arrive|bar\.sync|bar\.arrive)[\w.]*", open(path).read()):
            found += 1
            # bar.sync and bar.arrive are barrier.sync.aligned and barrier.arrive.aligned
            assert ".aligned" not in op and not op.startswith("bar."), (os.path.basename(path), op)
    assert found >= 3
