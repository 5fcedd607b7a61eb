"""The bar.* instructions want every thread of a warp at once: the kernels name
barriers through two helpers that bring the warp together first, and nowhere
else."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1803_00113_gb300", "csrc")
BARRIER = re.compile(r'asm[^;]*?"\s*(?:bar|barrier)(?:\.cta)?\.(sync|arrive|red)\b')


def test_named_barriers_bring_the_warp_together():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        text = open(path).read()
        for m in BARRIER.finditer(text):
            body = text[:m.start()]
            body = body[body.rindex("{"):]           # from the helper's opening brace
            found.append((os.path.basename(path), m.group(1)))
            assert body.split() == ["{", "__syncwarp();"], found[-1]
    assert sorted(found) == [("internal.cuh", "arrive"), ("internal.cuh", "sync")]
