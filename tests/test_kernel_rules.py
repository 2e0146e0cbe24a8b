"""Rules that the kernels' sources keep, read from the sources themselves
(breaking one would race or hang on the device, so no test shows it there)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_02930_gb300", "csrc")


def sources():
    out = {}
    for fn in sorted(os.listdir(CSRC)):
        if fn.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(CSRC, fn)) as f:
                out[fn] = re.sub(r"//[^\n]*", "", f.read())
    return out


def test_named_barriers_take_diverged_warps():
    """Named barriers follow branches that single lanes take.  The aligned forms
    (bar.sync, bar.arrive, barrier.*.aligned) need a converged warp, so only
    the others are written, each behind a __syncwarp()."""
    used = 0
    for fn, src in sources().items():
        assert not re.search(r'"\s*bar\.(cta\.)?(sync|arrive|red)', src), fn
        assert not re.search(r"barrier\.[\w.]*aligned", src), fn
        for m in re.finditer(r"barrier\.cta\.(sync|arrive) ", src):
            used += 1
            assert "__syncwarp();" in src[:m.start()].rsplit("{", 1)[1], fn
    assert used == 2
