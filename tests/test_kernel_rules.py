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


def test_dependent_launches_keep_their_rule():
    """Kernels launched dependently (launch_after) wait for the kernel before them
    in every thread, and no kernel parameter that points to memory a kernel of
    the step writes is declared restrict: a read-only load of it could move
    above the wait.  Porosity and the fixed temperature are constants."""
    text = "\n".join(sources().values())
    kernels = set(re.findall(r"launch_after\(\s*(k_\w+)", text))
    for m in re.finditer(r"launch_after\(\s*kern\b", text):        # the kernel named just before
        kernels |= set(re.findall(r"\bk_\w+(?=<)", text[:m.start()].rsplit("auto kern", 1)[1]))
    assert {"k_split2d", "k_tile2d", "k_march2d", "k_collide3", "k_adj_macro"} <= kernels
    for k in sorted(kernels):
        m = re.search(r"__global__[^;{]*?\b%s\((.*?)\)\s*\{" % k, text, re.S)
        assert m, k
        assert "after_previous();" in text[m.end():].split("__global__", 1)[0], k
        for arg in re.findall(r"__restrict__\s+(\w+)", m.group(1)):
            assert arg in ("phi",), (k, arg)
    for s in ("StepArgs", "AdjArgs", "ReactArgs"):
        body = re.search(r"struct %s \{(.*?)\n\};" % s, text, re.S).group(1)
        for arg in re.findall(r"__restrict__\s+(\w+)", body):
            assert arg in ("phi", "Tfix"), (s, arg)
