"""Kernels launched programmatically dependent on their predecessor (`pass` in af_stage.cuh) run
beside it: each must wait (pass_begin) before it touches memory, and none may read the stage's arrays
through the read-only path, whose data must not change while the kernel lives.  None starts its
successor early either: blocks that wait hold the SMs against the point list on the second stream.
Checked on the source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_04857_gb300", "csrc")
FILES = ["af_math.cuh", "af_device.cuh", "af_stage.cuh", "af_kernels1d.cuh", "af_kernels.cu", "af_kernels_lat.cu"]


def code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_no_read_only_loads():
    for name in FILES:
        assert not re.search(r"__ldg|\bld\.global\.nc|__ldcg", code(name)), name


def test_dependent_kernels_wait_first():
    src = "".join(code(f) for f in FILES)
    launched = set(re.findall(r"\b(?:pass|go)\(\s*(k1?_\w+)", src))
    assert {"k_pointdata", "k_points", "k_faces", "k_cells", "k_final", "k1_pointdata"} <= launched
    for k in launched:
        bodies = re.findall(r"__global__[^;{]*?\b%s\([^{]*\)\s*\{\s*([^\n]*)" % k, src)
        assert bodies, k
        for b in bodies:
            assert b.strip() == "pass_begin();", (k, b)


def test_no_early_start():
    assert "launch_dependents" not in "".join(code(f) for f in FILES)


def test_no_build_time_overrides():
    """Tile sizes, lines between forms and launch bounds stand once: a size that a build could change in
    one place and not in the others (the quiet tiles and the blocks of the passes) would skip tiles."""
    for name in sorted(os.listdir(CSRC)):
        if name == "af_internal.h":   # AF_NCOEF, a public constant af.h defines as well
            continue
        assert not re.search(r"#\s*ifn?def\s+AF_(?!LAT\b)", code(name)), name
