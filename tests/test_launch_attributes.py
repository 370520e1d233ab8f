"""Launch rules that hold by the text of the sources.

A kernel's shared-memory limit is an attribute of the kernel on one device: every fas_create sets it, on the device
that is current then. Setting it once per process would leave the kernels of a second device without.

The launchers of the tile, column and sweep kernels return their launch error and clear it, so a caller that drops it
would go on with the results of an earlier launch."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_11152_gb300", "csrc")


def _functions(text):
    """(name, body) of every function whose name ends in _prepare or _attr."""
    for m in re.finditer(r"cudaError_t (\w+_(?:prepare|attr))\(\) \{\n(.*?)\n\}\n", text, re.S):
        yield m.group(1), m.group(2)


def test_limits_are_not_set_once_per_process():
    seen = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        with open(path) as f:
            for name, body in _functions(f.read()):
                seen.add(name)
                assert "call_once" not in body and "static" not in body, name
    assert {"tile2d_prepare", "col3d_prepare", "stream2d_prepare", "ir_strip_prepare", "sweep3d_prepare",
            "coarse_attr"} <= seen
    with open(os.path.join(CSRC, "fas_api.cu")) as f:
        api = f.read()
    create = api[api.index("fas_status fas_create("):api.index("fas_status fas_destroy(")]
    for name in seen - {"pre_attr", "col_attr"}:
        assert name in create, name


def test_launch_errors_are_not_dropped():
    with open(os.path.join(CSRC, "fas_api.cu")) as f:
        api = f.read()
    calls = [m for m in re.finditer(r"\blaunch_(?:tile_\w+|col3d_\w+|stream2d_\w+|sweep3d|ir_strip)(?:<T>)?\(", api)]
    assert len(calls) >= 8
    for m in calls:
        before = api[max(0, m.start() - 40):m.start()]
        assert re.search(r"(launched\(|cudaError_t e\w* =\s*|&&\s*|\be =\s*)$", before), before + m.group(0)
