"""Sources of the kernels that may be launched programmatically (launch_chain): such a kernel
comes up while the one before it still writes, and what it waits for is promised to ordinary
accesses only, so none of its loads may take the read-only path.  The instances that do take it
are launched by launch_alone only."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_18437_gb300", "csrc")


def code():
    text = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            text[os.path.basename(path)] = re.sub(r"//[^\n]*", "", f.read())
    return text


def test_programmatic_kernels_make_no_read_only_loads():
    src = code()
    whole = "\n".join(src.values())
    calls = re.findall(r"launch_chain\(([^;]*);", whole)
    kernels = {k for c in calls for k in re.findall(r"\bk_\w+", c)}
    assert {"k_scan", "k_scatter", "k_p2g", "k_grid", "k_g2p", "k_g2p_vc", "k_g2p_adj", "k_p2g_adj"} <= kernels
    for name in sorted(kernels):
        heads = re.findall(r"__global__[^;{]*?\b%s\s*\(([^)]*)\)\s*\{" % name, whole)
        assert heads, name
        for args in heads:
            assert "__restrict__" not in args, name
    # the one read-only load of the device code that they share, and of their own, has an ordinary twin ...
    shared = "\n".join(src[f] for f in ("mpm_transfer.cuh", "mpm_device.cuh", "mpm_kernels.cu", "mpm_adjoint.cu"))
    assert re.findall(r"[^;\n]*__ldg\s*\([^;]*;", shared) == re.findall(r"[^;\n]*READ_ONLY \? __ldg\(at\) : \*at;", shared)
    assert not re.search(r"ld\.(weak\.)?global\.nc", shared)
    # ... and the instances with the read-only one are not launched programmatically
    for c in calls:
        assert "RO" not in re.findall(r"\w+", c) and "kG2PReadOnly" not in c, c
        for name in ("k_g2p_vc", "k_g2p_adj", "k_p2g_adj"):
            assert not re.search(name + r"(?!\w)(?!<false>)", c), c
