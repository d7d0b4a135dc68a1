"""Kernels that are placed before their predecessor has completed (they call
wait_for_predecessor) must not read its output by the read-only path, which is
defined only for data that nothing writes while the kernel lives.  Nothing a
run can show: read from the sources, which arrays of the pass (y: channelised
cube, z: windows, R: covariances, c: weights) enter such a kernel as const
__restrict__ pointers or are read by __ldg there."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_11790_gb300", "csrc")
ARRAYS = "y|z|R|c"
ALIASES = ARRAYS + "|zg|Rg|cg|src|row"   # pointers into them in these files


def _sources():
    return {os.path.basename(p): open(p).read() for p in glob.glob(os.path.join(CSRC, "*.cu*"))}


def _kernels(text):
    """(name, parameters, body) of the kernels of a file."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^{;]*?\)\s*)?\s*(\w+)\s*\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params, body0 = text[m.end():i - 1], text.index("{", i)
        depth, j = 1, body0 + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        yield m.group(1), params, text[body0:j]


def test_predecessors_output_is_not_read_as_read_only():
    found = set()
    for name, text in _sources().items():
        dependent = [(k, p) for k, p, b in _kernels(text) if "wait_for_predecessor()" in b]
        if not dependent and name != "solve_dev.cuh":
            continue
        for k, params in dependent:
            found.add(k)
            for p in params.split(","):
                m = re.match(r"\s*const\s+\w+\s*\*\s*__restrict__\s*(\w+)\s*$", p)
                assert not (m and re.fullmatch(ARRAYS, m.group(1))), f"{name}: {k}: {m.group(1)}"
        bad = re.findall(r"__ldg\(\s*&?\s*(?:wa\.)?(?:%s)\b[^)]*\)" % ALIASES, text)
        assert not bad, f"{name}: {bad}"
    assert found >= {"beamspace_kernel", "beamspace_warp_kernel", "window_cov_kernel", "window_cov_warp_kernel",
                     "window_cov_mma_kernel", "mvdr_solve_w_kernel", "apply_kernel", "apply_blocks_kernel"}
    assert not re.search(r"const\s+double2\s*\*\s*__restrict__\s*Rg", _sources()["solve_dev.cuh"])
