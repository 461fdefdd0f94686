"""The kernels that are launched while the kernel before them in the stream may still run (launch_pdl) must not promise the
compiler that what that kernel writes is read-only: a `const T* __restrict__` parameter and __ldg() both do, for the whole
kernel, and a load under that promise may come from a cache that is not kept coherent or be moved above the wait.  Read from
the sources, on the CPU: no run shows it, the promise is simply not one the code can keep.

Excepted is what is complete before the launch: the inputs that the interface requires to be (a query, the lengths, the
predictor's weights), and what an earlier kernel of the same call has waited for before it released its successor."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_20888_b200", "csrc")

READ_ONLY = {
    "predict_threshold_kernel": {"q", "W", "bias"},        # required complete by the interface
    "calib_hist_kernel": {"tau"},                          # calib_clear_kernel has waited for everything before the call
    "build_summaries_kernel": {"K", "seq_lens", "table"},  # launched only when everything before it has ended
}
LDG = {
    "eta_decode.cu": {"a.seq_lens", "qp"},
    "eta_predict.cu": {"W"},
    "eta_screen.cu": {"a.seq_lens"},
    "eta_summary.cu": {"base", "p"},                       # the build (the append takes the other side of FRESH)
}


def _source(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_dependent_launches_make_no_read_only_promise(path):
    src = _source(path)
    for head in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(([^{]*)\)\s*\{", src):
        promised = set(re.findall(r"const\s+[\w:]+(?:\s+\w+)?\s*\*\s*__restrict__\s+(\w+)", head[2]))
        assert promised <= READ_ONLY.get(head[1], set()), head[1]
    for load in re.finditer(r"__ldg\((?:reinterpret_cast<[^>]*>\()?([\w.]+)", src):
        assert load[1] in LDG.get(os.path.basename(path), set()), load[0]


def test_the_patterns_find_what_they_look_for():
    """Every kernel of the sources is seen, and a promise in one of them would be."""
    names = []
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        src = _source(path)
        found = re.findall(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(([^{]*)\)\s*\{", src)
        assert len(found) == src.count("__global__")
        names += [n for n, _ in found]
    assert set(READ_ONLY) <= set(names) and "calib_bisect_kernel" in names and "score_dual_kernel" in names
