"""Loads under a promise of read-only data (__ldg(), `const T* __restrict__`) in the headers that kernels share, which the check of
the kernels' own files does not read.  A kernel that is launched beside its predecessor may make that promise only of what is
complete before its launch (see test_launch_order_sources.py); each load that makes it stands here with its reason, and nothing
stands here that is not in the sources."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_20888_b200", "csrc")

LDG = {
    "eta_attend.cuh": {"q"},               # the query: the interface requires it to be complete before the launch
    "eta_decode.cu": {"a.seq_lens"},       # the lengths likewise
    "eta_predict.cu": {"W"},               # the predictor's weights likewise
    "eta_screen.cu": {"a.seq_lens"},
    "eta_summary.cu": {"base", "p"},       # the build is launched only when everything before it has ended
}
READ_ONLY = {
    "eta_bounds.cuh": {"qw"},              # bound_one's queries, in shared memory behind a barrier
}


def _source(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def _ldg(src):
    return set(re.findall(r"__ldg\((?:reinterpret_cast<[^>]*>\()?([\w.]+)", src))


def _read_only(src):
    return set(re.findall(r"const\s+[\w:]+(?:\s+\w+)?\s*\*\s*__restrict__\s+(\w+)", src))


def test_every_read_only_load_is_known_and_every_known_one_exists():
    found = {os.path.basename(p): _ldg(_source(p)) for p in glob.glob(os.path.join(CSRC, "*.cu*"))}
    assert {name: loads for name, loads in found.items() if loads} == LDG
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert len(re.findall(r"__ldg\(", _source(path))) == len(re.findall(r"__ldg\((?:reinterpret_cast<[^>]*>\()?[\w.]+", _source(path)))


def test_headers_promise_nothing_else():
    found = {os.path.basename(p): _read_only(_source(p)) for p in glob.glob(os.path.join(CSRC, "*.cuh"))}
    assert {name: names for name, names in found.items() if names} == READ_ONLY


def test_the_query_is_read_from_where_the_interface_says():
    """What the early kernels load under the promise is the query argument itself, in both kernels that share the load."""
    for name in ("eta_decode.cu", "eta_step.cu"):
        calls = re.findall(r"\bat\.load_q\(([^;]*)\);", _source(os.path.join(CSRC, name)))
        assert calls and all(c.startswith("a.q + ") for c in calls)
