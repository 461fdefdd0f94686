"""Which clusters the one-kernel step is launched in, on the CPU: only ones of which the GPU holds as many as there are rows, by its own
answer (a part of a GPU, or groups with fewer SMs, may hold none of a size; the launch would be refused there)."""
import ctypes

from paper_2609_20888_b200 import binding as eb
from paper_2609_20888_b200 import build as ebuild


def test_clusters_that_do_not_fit_are_not_launched():
    """A self-check of the library with made-up devices: the answer is asked for once per (device, kernel), a query that fails
    counts as "none" and is not remembered, and the rule falls back to smaller clusters or to the general path; with a B200's
    answers, problems on either side of the line.  0 = every expectation held."""
    ebuild.build()
    lib = eb.load()
    lib.eta_selftest_cluster_table.restype = ctypes.c_int
    assert lib.eta_selftest_cluster_table() == 0
