"""Runs the kernel forms of tests/_forms.py and a gradient with the fallback pass through the bounds-checked
library and prints the index-violation report as one JSON line.  Started by
tests/test_gpu_debug_bounds_forms.py in a child process with LISA_DEBUG_BOUNDS=1."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

from paper_2507_06300_gb300 import binding as B  # noqa: E402
from paper_2507_06300_gb300 import synth  # noqa: E402
from tests import _forms  # noqa: E402
from tests._workloads import gpu_eval, oracle_dataset  # noqa: E402
from tests.test_gpu_grad import gpu_grad  # noqa: E402


def main():
    assert B.debug_requested(), "LISA_DEBUG_BOUNDS=1 must be set"
    B.debug_bounds(reset=True)
    finite = True
    for n_bins, n_states in ((1, 65), (66, 128), (577, 129)):
        wl, P = _forms.chunk_workload(n_bins, n_states, 3, 1)
        L, St = gpu_eval(wl, P, 0)
        L2, _ = _forms.eval_beside(wl, P)
        finite &= bool(np.array_equal(L, L2))
    for n_bins, n_states in ((2, 65), (130, 129), (1025, 66)):
        wl, P9 = _forms.dense_workload(n_bins, n_states, 1)
        for sc in (128, 64):
            L, St = _forms.dense_eval(wl, P9, sc)
            finite &= bool(np.all(np.isfinite(L[St == 0])))
    for n_bins, n_states in ((129, 320), (2049, 90)):
        wl = synth.workload("tiny", n_bins=n_bins, n_states=n_states, kmin=0, kmax_draw=8)
        wl.knots.w[:, 0, :] += 45.0
        L, G, St, _ = gpu_grad(wl, oracle_dataset(wl)["P"], 0)
        finite &= bool(np.all(np.isfinite(G)))
    print(json.dumps({"enabled": B.debug_bounds_enabled(), "finite": finite, "bounds": B.debug_bounds(reset=True)}))


if __name__ == "__main__":
    main()
