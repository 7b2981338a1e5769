"""The iterative solves' value rows, asked for all at once after the solve: candidate counts around the rounds of 64 rows of a
block (in the last one some groups of lanes have fewer rows), and sequences with fewer tokens than candidates."""
import math

import pytest

from test_gpu_solver import compare_entropic, compare_fw, run_entropic, run_fw, spec
from workloads import make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K_c", [2, 63, 64, 65, 128, 129, 191, 192, 193, 255])
def test_candidate_counts(K_c):
    w = make_workload(spec(P=18, K_c=K_c, seq_lens=(700, 150, 60)), seed=8800 + K_c)
    w.gap_threshold = -math.inf          # no unit's output is replaced by the dense pass
    compare_entropic(w, run_entropic(w, 2), 2)
    compare_entropic(w, run_entropic(w, 2, fused=True), 2)
    compare_fw(w, run_fw(w, 2, fused=True), 2)
