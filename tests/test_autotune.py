"""The autotuner's candidates cover the library's own automatic shapes (host arithmetic; the tuning itself is in
test_gpu_scheduling.py)."""
import os
import re

import pytest

from paper_2105_12070_gb300 import autotune, chem

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_12070_gb300", "csrc")


@pytest.mark.parametrize("precision", [chem.CHEM_PREC_FP64, chem.CHEM_PREC_MIXED, chem.CHEM_PREC_MIXED_FF])
@pytest.mark.parametrize("solver", [chem.CHEM_SOLVER_ROSENBROCK, chem.CHEM_SOLVER_SEULEX])
def test_candidates_reach_the_kernels_cta_sizes(precision, solver):
    threads = int(re.search(r"#define CHEM_MAX_THREADS_PER_CTA (\d+)", open(os.path.join(CSRC, "integrate.h")).read()).group(1))
    default = precision == chem.CHEM_PREC_FP64 and solver == chem.CHEM_SOLVER_ROSENBROCK
    for G in (1, 2, 4, 8):
        most = threads // 4 * 5 if G == 2 and default else threads  # integrate_max_threads
        assert [c for g, c in autotune.candidates(precision, solver) if g == G] == list(range(1, most // (32 * G) + 1))
