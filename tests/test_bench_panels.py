"""bench.panel_work: the tangent work counted panel by panel."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402
from paper_2508_06302_gb300 import inputs as I  # noqa: E402


def test_panels_of_the_shell_workload():
    # bending, membrane and drilling dofs of the 312 free nodes; half-bandwidths of the grid's short side
    m = I.workload_shell1872().model
    assert [p[:2] for p in bench.tangent_panels(m)] == [(936, 44), (624, 29), (312, 0)]
    w = bench.panel_work(m, 64, 4)
    assert w["sens_rhs"][1] == pytest.approx(3 * 4 * 64 * sum(n * (2 * n + 1) for n in (936, 624, 312)))


def test_undivided_models_count_as_a_whole():
    m = I.eb_beam()
    p, = bench.tangent_panels(m)
    assert bench.panel_work(m, 5, 8) == bench.step_work(m, 5, p.band, 0, 8)
