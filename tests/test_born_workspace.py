"""Device memory of Born modelling (host only): in 2D two background and two scattered
levels per shot and one perturbation for all shots, beside what forward modelling
(two levels) takes; in 3D a third background level."""
import numpy as np
import pytest

from paper_2304_05592_gb300 import wave
from paper_2304_05592_gb300.wave import Grid


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2304_05592_gb300 import build

    build.build()


@pytest.mark.parametrize("ndim,levels", [(2, 4), (3, 5)])
def test_levels_of_a_born_workspace(ndim, levels):
    g = Grid(ndim, 93, 61, 10.0, 1e-3, 50, 10, ny=21 if ndim == 3 else 1)
    none = np.zeros

    def more(nshot):  # bytes beyond those of forward modelling, no taps
        pts = none((nshot, 0, ndim))
        return (wave.wave_workspace_size(g, wave.OP_BORN, pts, pts) - wave.wave_workspace_size(g, wave.OP_FORWARD, pts, pts))

    cell = (more(9) - more(1)) / (8.0 * (levels - 2))  # bytes of one level of one shot
    assert abs(more(1) - (levels - 1) * cell) <= 1024  # the levels and the perturbation; arrays start at 256 bytes
