"""The estimated time of a launched 2D step, by which the kernels of a call are chosen
(host only): a batch smaller than a group of shots does its own work and no less."""
import ctypes

import pytest

from paper_2304_05592_gb300 import wave
from paper_2304_05592_gb300.wave import Grid


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2304_05592_gb300 import build

    build.build()


def _step(nx, nz, nshot, adjoint):
    f = ctypes.CDLL(wave.library_path()).wave_shot_group
    g = Grid(2, nx, nz, 10.0, 1e-3, 100, 0).c()
    us = ctypes.c_float(0.0)
    return f(ctypes.byref(g), nshot, adjoint, ctypes.byref(us)), us.value


@pytest.mark.parametrize("adjoint", [0, 1])
@pytest.mark.parametrize("nx,nz", [(91, 69), (592, 336), (1280, 580), (3000, 1500), (8000, 6000)])
def test_a_shot_takes_no_less_than_its_share_of_a_batch(nx, nz, adjoint):
    # (shots of a batch share the set-up of their tiles and fill each other's gaps)
    share = _step(nx, nz, 32, adjoint)[1] / 32
    for nshot in (1, 2, 3, 5):
        assert _step(nx, nz, nshot, adjoint)[1] >= 0.999 * nshot * share, nshot
