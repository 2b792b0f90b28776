"""Many shots of a small grid over few steps: the host's choice between the on-chip loop
and a launch per step takes little beside the tap tables, which either needs."""
import time

import pytest
import torch

from paper_2304_05592_gb300 import synth, wave
from paper_2304_05592_gb300.wave import Grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.fixture(autouse=True)
def restore_variants():
    yield
    wave.wave_set_variant(0, -1)
    wave.wave_set_variant(1, -1)


def _seconds(f):
    f()
    torch.cuda.synchronize()
    out = []
    for _ in range(7):
        t = time.perf_counter()
        f()
        torch.cuda.synchronize()
        out.append(time.perf_counter() - t)
    return sorted(out)[3]


def test_choosing_the_loop_costs_little_for_many_shots():
    p = synth.small_2d(61, nt=4, nshot=1000, nrec=200)
    p.rec[:, :, 1] = 2.5 * p.h
    g, v = Grid.of(p), torch.from_numpy(p.vel).cuda()
    q = torch.ones((p.nshot, p.nt, 1), device="cuda")
    d = torch.ones((p.nshot, p.nt, p.rec.shape[1]), device="cuda")

    def call():
        return wave.wave_gradient(g, v, p.src, q, p.rec, d, store=wave.STORE_BF16)

    own = _seconds(call)
    wave.wave_set_variant(0, 44)  # shot groups: no choice to make
    wave.wave_set_variant(1, 42)
    assert own <= 1.5 * _seconds(call)
