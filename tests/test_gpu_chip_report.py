"""What the on-chip 2D time loop reports: launches that CUDA refuses (on the host: a
request for more shared memory than there is), and profile samples of launches that
hold many time steps."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2304_05592_gb300 import synth, wave
from paper_2304_05592_gb300.wave import Grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


def _refuse(on):
    f = ctypes.CDLL(wave.library_path()).wave_chip_force
    f.argtypes, f.restype = [ctypes.c_int] * 3, ctypes.c_int
    f(-1, 0, int(on))


@pytest.fixture(autouse=True)
def restore():
    yield
    _refuse(False)
    torch.cuda.synchronize()


def _case(nt=80):
    p = synth.small_2d(41, nt=nt, nshot=2)
    rng = np.random.default_rng(1)
    q = torch.from_numpy(rng.standard_normal((p.nshot, p.nt, 1)).astype(np.float32)).cuda()
    d = torch.from_numpy(rng.standard_normal((p.nshot, p.nt, p.rec.shape[1])).astype(np.float32)).cuda()
    return p, Grid.of(p), torch.from_numpy(p.vel).cuda(), q, d


@pytest.mark.parametrize("op", ["forward", "adjoint", "gradient"])
def test_a_refused_launch_is_reported_once(op):
    p, g, v, q, d = _case()
    call = {"forward": lambda: wave.wave_forward(g, v, p.src, q, p.rec),
            "adjoint": lambda: wave.wave_adjoint(g, v, p.src, p.rec, d),
            "gradient": lambda: wave.wave_gradient(g, v, p.src, q, p.rec, d, nsnap=5)}[op]
    first = call()
    n = wave.wave_launch_count()
    call()
    assert wave.wave_launch_count() - n < p.nt - 1  # the loop, not a launch per step
    _refuse(True)
    with pytest.raises(wave.WaveError) as e:
        call()
    assert e.value.status == 5  # WAVE_ERR_CUDA
    _refuse(False)
    again = call()  # its first check of CUDA's last error must not find the old one
    a, b = (x if torch.is_tensor(x) else x[1] for x in (first, again))
    assert torch.equal(a, b)


def test_autotune_does_not_pick_a_loop_that_cannot_be_launched():
    p = synth.small_2d(42, nx=71, nz=47, nt=60, nshot=2)  # (a size of its own: the choice is remembered)
    g, v = Grid.of(p), torch.from_numpy(p.vel).cuda()
    q = torch.ones((p.nshot, p.nt, 1), device="cuda")
    last = [wave.wave_variant_count(w) - 1 for w in (0, 1)]
    _refuse(True)
    picked = wave.wave_autotune(g, v, p.src, q, p.rec, steps=4)
    _refuse(False)
    again = wave.wave_autotune(g, v, p.src, q, p.rec, steps=4)
    assert picked[0] != last[0] and picked[1] != last[1], (picked, again)


@pytest.mark.parametrize("every", [1, 10, 60])
def test_profile_samples_every_nth_step(every):
    """`every` counts time steps: a launch that holds many of them is sampled if one of them is due.  80
    samples: 79 forward steps, then 79 adjoint steps."""
    p, g, v, q, d = _case()
    wave.wave_gradient(g, v, p.src, q, p.rec, d, store=wave.STORE_FP32)
    wave.wave_profile_start(every)
    wave.wave_gradient(g, v, p.src, q, p.rec, d, store=wave.STORE_FP32)
    fms, fn, ams, an = wave.wave_profile_stop()
    assert fn == p.nt - 1 and fms > 0.0
    assert an == p.nt - 1 and ams > 0.0
