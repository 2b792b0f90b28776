"""The on-chip 2D time loop (many steps per launch, one cluster per shot) against
the step-per-launch kernels: records are bitwise those of the direct kernel
(variant 0), gradients agree to rounding (the shot sum and the receivers' share
are grouped differently), for strips, remainders and tap layouts at the edges of
what the loop takes."""
import numpy as np
import pytest
import torch

from paper_2304_05592_gb300 import synth, wave
from paper_2304_05592_gb300.wave import Grid

pytestmark = pytest.mark.gpu

TOL_GRAD = 1e-5  # FP32 sums in another order, as between the other step kernels


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.fixture(autouse=True)
def restore_variants():
    yield
    wave.wave_set_variant(0, -1)
    wave.wave_set_variant(1, -1)


def _lines(p, depth):
    """Sources and receivers of p on lines at the given depth (cells), off the grid for a fractional one."""
    p.src[:, :, 1] = depth * p.h
    p.rec[:, :, 1] = depth * p.h
    return p


def _borehole(p):
    """Receivers down a vertical line: taps in every row."""
    p.rec[:, :, 0] = 0.37 * (p.nx - 1) * p.h
    p.rec[:, :, 1] = np.linspace(0.0, (p.nz - 1) * p.h, p.rec.shape[1])
    return p


CASES = {
    "one_strip_row": lambda: synth.small_2d(1, nx=9, nz=5, nt=30, nb=0, nshot=1, nrec=3),
    "ragged_x_1": lambda: _lines(synth.small_2d(2, nx=61, nz=40, nt=90, nb=12, nshot=2, nrec=21), 2),
    "ragged_x_3": lambda: _lines(synth.small_2d(3, nx=63, nz=41, nt=91, nb=8, nshot=3, nrec=17), 2.4),
    "border_taps": lambda: _lines(synth.small_2d(4, nx=200, nz=120, nt=70, nb=20, nshot=2, nrec=200), 10),
    "borehole": lambda: _borehole(synth.small_2d(5, nx=150, nz=97, nt=80, nb=16, nshot=2, nrec=60)),
    "two_steps": lambda: synth.small_2d(6, nx=70, nz=50, nt=3, nshot=2, nrec=9),
    "no_steps": lambda: synth.small_2d(7, nx=70, nz=50, nt=1, nshot=2, nrec=9),
    "more_shots_than_clusters": lambda: _lines(synth.small_2d(8, nx=160, nz=100, nt=40, nb=30, nshot=37, nrec=40), 3),
    "tall_rows": lambda: synth.small_2d(9, nx=520, nz=250, nt=24, nb=40, nshot=2, nrec=90),
    "wide": lambda: synth.small_2d(10, nx=1500, nz=60, nt=24, nb=10, nshot=1, nrec=50),
    "too_large": lambda: synth.small_2d(11, nx=1300, nz=700, nt=12, nb=10, nshot=1, nrec=50),
    "long_table": lambda: synth.small_2d(12, nx=40, nz=30, nt=4400, nb=6, nshot=1, nrec=5),
}


def _run(p, vf, va, store, nsnap):
    g = Grid.of(p)
    rng = np.random.default_rng(3)
    q = torch.from_numpy(rng.standard_normal((p.nshot, p.nt, 1)).astype(np.float32)).cuda()
    r = torch.from_numpy(rng.standard_normal((p.nshot, p.nt, p.rec.shape[1])).astype(np.float32)).cuda()
    v = torch.from_numpy(p.vel).cuda()
    wave.wave_set_variant(0, vf)
    wave.wave_set_variant(1, va)
    d = wave.wave_forward(g, v, p.src, q, p.rec)
    a = wave.wave_adjoint(g, v, p.src, p.rec, r)
    phi, gr, ds = wave.wave_gradient(g, v, p.src, q, p.rec, 0.3 * r, store=store, nsnap=nsnap, want_dsyn=True)
    return d, a, phi, gr, ds


@pytest.mark.parametrize("name", list(CASES))
def test_on_chip_loop_matches_step_launches(name):
    p = CASES[name]()
    stores = [(wave.STORE_CHECKPOINT, 5), (wave.STORE_FP32, 1), (wave.STORE_BF16, 1)]
    if name == "long_table":
        stores = [(wave.STORE_CHECKPOINT, 3000), (wave.STORE_FP32, 1)]
    for store, nsnap in stores:
        ref = _run(p, 0, 0, store, nsnap)
        got = _run(p, wave.wave_variant_count(0) - 1, wave.wave_variant_count(1) - 1, store, nsnap)
        for k in (0, 1, 4):  # records, source-side adjoint, synthetic data
            assert torch.equal(got[k], ref[k]), (name, store, k)
        assert got[2] == ref[2]
        n = float(ref[3].norm())
        assert float((got[3] - ref[3]).norm()) <= TOL_GRAD * n, (name, store)


def test_checkpoint_runs_do_not_change_the_gradient():
    """The same steps split into launches at other places give the same bits."""
    p = _borehole(synth.small_2d(21, nx=130, nz=80, nt=203, nb=16, nshot=3, nrec=40))
    n0, n1 = wave.wave_variant_count(0) - 1, wave.wave_variant_count(1) - 1
    full = _run(p, n0, n1, wave.STORE_FP32, 1)[3]
    for nsnap in (1, 7, 40, 400):
        assert torch.equal(_run(p, n0, n1, wave.STORE_CHECKPOINT, nsnap)[3], full), nsnap
