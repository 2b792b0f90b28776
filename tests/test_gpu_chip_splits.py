"""The on-chip 2D time loop runs where it is expected to (told by the launches a call
makes), and every shape of it (rows per thread, sponge factors stored or formed) in
every mode, split over small and large clusters, gives the records of the direct
kernel bit for bit and its gradients to rounding."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2304_05592_gb300 import synth, wave
from paper_2304_05592_gb300.wave import Grid

pytestmark = pytest.mark.gpu

TOL_GRAD = 1e-5  # FP32 sums in another order, as between the other step kernels
FEW = 20         # launches of a call beside its time steps: set-up, residual, reductions


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.fixture(autouse=True)
def restore():
    yield
    _force(-1, 0)
    wave.wave_set_variant(0, -1)
    wave.wave_set_variant(1, -1)


def _force(shape, clusters, refuse=0):
    f = ctypes.CDLL(wave.library_path()).wave_chip_force
    f.argtypes, f.restype = [ctypes.c_int] * 3, ctypes.c_int
    return f(shape, clusters, refuse)


def _problem(name):
    if name == "surface":  # taps in few rows: injection in the row loop; the padded grid is 91 x 69
        p = synth.small_2d(31, nt=61, nshot=2, nrec=40)
        p.src[:, :, 1] = 2.5 * p.h
        p.rec[:, :, 1] = 1.5 * p.h
    elif name == "borehole":  # taps in every row, the strips' borders among them: injection between barriers
        p = synth.small_2d(32, nt=61, nshot=2, nrec=50)
        p.rec[:, :, 0] = 0.41 * (p.nx - 1) * p.h
        p.rec[:, :, 1] = np.linspace(0.0, (p.nz - 1) * p.h, 50)
    else:  # one quad of live points past a multiple of 4, 137 x 150 padded
        p = synth.small_2d(33, nx=97, nz=110, nb=20, nt=61, nshot=3, nrec=30)
    return p


def _calls(p):
    """The five modes: records, source-side adjoint, gradients with the forward levels in FP32 and BF16; with
    the launches each call made."""
    g = Grid.of(p)
    rng = np.random.default_rng(5)
    q = torch.from_numpy(rng.standard_normal((p.nshot, p.nt, 1)).astype(np.float32)).cuda()
    r = torch.from_numpy(rng.standard_normal((p.nshot, p.nt, p.rec.shape[1])).astype(np.float32)).cuda()
    v = torch.from_numpy(p.vel).cuda()
    out = []
    for f in (lambda: wave.wave_forward(g, v, p.src, q, p.rec),
              lambda: wave.wave_adjoint(g, v, p.src, p.rec, r),
              lambda: wave.wave_gradient(g, v, p.src, q, p.rec, 0.3 * r, store=wave.STORE_FP32, want_dsyn=True),
              lambda: wave.wave_gradient(g, v, p.src, q, p.rec, 0.3 * r, store=wave.STORE_BF16, want_dsyn=True)):
        n = wave.wave_launch_count()
        o = f()
        out.append((o, wave.wave_launch_count() - n))
    return out


@pytest.mark.parametrize("name", ["surface", "borehole", "wider"])
def test_every_shape_and_cluster_size(name):
    p = _problem(name)
    wave.wave_set_variant(0, 0)
    wave.wave_set_variant(1, 0)
    ref = _calls(p)
    assert all(n > p.nt - 1 for _, n in ref)
    wave.wave_set_variant(0, wave.wave_variant_count(0) - 1)
    wave.wave_set_variant(1, wave.wave_variant_count(1) - 1)
    nshape = _force(-1, 0)
    ran = {}
    for shape in range(nshape):
        for clusters in (1, 2, 3, 4, 5, 7, 8, 11, 13, 16):
            _force(shape, clusters)
            got = _calls(p)
            on_chip = [n < p.nt - 1 for _, n in got]
            if on_chip[0]:
                ran.setdefault((shape, 0), set()).add(clusters)
                assert torch.equal(got[0][0], ref[0][0]), (shape, clusters)
            if on_chip[1]:
                ran.setdefault((shape, 2), set()).add(clusters)
                assert torch.equal(got[1][0], ref[1][0]), (shape, clusters)
            for k, modes in ((2, (3,)), (3, (1, 4))):
                phi, gr, ds = got[k][0]
                phi0, gr0, ds0 = ref[k][0]
                assert phi == phi0 and torch.equal(ds, ds0), (shape, clusters, k)
                assert float((gr - gr0).norm()) <= TOL_GRAD * float(gr0.norm()), (shape, clusters, k)
                if on_chip[k]:  # both directions
                    for m in modes:
                        ran.setdefault((shape, m), set()).add(clusters)
    missing = [(s, m) for s in range(nshape) for m in range(5) if (s, m) not in ran]
    assert not missing, (missing, {k: sorted(v) for k, v in ran.items()})


@pytest.mark.parametrize("mk,expected", [
    (lambda: synth.small_2d(34, nt=120, nshot=3), True),
    (lambda: synth.small_2d(35, nx=140, nz=100, nb=20, nt=90, nshot=2, nrec=100), True),
    (lambda: synth.small_2d(11, nx=1300, nz=700, nt=12, nb=10, nshot=1, nrec=50), False),
])
def test_the_loop_runs_by_itself_where_it_is_expected(mk, expected):
    p = mk()
    for o, n in _calls(p):
        steps = p.nt - 1
        if expected:
            assert n <= FEW, n
        else:
            assert n >= steps, n
