"""The 2D Born step with 2 and 4 shots per CTA, full and partial last groups, ragged
tiles and taps on tile edges: the same bits as shot by shot (one shot per CTA), and
the FP64 oracle's records."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2304_05592_gb300 import synth, wave
from paper_2304_05592_gb300.wave import Grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


def _problem(nshot, nt=40):
    # padded 589 x 333: 5 x 21 tiles of 128 x 16, the last 77 points wide and 13 high
    p = synth.small_2d(51, nx=549, nz=293, nb=20, nt=nt, nshot=nshot, nrec=64)
    rng = np.random.default_rng(2)
    for s in range(nshot):  # sources and half of the receivers beside tile edges, in either direction
        p.src[s, 0] = ((128 * rng.integers(1, 4) - 20 - 1 + rng.random()) * p.h, (16 * rng.integers(2, 6) - 20 - 0.5) * p.h)
        p.rec[s, ::2, 0] = (128 * rng.integers(1, 5, 32) - 20 - 1) * p.h
        p.rec[s, ::2, 1] = (16 * rng.integers(2, 19, 32) - 20 - rng.random(32)) * p.h
    return p


def _shots_per_cta(g, nshot):
    f = ctypes.CDLL(wave.library_path()).wave_shot_group
    gc, us = g.c(), ctypes.c_float(0.0)
    return f(ctypes.byref(gc), nshot, 1, ctypes.byref(us))


@pytest.mark.parametrize("nshot,group", [(13, 2), (14, 2), (33, 4), (34, 4), (35, 4), (36, 4)])
def test_groups_match_single_shots(nshot, group):
    p = _problem(nshot)
    g = Grid.of(p)
    assert _shots_per_cta(g, nshot) == group and _shots_per_cta(g, 1) == 1
    rng = np.random.default_rng(3)
    q = torch.from_numpy(rng.standard_normal((nshot, p.nt, 1)).astype(np.float32)).cuda()
    v = torch.from_numpy(p.vel).cuda()
    m = 1.0 / p.vel.astype(np.float64) ** 2
    dm = (m * 0.05 * rng.standard_normal(m.shape)).astype(np.float32)
    dmd = torch.from_numpy(dm).cuda()
    got = wave.wave_born(g, v, p.src, q, p.rec, dmd)
    for s in range(nshot):
        one = wave.wave_born(g, v, p.src[s:s + 1], q[s:s + 1].contiguous(), p.rec[s:s + 1], dmd)
        assert torch.equal(got[s], one[0]), s
    og = oracle.Grid(p.ndim, p.nx, p.nz, p.h, p.dt, p.nt, p.nb, ny=p.ny, vref=p.vref)
    ref = oracle.born(og, p.vel, p.src, q.cpu().numpy(), p.rec, dm)
    d = got.cpu().numpy().astype(np.float64)
    assert float(np.linalg.norm(d - ref)) < 2e-4 * float(np.linalg.norm(ref))  # as for the other Born tests
