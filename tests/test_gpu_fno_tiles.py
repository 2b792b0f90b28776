"""The register-tiled FP32 kernels of the FNO at the edges of their tiles: x
transforms of few and of very many rows, channel mixes with odd row counts and
ragged strips, z transforms across chunk borders, weight gradients for every
block height.  Against float64 sums; the tolerance is the FP32 rounding bound of a
dot product of n terms, n 2^-24 on the sum of the terms' magnitudes (with the
table's own rounding, one more 2^-24)."""
import numpy as np
import pytest
import torch

from paper_2304_05592_gb300 import fno

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


def _rand(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda")


def _close(got, ref, mag, n):
    bad = (got.double() - ref).abs() > (n + 2) * EPS * mag + 1e-30
    assert not bool(bad.any()), float(((got.double() - ref).abs() / mag).max())


@pytest.mark.parametrize("rows,Nx", [(1, 32), (129, 36), (300, 64), (4000, 516), (155648 + 37, 32), (155648, 52)])
def test_x_transform_tiles(rows, Nx):
    x, t = _rand((rows, Nx), 1), _rand((Nx, 16, 2), 2)
    got = fno.fno_dft_x(x, 16, t).reshape(rows, 32)
    tab = t.reshape(Nx, 32).double()
    _close(got, x.double() @ tab, x.double().abs() @ tab.abs(), Nx)


@pytest.mark.parametrize("ci,co,Nz,Nx,spec", [(32, 32, 9, 132, True), (32, 32, 1, 128, True), (5, 32, 17, 260, True),
                                             (32, 64, 11, 100, False), (64, 32, 8, 516, True), (3, 64, 23, 128, True)])
@pytest.mark.parametrize("trans", [False, True])
def test_channel_mix_tiles(ci, co, Nz, Nx, spec, trans):
    B, mx = 2, 16
    v, M, b = _rand((B, ci, Nz, Nx), 3), _rand((ci, co) if trans else (co, ci), 4), _rand((co,), 5)
    T, tab = _rand((B, co, Nz, mx, 2), 6), _rand((Nx, mx, 2), 7)
    got = fno.fno_combine(v, M, co, m_trans=trans, bias=b, T=T if spec else None, table=tab if spec else None, mx=mx)
    W = (M.t() if trans else M).double()
    ref = torch.einsum("oi,bizx->bozx", W, v.double()) + b.double()[None, :, None, None]
    mag = torch.einsum("oi,bizx->bozx", W.abs(), v.double().abs()) + b.double().abs()[None, :, None, None]
    if spec:
        Td, td = T.double(), tab.double()
        ref += torch.einsum("bozk,xk->bozx", Td[..., 0], td[..., 0]) - torch.einsum("bozk,xk->bozx", Td[..., 1], td[..., 1])
        mag += torch.einsum("bozk,xk->bozx", Td[..., 0].abs(), td[..., 0].abs())
        mag += torch.einsum("bozk,xk->bozx", Td[..., 1].abs(), td[..., 1].abs())
    _close(got, ref, mag, ci + 33)


@pytest.mark.parametrize("Nz,mz", [(64, 16), (65, 16), (127, 20), (48, 8)])
def test_z_transform_chunks(Nz, mz):
    nb, mx = 5, 12
    x, tz = _rand((nb, Nz, mx, 2), 8), _rand((Nz, 2 * mz, 2), 9)
    got = torch.view_as_complex(fno.fno_dft_z(x, nb, Nz, mz, mx, tz).double())
    X, E = torch.view_as_complex(x.double()), torch.view_as_complex(tz.double()).conj()
    mag = torch.einsum("bzk,za->bak", X.abs(), E.abs())
    err = (got - torch.einsum("bzk,za->bak", X, E)).abs()
    assert bool((err <= 4 * (Nz + 2) * EPS * mag).all())


@pytest.mark.parametrize("ci,co,npix", [(3, 32, 1000), (32, 32, 4096), (32, 64, 2050), (64, 1, 777), (7, 9, 64), (64, 64, 513),
                                       (1, 3, 5)])
def test_weight_gradient_blocks(ci, co, npix):
    B = 3
    dU, v = _rand((B, co, 1, npix), 10), _rand((B, ci, 1, npix), 11)
    dM, db = torch.empty((co, ci), device="cuda"), torch.empty((co,), device="cuda")
    work = torch.empty(fno.fno_wgrad_work_floats(B, ci, co, npix), device="cuda")
    fno.fno_wgrad(dU, v, dM, db, work)
    d, x = dU.double().reshape(B, co, -1), v.double().reshape(B, ci, -1)
    _close(dM, torch.einsum("bop,bip->oi", d, x), torch.einsum("bop,bip->oi", d.abs(), x.abs()), B * npix)
    _close(db, d.sum((0, 2)), d.abs().sum((0, 2)), B * npix)
