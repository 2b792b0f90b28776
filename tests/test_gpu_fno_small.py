"""FNO kernels whose launch depends on how much there is to do: channel mixes with 1 to 8
rows per block, weight gradients with either block height, z transforms by pairs of
modes and singly.  Small maps must not pay for what large ones gain."""
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


def _us(f, n=16):
    """Device time of a call (us): n calls in a graph, the best of 7 replays."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        f()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for _ in range(n):
                f()
        best = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(s)
            g.replay()
            b.record(s)
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3 / n)
    return best


def _mix(B, ci, co, Nz, Nx, spec, seed=1):
    v, M, b = _rand((B, ci, Nz, Nx), seed), _rand((co, ci), seed + 1), _rand((co,), seed + 2)
    T, tab = _rand((B, co, Nz, 16, 2), seed + 3), _rand((Nx, 16, 2), seed + 4)
    return v, M, b, (T if spec else None), (tab if spec else None)


# rows per block: 2, 4, 8 with 32 outputs, 1, 2, 4, 8 with 64 (152 SMs), ragged last blocks and strips
@pytest.mark.parametrize("co,B,Nz", [(32, 1, 33), (32, 3, 601), (32, 3, 1037), (64, 1, 33), (64, 3, 301), (64, 3, 603),
                                     (64, 3, 1037)])
@pytest.mark.parametrize("ci,spec", [(5, True), (32, False)])
def test_channel_mix_gives_the_same_bits_for_any_rows_per_block(co, B, Nz, ci, spec):
    Nx = 132
    v, M, b, T, tab = _mix(B, ci, co, Nz, Nx, spec)
    got = fno.fno_combine(v, M, co, bias=b, T=T, table=tab, mx=16, act=fno.ACT_GELU)
    for z0 in range(0, Nz, 29):  # few rows: one or two per block
        z1 = min(z0 + 29, Nz)
        part = fno.fno_combine(v[:, :, z0:z1].contiguous(), M, co, bias=b, T=T[:, :, z0:z1].contiguous() if spec else None,
                               table=tab, mx=16, act=fno.ACT_GELU)
        assert torch.equal(got[:, :, z0:z1], part), z0


@pytest.mark.parametrize("co", [32, 64])
@pytest.mark.parametrize("spec", [True, False])
def test_a_small_channel_mix_takes_a_fraction_of_a_larger_one(co, spec):
    def t(B):
        v, M, b, T, tab = _mix(B, co, co, 90, 72, spec)
        out = torch.empty((B, co, 90, 72), device="cuda")
        return _us(lambda: fno.fno_combine(v, M, co, bias=b, T=T, table=tab, mx=16, act=fno.ACT_GELU, out=out))

    assert t(1) < 0.75 * t(8)  # (equal with 8 rows per block for both)


def _wgrad(B, ci, co, npix):
    dU, v = _rand((B, co, 1, npix), 10), _rand((B, ci, 1, npix), 11)
    dM, db = torch.empty((co, ci), device="cuda"), torch.empty((co,), device="cuda")
    work = torch.empty(max(1, fno.fno_wgrad_work_floats(B, ci, co, npix)), device="cuda")
    return dU, v, dM, db, work


# either side of 2 x 152 blocks of 512 pixels, of 8 outputs and of 4 inputs
@pytest.mark.parametrize("B,npix", [(1, 1), (2, 130), (1, 303 * 512), (1, 304 * 512 + 3), (5, 40000)])
@pytest.mark.parametrize("ci,co", [(1, 16), (3, 64), (4, 8), (4, 7), (33, 20), (64, 64)])
def test_weight_gradients_either_side_of_the_rule(B, npix, ci, co):
    dU, v, dM, db, work = _wgrad(B, ci, co, npix)
    fno.fno_wgrad(dU, v, dM, db, work)
    d, x = dU.double().reshape(B, co, -1), v.double().reshape(B, ci, -1)
    for got, ref, mag in ((dM, torch.einsum("bop,bip->oi", d, x), torch.einsum("bop,bip->oi", d.abs(), x.abs())),
                          (db, d.sum((0, 2)), d.abs().sum((0, 2)))):
        assert not bool(((got.double() - ref).abs() > (B * npix + 2) * EPS * mag + 1e-30).any())


def test_one_input_channel_takes_no_longer_than_sixteen():
    def t(ci):
        dU, v, dM, db, work = _wgrad(1, ci, 16, 4096)
        return _us(lambda: fno.fno_wgrad(dU, v, dM, db, work))

    assert t(1) <= t(16)


@pytest.mark.parametrize("mx", [1, 7, 8, 15, 16])
@pytest.mark.parametrize("Nz,mz", [(31, 3), (64, 16), (131, 9)])
@pytest.mark.parametrize("shift", [0, 1])
def test_z_transform_by_pairs_and_singly(mx, Nz, mz, shift):
    """shift: inputs one complex number past a 16-byte boundary."""
    nb = 3
    x, tz = (_rand((n + 2 * shift,), 8 + n)[2 * shift:].view(*s, 2) for n, s in
             ((nb * Nz * mx * 2, (nb, Nz, mx)), (Nz * 2 * mz * 2, (Nz, 2 * mz))))
    assert x.data_ptr() % 16 == 8 * shift
    got = torch.view_as_complex(fno.fno_dft_z(x, nb, Nz, mz, mx, tz).double())
    X, E = torch.view_as_complex(x.double()), torch.view_as_complex(tz.double()).conj()
    mag = torch.einsum("bzk,za->bak", X.abs(), E.abs())
    err = (got.view(nb, 2 * mz, mx) - torch.einsum("bzk,za->bak", X, E)).abs()
    assert bool((err <= 4 * (Nz + 2) * EPS * mag).all())


@pytest.mark.parametrize("ci,co", [(43, 64), (43, 7)])
def test_odd_maps_take_little_more_than_even_ones(ci, co):
    """Rows that do not begin at 16 bytes are loaded pixel by pixel, with enough loads in flight."""
    def t(npix):
        dU, v, dM, db, work = _wgrad(3, ci, co, npix)
        return _us(lambda: fno.fno_wgrad(dU, v, dM, db, work))

    assert t(131071) < 1.6 * t(131072)
