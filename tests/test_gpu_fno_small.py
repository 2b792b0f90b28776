"""FNO channel mixes with 1 to 8 rows per block, by how much there is to do.  Small maps
must not pay for what large ones gain."""
import pytest
import torch

from paper_2304_05592_gb300 import fno

pytestmark = pytest.mark.gpu


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
