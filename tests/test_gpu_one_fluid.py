"""The launches that a tile can be done by: those for one fluid, which move nine populations per node,
those that move all 27 by bulk copies or plain loads, and the one launch of all tiles: the same bits,
whichever takes it.  LBM3_ONE_TILES, LBM3_DISABLE_TMA, LBM3_CHAIN_TILES and LBM3_PURE_KERNEL
choose at lbm3_create."""
import numpy as np
import pytest

from paper_2102_04709_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2102_04709_gb300 import build, lbm3
    build.build()
    lbm3.load()
    return lbm3


def variants(gpu, monkeypatch, w, precision):
    sims, kernels = [], [4, 2, 2, 1]
    ways = [("1", "0", "0", ""), ("1000000000", "0", "0", ""), ("1000000000", "0", "1", ""), ("1", "1000000000", "0", "")]
    if precision == 0 and w.nx % 4 == 0:
        ways.append(("1", "0", "0", "tma"))  # the two-blocks-per-SM kernel takes every pure tile
        kernels.append(2)
    for one, chain, plain, pure in ways:
        monkeypatch.setenv("LBM3_ONE_TILES", one)
        monkeypatch.setenv("LBM3_CHAIN_TILES", chain)
        monkeypatch.setenv("LBM3_DISABLE_TMA", plain)
        monkeypatch.setenv("LBM3_PURE_KERNEL", pure)
        sims.append(gpu.Lbm3.from_workload(w, precision=precision))
    assert [s.info()["step_kernels"] for s in sims] == kernels
    return sims


def same(a, *others):
    x = a.get_state() + a.fields() + (a.diag(check=False),)
    for b in others:
        for p, q in zip(x, b.get_state() + b.fields() + (b.diag(check=False),)):
            assert np.array_equal(p, q, equal_nan=True)


# nx a multiple of 8 (bulk copies), of 4 (FP32 only) and odd (plain loads); a droplet that moves and
# spreads over tiles that held one fluid before
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nx,ny", [(320, 120), (324, 119), (319, 123)])
def test_every_launch_gives_the_same_bits(gpu, monkeypatch, precision, nx, ny):
    w = W.pillars(nx=nx, ny=ny, count=3, r_lo=6.0, r_hi=9.0, x_lo=150.0, x_hi=260.0, gap=8.0, seed=5,
                  drop=(60.0, 60.0), r_core=8.0, r_shell=14.0, u_in=0.05)
    sims = variants(gpu, monkeypatch, w, precision)
    for n in (1, 2, 13, 60):  # odd and even counts: either buffer, single launches and graphs
        for s in sims:
            s.step(n)
        same(*sims)
    f, c = sims[0].get_state()
    for s in sims:
        s.set_state(f, c)
        s.step(11)
    same(*sims)


# a density without a fraction (0, infinite, NaN) in a region of one fluid spreads to the absent
# fluids' populations as it does in the general kernels
@pytest.mark.parametrize("precision", [0, 1], ids=["fp32", "fp16"])
@pytest.mark.parametrize("value", [0.0, np.inf, np.nan])
def test_one_fluid_tiles_without_a_fraction(gpu, monkeypatch, precision, value):
    w = W.janus_cylinder(nx=256, ny=128, Rs=10.0, Rj=9.0)
    sims = variants(gpu, monkeypatch, w, precision)
    for s in sims:
        s.step(20)
    f, c = sims[0].get_state()
    f[:, :, 30, 60] = 0.0
    f[1, :, 30, 60] = value
    for n in (1, 6):
        for s in sims:
            if n == 1:
                s.set_state(f, c)
            s.step(n)
        same(*sims)


# tiles with only traces of all fluids but one take no gradients: the same bits as with them, which every
# tile takes in the step after a set_state; pillars among the traces, in every launch that has both ways
@pytest.mark.parametrize("nx,ny,chain", [(320, 120, "1000000000"), (320, 120, "0"), (319, 123, "0")],
                         ids=["one-launch", "ring", "plain"])
def test_traces_match_the_general_way(gpu, monkeypatch, nx, ny, chain):
    w = W.pillars(nx=nx, ny=ny, count=6, r_lo=5.0, r_hi=8.0, x_lo=110.0, x_hi=280.0, gap=8.0, seed=5,
                  drop=(60.0, 60.0), r_core=8.0, r_shell=14.0, u_in=0.02)
    monkeypatch.setenv("LBM3_ONE_TILES", "1")
    monkeypatch.setenv("LBM3_CHAIN_TILES", chain)
    a = gpu.Lbm3.from_workload(w)
    b = gpu.Lbm3.from_workload(w)
    a.step(150)
    r = np.abs(a.fields()[0])
    assert np.count_nonzero((r > 0) & (r < 1e-13)) > nx * ny // 4  # there are traces, and over many tiles
    b.set_state(*a.get_state())
    for _ in range(40):
        b.set_state(*b.get_state())
        a.step(1)
        b.step(1)
    same(a, b)
