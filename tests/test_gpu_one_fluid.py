"""Pure tiles with one fluid around (their own launch, which moves nine populations per node) against
the launches that move all 27: the same bits, whichever takes a tile.  LBM3_ONE_TILES moves the
line between the two at lbm3_create."""
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


def pair(gpu, monkeypatch, w, precision):
    sims = []
    for line in ("1", "1000000000"):
        monkeypatch.setenv("LBM3_ONE_TILES", line)
        sims.append(gpu.Lbm3.from_workload(w, precision=precision))
    assert sims[0].info()["step_kernels"] == sims[1].info()["step_kernels"] + 1
    return sims


def same(a, b):
    for x, y in zip(a.get_state() + a.fields(), b.get_state() + b.fields()):
        assert np.array_equal(x, y, equal_nan=True)
    assert np.array_equal(a.diag(check=False), b.diag(check=False), equal_nan=True)


# nx a multiple of 8 (bulk copies), of 4 (FP32 only) and odd (plain loads); a droplet that moves and
# spreads over tiles that held one fluid before
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nx,ny", [(320, 120), (324, 119), (319, 123)])
def test_one_fluid_tiles_match_the_general_kernels(gpu, monkeypatch, precision, nx, ny):
    w = W.pillars(nx=nx, ny=ny, count=3, r_lo=6.0, r_hi=9.0, x_lo=150.0, x_hi=260.0, gap=8.0, seed=5,
                  drop=(60.0, 60.0), r_core=8.0, r_shell=14.0, u_in=0.05)
    a, b = pair(gpu, monkeypatch, w, precision)
    for n in (1, 2, 13, 60):  # odd and even counts: either buffer, single launches and graphs
        a.step(n)
        b.step(n)
        same(a, b)
    f, c = a.get_state()
    a.set_state(f, c)
    b.set_state(f, c)
    a.step(11)
    b.step(11)
    same(a, b)


# a density without a fraction (0, infinite, NaN) in a region of one fluid spreads to the absent
# fluids' populations as it does in the general kernels
@pytest.mark.parametrize("precision", [0, 1], ids=["fp32", "fp16"])
@pytest.mark.parametrize("value", [0.0, np.inf, np.nan])
def test_one_fluid_tiles_without_a_fraction(gpu, monkeypatch, precision, value):
    w = W.janus_cylinder(nx=256, ny=128, Rs=10.0, Rj=9.0)
    a, b = pair(gpu, monkeypatch, w, precision)
    a.step(20)
    b.step(20)
    f, c = a.get_state()
    f[:, :, 30, 60] = 0.0
    f[1, :, 30, 60] = value
    for s in (a, b):
        s.set_state(f, c)
        s.step(1)
    same(a, b)
    a.step(6)
    b.step(6)
    same(a, b)
