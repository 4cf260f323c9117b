"""The launches that a step is made of on larger grids -- the persistent kernels of the pure tiles, the
one-fluid launches, the tiles near solids beside them -- on grids small enough for the oracle, which by
themselves would be done by one launch of every tile (LBM3_CHAIN_TILES=0 splits them); and what the
tiles' words and cached lines say after a change from outside."""
import ctypes

import numpy as np
import pytest

from paper_2102_04709_gb300 import workloads as W
from tests.test_gpu_one_fluid import same, variants

pytestmark = pytest.mark.gpu

# against the FP64 oracle, as the parity tests: FP32, and the stated errors of the 16-bit storages
TOL_RHO, TOL_U = {0: 1e-5, 1: 5e-3, 2: 2e-2}, 1e-6
NEVER, ALWAYS = "1000000000", "1"


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2102_04709_gb300 import build, lbm3
    build.build()
    lbm3.load()
    return lbm3


def choose(monkeypatch, one=NEVER, chain="0", plain="0", pure=""):
    monkeypatch.setenv("LBM3_ONE_TILES", one)
    monkeypatch.setenv("LBM3_CHAIN_TILES", chain)
    monkeypatch.setenv("LBM3_DISABLE_TMA", plain)
    monkeypatch.setenv("LBM3_PURE_KERNEL", pure)


def pillars(nx=320, ny=120, u_in=0.05):
    return W.pillars(nx=nx, ny=ny, count=6, r_lo=5.0, r_hi=8.0, x_lo=110.0, x_hi=280.0, gap=8.0, seed=5,
                     drop=(60.0, 60.0), r_core=8.0, r_shell=14.0, u_in=u_in)


# ---- the tiles' words when the launches change ----
# A copy-wait limit other than the default takes a small grid from one launch of every tile to the split
# ones, and back: whatever launch takes over, the words must describe the state that the others left.
# (2^20 polls: no wait runs out.)
@pytest.mark.parametrize("precision,pure", [(0, "tma"), (0, ""), (1, "")], ids=["fp32-tma", "fp32-ring", "fp16"])
def test_a_change_of_the_wait_limit_keeps_the_state(gpu, monkeypatch, precision, pure):
    w = pillars()
    choose(monkeypatch, chain=NEVER, pure=pure)
    a = gpu.Lbm3.from_workload(w, precision=precision)
    b = gpu.Lbm3.from_workload(w, precision=precision)
    assert a.info()["step_kernels"] == 1
    for n in (41, 60):
        a.step(20)
        a.set_copy_wait_limit(1 << 20)
        assert a.info()["step_kernels"] == 2
        a.step(n)
        a.set_copy_wait_limit(-1)
        assert a.info()["step_kernels"] == 1
        a.step(30)
        b.step(20 + n + 30)
        same(a, b)


# ---- lines and words after new wall angles ----
# A step reads lines that the step before looked for, and looks anew only where wall values change: new
# angles have to replace them all at once.  Against a handle made with the new angles.
def turned(w, theta):
    new = w.angles.copy()
    new[..., 0], new[..., 2] = theta, 180.0 - theta
    return new


@pytest.mark.parametrize("precision", [0, 1], ids=["fp32", "fp16"])
@pytest.mark.parametrize("chain", [NEVER, "0"], ids=["one-launch", "split"])
def test_wall_angles_replaced_between_steps(gpu, monkeypatch, precision, chain):
    w = W.janus_cylinder(nx=256, ny=128, Rs=16.0, Rj=14.0)
    choose(monkeypatch, one=ALWAYS, chain=chain)
    a = gpu.Lbm3.from_workload(w, precision=precision)
    a.step(20)
    for theta in (70.0, 50.0):
        f, c = a.get_state()
        w.angles = turned(w, theta)
        b = gpu.Lbm3.from_workload(w, precision=precision)
        b.set_state(f, c)
        a.set_state(f, c)  # the same encoding as b's, the lines still those of the old angles
        a.set_wall_angles(w.angles.reshape(-1, 3)[a.wall_nodes()])
        a.step(15)
        b.step(15)
        same(a, b)


# Tiles near solids whose words say that nothing of the wetting changes, until the droplet's traces come.
# (FP32: its populations survive get_state bit for bit, so a goes on without a set_state.)
def test_wall_angles_replaced_in_settled_tiles(gpu, monkeypatch):
    w = pillars(u_in=0.02)
    choose(monkeypatch, one=ALWAYS)
    a = gpu.Lbm3.from_workload(w)
    a.step(20)
    for theta in (70.0, 110.0):
        w.angles = turned(w, theta)
        b = gpu.Lbm3.from_workload(w)
        b.set_state(*a.get_state())
        a.set_wall_angles(w.angles.reshape(-1, 3)[a.wall_nodes()])
        a.step(50)
        b.step(50)
        same(a, b)


# ---- the split launches against the oracle ----
def scene(name):
    if name == "pillars":    # open columns
        return W.pillars(nx=200, ny=96, count=4, r_lo=8.0, r_hi=14.0, x_lo=90.0, x_hi=180.0, gap=6.0, seed=11,
                         drop=(50.0, 48.0), r_core=12.0, r_shell=22.0, theta_range=(60.0, 120.0), u_in=0.02)
    if name == "capillary":  # the seam
        return W.capillary(nx=160, ny=40, y_lo=6, y_hi=34, s0=40, Lg=40, nu=(0.1, 0.01, 0.02))
    return W.janus_cylinder(nx=136, ny=90, Rs=16.0, Rj=14.0)  # periodic


@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("way", ["bulk", "bulk+one", "plain", "plain+one"])
@pytest.mark.parametrize("name", ["pillars", "capillary", "cylinder"])
def test_split_launches_match_oracle(gpu, oracle_mod, monkeypatch, name, way, precision):
    w = scene(name)
    choose(monkeypatch, one=ALWAYS if "one" in way else NEVER, plain="1" if "plain" in way else "0")
    g = gpu.Lbm3.from_workload(w, precision=precision)
    assert g.info()["step_kernels"] == (4 if "one" in way else 2)
    assert g.info()["tma"] == ("bulk" in way)
    o = oracle_mod.Oracle.from_workload(w, threads=0)
    g.step(200)
    o.step(200)
    assert np.abs(g.fields()[0] - o.fields()[0]).max() <= TOL_RHO[precision]
    if precision == 0:
        assert np.abs(g.fields()[1] - o.fields()[1]).max() <= TOL_U


def test_bulk_copies_with_two_blocks_per_sm_match_oracle(gpu, oracle_mod, monkeypatch):
    w = scene("pillars")
    choose(monkeypatch, pure="tma")
    g = gpu.Lbm3.from_workload(w)
    assert g.info()["pure_kernel"] == "bulk copies" and g.info()["step_kernels"] == 2
    o = oracle_mod.Oracle.from_workload(w, threads=0)
    g.step(200)
    o.step(200)
    assert np.abs(g.fields()[0] - o.fields()[0]).max() <= TOL_RHO[0]
    assert np.abs(g.fields()[1] - o.fields()[1]).max() <= TOL_U


# ---- the same bits from every launch, where the seam and thick walls are ----
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nx", [160, 163])
def test_every_launch_gives_the_same_bits_across_the_seam(gpu, monkeypatch, precision, nx):
    w = W.capillary(nx=nx, ny=60, y_lo=6, y_hi=54, s0=40, Lg=40, nu=(0.1, 0.02, 0.1))
    sims = variants(gpu, monkeypatch, w, precision)
    for n in (1, 2, 13, 90):
        for s in sims:
            s.step(n)
        same(*sims)


# ---- the one-fluid and the trace way against the general one, in every storage ----
# New wall angles (here the same ones) make every tile's word say "all fluids": the step after that takes
# no short way anywhere.
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("name,nx,ny,chain", [("pillars", 320, 120, NEVER), ("pillars", 320, 120, "0"),
                                              ("pillars", 319, 123, "0"), ("capillary", 320, 60, "0"),
                                              ("capillary", 320, 60, NEVER)],
                         ids=["one-launch", "bulk", "plain", "seam", "seam-one-launch"])
def test_short_ways_match_the_general_one(gpu, monkeypatch, precision, name, nx, ny, chain):
    if name == "pillars":
        w = pillars(nx, ny, u_in=0.02)
    else:
        w = W.capillary(nx=nx, ny=ny, y_lo=6, y_hi=54, s0=60, Lg=60, nu=(0.1, 0.02, 0.1))
    choose(monkeypatch, one=ALWAYS, chain=chain)
    a = gpu.Lbm3.from_workload(w, precision=precision)
    b = gpu.Lbm3.from_workload(w, precision=precision)
    angles = w.angles.reshape(-1, 3)[a.wall_nodes()]
    for n in (60, 120):
        a.step(n)
        for _ in range(n):
            b.set_wall_angles(angles)
            b.step(1)
        same(a, b)
    # there were traces to leave out, below the threshold of every storage, over many tiles
    r = np.abs(a.fields()[0])
    assert np.count_nonzero((r > 0) & (r < 1e-14)) > nx * ny // 16


# ---- a region of one fluid that diverges ----
# Opposed streams just below the largest float: within some steps populations overflow, in the middle of
# tiles whose words name that fluid alone.  What the collision makes of them -- infinities, NaN -- spreads
# to the absent fluids and, through a density without a fraction, to the wall values as it does in the
# general way (all words set to "all fluids" before every step).
@pytest.mark.parametrize("precision", [0, 2], ids=["fp32", "bf16"])
@pytest.mark.parametrize("chain,plain", [(NEVER, "0"), ("0", "0"), ("0", "1")], ids=["one-launch", "bulk", "plain"])
@pytest.mark.parametrize("y,x", [(30, 60), (52, 128)], ids=["away", "at-the-wall"])
def test_one_fluid_that_overflows(gpu, monkeypatch, precision, chain, plain, y, x):
    w = W.janus_cylinder(nx=256, ny=128, Rs=10.0, Rj=9.0, nu=(0.01, 0.01, 0.01))
    choose(monkeypatch, one=ALWAYS, chain=chain, plain=plain)
    a = gpu.Lbm3.from_workload(w, precision=precision)
    b = gpu.Lbm3.from_workload(w, precision=precision)
    angles = w.angles.reshape(-1, 3)[a.wall_nodes()]
    f, c = a.get_state()
    f[1, 1, y, x - 3:x + 3] += 1e35
    f[1, 3, y, x - 3:x + 3] -= 0.875e35
    finite = []
    for s in (a, b):
        s.set_state(f, c)
    for _ in range(12):
        b.set_wall_angles(angles)
        for s in (a, b):
            s.step(1)
        same(a, b)
        finite.append(bool(np.isfinite(a.fields()[0]).all()))
    assert finite[1] and not finite[-1]  # when it overflowed, words had come to name one fluid


# What a collision makes of a density just below the largest float, in the general way: infinities in the
# planes of one fluid, NaN in those of the absent ones, which the words of the next step must name.
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("chain", [NEVER, "0"], ids=["one-launch", "split"])
def test_words_after_an_overflow_in_the_general_way(gpu, monkeypatch, precision, chain):
    w = W.janus_cylinder(nx=256, ny=128, Rs=10.0, Rj=9.0, nu=(1.0, 1.0, 1.0))
    choose(monkeypatch, one=ALWAYS, chain=chain)
    a = gpu.Lbm3.from_workload(w, precision=precision)
    b = gpu.Lbm3.from_workload(w, precision=precision)
    angles = w.angles.reshape(-1, 3)[a.wall_nodes()]
    f, c = a.get_state()
    f[1, 1, 53, 127] = f[1, 3, 53, 129] = f[1, 2, 52, 128] = f[1, 2, 53, 128] = 1e38
    for s in (a, b):
        s.set_state(f, c)  # the words say "all fluids"
        s.step(1)
    assert not np.isfinite(a.fields()[0]).all()
    for _ in range(4):
        b.set_wall_angles(angles)
        for s in (a, b):
            s.step(1)
        assert np.array_equal(a.get_state()[1], b.get_state()[1], equal_nan=True)
        same(a, b)


# Densities +V and -V at rest stay there in a collision (at this viscosity 1 / tau = V / 3000, and what it
# takes of the rounded moments is far below the last bit); streamed, they cancel exactly at the two nodes that
# bracket the crossings of the characteristic lines of the wall node at the cylinder's lowest point: 16 + 1
# (its own populations, one of them back from the wall) - 4 x 4 + 1 - 2 thirty-sixths of V.  No fraction
# there, so the wall values change in that step, in which the words still name one fluid.
@pytest.mark.parametrize("chain", [NEVER, "0"], ids=["one-launch", "split"])
def test_a_density_that_vanishes_reaches_the_wall_at_once(gpu, monkeypatch, chain):
    w = W.janus_cylinder(nx=256, ny=128, Rs=10.0, Rj=9.0, nu=(1e3, 1e3, 1e3))
    assert w.solid[54, 128] and not w.solid[54, 127] and not w.solid[54, 129]
    choose(monkeypatch, one=ALWAYS, chain=chain)
    a = gpu.Lbm3.from_workload(w)
    b = gpu.Lbm3.from_workload(w)
    angles = w.angles.reshape(-1, 3)[a.wall_nodes()]
    f, c = a.get_state()
    weight = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, np.float32)
    for side in (-1, 1):
        x = 128 + side
        plus, minus = [(53, x), (54, x + side)], [(53, x - 1), (53, x + 1), (52, x), (54, x), (52, x - 1), (52, x + 1)]
        for sign, nodes in ((1.0, plus), (-1.0, minus)):
            for yy, xx in nodes:
                f[1, :, yy, xx] = sign * 2.0 ** -20 * weight
    for s in (a, b):
        s.set_state(f, c)
        s.step(1)
    # (lbm3_fields sums in another order, in which multiples of V / 36 are rounded on the way)
    assert np.abs(a.fields()[0][:, 53, [127, 129]]).max() < 2.0 ** -45 and np.isfinite(a.get_state()[0]).all()
    old = b.get_state()[1][1, 54, 128]
    for n in range(3):
        b.set_wall_angles(angles)
        for s in (a, b):
            s.step(1)
        if n == 0:
            assert b.get_state()[1][1, 54, 128] != old
        assert np.array_equal(a.get_state()[1], b.get_state()[1], equal_nan=True)
        same(a, b)


# ---- more boundary nodes in a tile's region than two passes of the wetting take ----
# 2 x 2 posts at a spacing of 3: every 36 x 12 region holds 192 boundary nodes, three passes of 64.  (In the
# oracle a disturbance of 1e-7 stays below 3e-7 over 80 steps of this set-up.)
@pytest.mark.parametrize("bc_x", [W.BC_PERIODIC, W.BC_MODPER], ids=["periodic", "seam"])
@pytest.mark.parametrize("chain", [NEVER, "0"], ids=["one-launch", "split"])
def test_three_passes_of_boundary_nodes_match_oracle(gpu, oracle_mod, monkeypatch, bc_x, chain):
    w = W.janus_cylinder(nx=72, ny=36, Rs=4.0, Rj=10.0, sigma=(0.01, 0.01, 0.01),
                         triple=(85.0, 75.0, 105.0) if bc_x == W.BC_PERIODIC else (90.0, 135.0, 45.0))
    w.solid[:] = 0
    for y in range(0, 36, 3):
        for x in range(0, 72, 3):
            w.solid[y:y + 2, x:x + 2] = 1
    w.rho[:, w.solid == 1] = 0.0
    w.rho[1][(w.rho.sum(0) == 0) & (w.solid == 0)] = 1.0
    w.bc_x = bc_x
    assert w.solid[6:18, 30:66].sum() == 192
    choose(monkeypatch, chain=chain)
    g = gpu.Lbm3.from_workload(w)
    o = oracle_mod.Oracle.from_workload(w)
    for n in (1, 2, 37):
        g.step(n)
        o.step(n)
        assert np.abs(g.fields()[0] - o.fields()[0]).max() <= TOL_RHO[0]
        assert np.abs(g.fields()[1] - o.fields()[1]).max() <= TOL_U


# ---- graphs, timed steps and states with the split launches ----
@pytest.mark.parametrize("precision", [0, 1], ids=["fp32", "fp16"])
@pytest.mark.parametrize("one", [NEVER, ALWAYS], ids=["two-launches", "four-launches"])
def test_split_steps_do_not_depend_on_the_call(gpu, monkeypatch, precision, one):
    choose(monkeypatch, one=one)
    sims = [gpu.Lbm3.from_workload(pillars(), precision=precision) for _ in range(3)]
    a, b, c = sims
    a.step(37)                 # graphs of eight steps, and single ones
    for _ in range(37):
        b.step(1)
    t = c.step_timed_detail(37)
    same(*sims)
    assert 0 < t[1] <= t[4] and 0 < t[2] <= t[4]
    for s in sims:             # captured arguments are dropped
        s.set_inflow(0.03)
    a.step(20)
    b.step(3)
    b.step(17)
    c.step_timed(20)
    same(*sims)
    f, w = a.get_state()
    for s, parts in ((a, (25,)), (b, (9, 16)), (c, (1, 24))):
        s.set_state(f, w)
        for n in parts:
            s.step(n)
    same(*sims)


# ---- times of launches that a step does not have ----
def test_times_of_the_launches_there_are(gpu, monkeypatch):
    """The wetting and the edge tiles have no launch of their own: exactly 0.  Where a step is one launch,
    it is all of the run, which the timing must not slow down with events between the steps."""
    choose(monkeypatch)
    t = gpu.Lbm3.from_workload(pillars()).step_timed_detail(20)
    assert t[0] == 0.0 and t[3] == 0.0 and 0.0 < t[1] <= t[4] and 0.0 < t[2] <= t[4]
    choose(monkeypatch, chain=NEVER)
    s = gpu.Lbm3.from_workload(pillars())
    t = s.step_timed_detail(20)
    assert t[:2] == (0.0, 0.0) and t[3] == 0.0 and t[2] == t[4] > 0.0
    assert s.step_timed(3)[:2] == (0.0, 0.0)


# ---- what a failed read-back leaves ----
def test_fields_that_fail_leave_the_arrays(gpu):
    """lbm3_fields cannot be captured (it waits for the device): it says so and writes nothing."""
    import torch
    w = pillars()
    stream = torch.cuda.Stream()
    sim = gpu.Lbm3.from_workload(w, stream=stream.cuda_stream)
    sim.step(3)
    want = sim.fields()
    rho, u = np.full(3 * w.n, 7.5), np.full(2 * w.n, -2.5)
    rt = ctypes.CDLL("libcudart.so.13")
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(handle, 1) == 0  # this thread's calls only
    code = gpu.load().lbm3_fields(sim._h, gpu._dp(rho), gpu._dp(u))
    rt.cudaStreamEndCapture(handle, ctypes.byref(graph))
    if graph.value:
        rt.cudaGraphDestroy(graph)
    rt.cudaGetLastError()
    assert code == gpu.LBM3_ERR_CUDA
    assert (rho == 7.5).all() and (u == -2.5).all()
    for p, q in zip(sim.fields(), want):
        assert np.array_equal(p, q)


# ---- SMs of the two-blocks-per-SM kernel ----
def test_the_kernel_that_takes_every_pure_tile_has_the_sms_for_it(gpu, monkeypatch):
    """The half of the SMs that the one-fluid launch gets on large grids is not taken from the kernel
    that leaves it no tile.  With 12 SMs left (the other tiles' share here) against half of 152, a step
    bound by that kernel takes up to 140 / 76 = 1.8 times as long; the line is drawn half way."""
    import torch
    nx, ny = 2048, 1024
    rho = np.zeros((3, ny, nx))
    rho[2] = 1.0
    w = W.Workload("box", nx, ny, 1, W.BC_PERIODIC, np.zeros((ny, nx), np.uint8), rho, np.full((ny, nx, 3), 90.0),
                   (0.01,) * 3, (0.1,) * 3)
    choose(monkeypatch, one="1200", chain="1200", pure="tma")
    monkeypatch.delenv("LBM3_SPARE_SMS", raising=False)
    a = gpu.Lbm3.from_workload(w)
    monkeypatch.setenv("LBM3_SPARE_SMS", "12")
    b = gpu.Lbm3.from_workload(w)
    assert a.info()["pure_kernel"] == "bulk copies" and a.info()["step_kernels"] == 2

    def time(s):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        e[0].record()
        s.step(65)
        e[1].record()
        torch.cuda.synchronize()
        return e[0].elapsed_time(e[1])

    for s in (a, b):
        s.step(40)
    ratio = sorted(time(a) / time(b) for _ in range(7))
    assert ratio[3] < 1.4


@pytest.mark.parametrize("precision", [0, 1], ids=["fp32", "fp16"])
def test_the_persistent_kernels_get_sms_back_when_every_tile_is_theirs(gpu, monkeypatch, precision):
    """All three fluids everywhere, as after a long run: no tile is the one-fluid launch's, and the SMs kept
    free for it (half of them, two fifths in the 16-bit storages) are the persistent kernel's.  With a fifth
    of 152 left from the start it has 122 SMs against 76 (92): 1.6 (1.33) times as fast where it bounds the
    step; the line is half of the smaller excess."""
    import torch
    nx, ny = 2048, 1024
    rho = np.empty((3, ny, nx))
    rho[0], rho[1], rho[2] = 0.3, 0.3, 0.4
    w = W.Workload("mixture", nx, ny, 1, W.BC_PERIODIC, np.zeros((ny, nx), np.uint8), rho,
                   np.full((ny, nx, 3), 90.0), (0.01,) * 3, (0.1,) * 3)
    choose(monkeypatch, one="1200", chain="1200")
    monkeypatch.delenv("LBM3_SPARE_SMS", raising=False)
    a = gpu.Lbm3.from_workload(w, precision=precision)
    monkeypatch.setenv("LBM3_SPARE_SMS", "30")
    b = gpu.Lbm3.from_workload(w, precision=precision)
    assert a.info()["tma"] and a.info()["step_kernels"] == 4

    def time(s):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        e[0].record()
        s.step(65)
        e[1].record()
        torch.cuda.synchronize()
        return e[0].elapsed_time(e[1])

    for s in (a, b):
        s.step(600)  # (the tiles are counted every 256 steps, and the count is taken when it has come)
        s.sync()
    ratio = sorted(time(a) / time(b) for _ in range(7))
    assert ratio[3] < 1.16


# the launch size changes between steps, with the state: the same bits
@pytest.mark.parametrize("precision", [0, 1], ids=["fp32", "fp16"])
def test_launch_sizes_that_follow_the_state(gpu, monkeypatch, precision):
    nx, ny = 1024, 512
    w = W.janus_cylinder(nx=nx, ny=ny, Rs=40.0, Rj=40.0)
    choose(monkeypatch, one="1200", chain="1200")
    monkeypatch.delenv("LBM3_SPARE_SMS", raising=False)
    a = gpu.Lbm3.from_workload(w, precision=precision)
    assert a.info()["step_kernels"] == 4
    monkeypatch.setenv("LBM3_SPARE_SMS", "30")
    b = gpu.Lbm3.from_workload(w, precision=precision)
    mixed = w.rho.copy()
    mixed[:, :, :600] = np.array([0.3, 0.3, 0.4])[:, None, None] * (w.solid[:, :600] == 0)
    for rho in (w.rho, mixed, w.rho):  # few tiles, more than 3/10 of them, few again
        for s in (a, b):
            s.set_fields(rho)
        for n in (270, 21, 1, 40):  # counted in the first, taken from the second on
            for s in (a, b):
                s.step(n)
            same(a, b)
