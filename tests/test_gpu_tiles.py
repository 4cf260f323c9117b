"""The kernel of the tiles near solids and domain edges (wetting included) against the FP64 oracle where
its lists and regions can go wrong: narrow last tiles, wrapped halos, thick walls whose boundary nodes
lie in tiles without a fluid node, tiles with more boundary nodes than one pass wets, open columns."""
import numpy as np
import pytest

from paper_2102_04709_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# as the parity tests: FP32 against FP64
TOL_RHO, TOL_U, STEPS = 1e-5, 1e-6, 120


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2102_04709_gb300 import build, lbm3
    build.build()
    lbm3.load()
    return lbm3


def posts(nx, ny, bc_x, triple=(85.0, 75.0, 105.0)):
    """A Janus droplet among 3 x 3 posts on a lattice of spacing 6: up to 8 boundary nodes per 36."""
    w = W.janus_cylinder(nx=nx, ny=ny, Rs=4.0, Rj=10.0, triple=triple, sigma=(0.01, 0.01, 0.01))
    w.solid[:] = 0
    for y in range(2, ny - 3, 6):
        for x in range(2, nx - 3, 6):
            w.solid[y:y + 3, x:x + 3] = 1
    w.rho[:, w.solid == 1] = 0.0
    fluid = (w.rho.sum(0) == 0) & (w.solid == 0)
    w.rho[1][fluid] = 1.0
    w.bc_x = bc_x
    return w


def case(name):
    if name.startswith("flat"):        # last tile 1, 2, 3 or 31 columns and 1, 3 or 7 rows wide
        nx, ny = {"flat_65x41": (65, 41), "flat_66x43": (66, 43), "flat_67x47": (67, 47), "flat_95x40": (95, 40)}[name]
        return W.janus_flat(nx=nx, ny=ny, R=11.0, triple=(80.0, 60.0, 110.0), sigma=(0.012, 0.009, 0.011))
    if name == "capillary_thick":      # walls of 11 rows: their boundary row lies in solid tiles
        return W.capillary(nx=97, ny=46, y_lo=11, y_hi=35, s0=24, Lg=24, nu=(0.1, 0.02, 0.1))
    if name == "capillary_narrow":     # 1 column of a third tile, at the seam
        return W.capillary(nx=65, ny=19, y_lo=1, y_hi=18, s0=16, Lg=16, nu=(0.1, 0.05, 0.1))
    if name == "posts_periodic":       # 200 boundary nodes in a tile's region: four passes
        return posts(72, 36, W.BC_PERIODIC)
    if name == "posts_seam":
        w = posts(72, 36, W.BC_MODPER, (90.0, 135.0, 45.0))
        w.periodic_y = 1
        return w
    # open columns, last tile 1 column wide
    return W.pillars(nx=129, ny=49, count=3, r_lo=5.0, r_hi=8.0, x_lo=45.0, x_hi=105.0, gap=6.0, seed=3,
                     drop=(24.0, 24.0), r_core=6.0, r_shell=12.0, theta_range=(60.0, 120.0), u_in=0.02)


@pytest.mark.parametrize("name", ["flat_65x41", "flat_66x43", "flat_67x47", "flat_95x40", "capillary_thick",
                                  "capillary_narrow", "posts_periodic", "posts_seam", "pillars_narrow"])
def test_tiles_match_oracle(gpu, oracle_mod, name):
    w = case(name)
    g = gpu.Lbm3.from_workload(w)
    o = oracle_mod.Oracle.from_workload(w)
    g.step(STEPS)
    o.step(STEPS)
    rg, ug = g.fields()
    ro, uo = o.fields()
    assert np.abs(rg - ro).max() <= TOL_RHO
    assert np.abs(ug - uo).max() <= TOL_U


@pytest.mark.parametrize("precision", [0, 1], ids=["fp32", "fp16"])
def test_new_wall_angles_take_effect_at_once(gpu, precision):
    """The lines of the next step are looked for at the end of a step: new angles must replace them."""
    w = W.janus_cylinder(nx=96, ny=90, Rs=16.0, Rj=14.0)
    a = gpu.Lbm3.from_workload(w, precision=precision)
    a.step(20)
    f, c = a.get_state()
    angles = w.angles.copy()
    angles[..., 0], angles[..., 2] = 70.0, 110.0
    nodes = a.wall_nodes()
    a.set_wall_angles(angles.reshape(-1, 3)[nodes])
    w.angles = angles
    b = gpu.Lbm3.from_workload(w, precision=precision)
    b.set_state(f, c)
    a.set_state(f, c)
    a.step(15)
    b.step(15)
    assert np.array_equal(a.get_state()[0], b.get_state()[0])
    a.set_wall_angles(angles.reshape(-1, 3)[nodes])
    a.step(15)
    b.step(15)
    assert np.array_equal(a.get_state()[0], b.get_state()[0])
