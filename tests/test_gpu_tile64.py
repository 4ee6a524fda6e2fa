"""The FP64 node update over its tile shapes and value ranges, against the
oracle bit for bit (needs a GPU)."""
import numpy as np
import pytest

from oracle.oracle import from_problem
from paper_2509_01827_gb300 import inputs
from tests._parity import compare_energy, compare_fp64

pytestmark = pytest.mark.gpu


# meshes one node below, at and above a tile's width or height, from one tile
# to the shape of large meshes; a field of ordinary size, and fields whose
# element sums are subnormal or straddle the range of the exponent arithmetic
# (2^-800 = 1.5e-241) inside one tile
@pytest.mark.parametrize("scale", [1.0, 1e-236, 1e-306])
@pytest.mark.parametrize("nx,ny,square", [(3, 2, True), (14, 2, False), (15, 7, True), (16, 12, False),
                                          (31, 33, True), (64, 23, False), (191, 95, True),
                                          (401, 161, False)])
def test_tiles_and_ranges(nx, ny, square, scale):
    from paper_2509_01827_gb300.cem import Solver
    rng = np.random.default_rng(nx)
    p = inputs.notched_plate(nx, ny, lx=nx * 1e-3, ly=ny * (1e-3 if square else 0.7e-3),
                             notch_len=min(nx // 3, 10) * 1e-3, traction=2e6 * scale,
                             phantom_cap=8 * nx * ny + 64, crack_cap=nx * ny + 16)
    p.energy_every = 3
    if nx >= 31:  # a hole
        act = np.ones((ny, nx), np.uint8)
        act[1:4, nx // 2 + 3:nx // 2 + 8] = 0
        p.active = act.reshape(-1)
    o, g = from_problem(p), Solver(p)
    n = o.counts()["nn"] + o.counts()["n_phantom"]
    # amplitudes over twelve decades side by side
    amp = scale * 10.0 ** rng.uniform(-12, 0, n)
    st = {k: rng.standard_normal(n) * amp * a for k, a in (("ux", 1e-8), ("uy", 1e-8),
                                                            ("vx", 0.3), ("vy", 0.3))}
    o.set_state(**st)
    g.set_state(**st)
    for steps in (1, 12):
        o.step(steps)
        g.step(steps)
        compare_fp64(o, g)
    if scale == 1.0:
        compare_energy(o, g)
