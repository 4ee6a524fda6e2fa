"""FP32-mixed node update: a mesh stepped alone picks its tile height from its
size (1 to 8 node rows), a batch marches tiles of 8 rows or more.  The height
decides which warp marches a node, not the node's arithmetic, so the fields
and cracks of both are identical, bit for bit (needs a GPU)."""
import numpy as np
import pytest

from paper_2509_01827_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_01827_gb300 import build
    build.build()


# the heights these sizes take alone: 1, 1, 3, 4, 6 and 8 rows
@pytest.mark.parametrize("nx,ny,steps", [(59, 23, 260), (100, 40, 260), (512, 512, 40),
                                         (770, 767, 20), (1030, 1021, 12), (1440, 1450, 8)])
def test_solo_heights_equal_batch(nx, ny, steps):
    from paper_2509_01827_gb300.cem import CEM_FP32_MIXED, Batch, Solver
    p = inputs.notched_plate(nx, ny, traction=1e6 if nx == 100 else 2.5e6, phantom_cap=8000, crack_cap=4000)
    p.energy_every = 7
    a, c = Solver(p, precision=CEM_FP32_MIXED), Solver(p, precision=CEM_FP32_MIXED)
    rng = np.random.default_rng(nx)
    n = a.nodes()["vx"].size
    v = dict(vx=rng.standard_normal(n) * 0.05, vy=rng.standard_normal(n) * 0.05)
    for s in (a, c):
        s.set_state(**v)
    a.step(steps)
    b = Batch([c])
    b.set_config(16, 152)
    b.step(steps)
    na, nc = a.nodes(), c.nodes()
    for k in ("ux", "uy", "vx", "vy", "m"):
        np.testing.assert_array_equal(na[k], nc[k], err_msg=k)
    ca, cc = a.cracks(), c.cracks()
    for k in ("elem", "ka", "kb", "step", "nodes"):
        np.testing.assert_array_equal(ca[k], cc[k], err_msg=k)
    # the records differ by the grouping of FP32 partial sums at most: sums of
    # non-negative terms, each partial of a few thousand terms rounded once a term
    ea, ec = a.energy(), c.energy()
    for k in ("KE", "SE"):
        np.testing.assert_allclose(ea[k], ec[k], rtol=4096 * 2.0 ** -24, err_msg=k)
    b.close()


@pytest.mark.parametrize("mode", ["neumann", "dirichlet"])
def test_loaded_edges_up_a_tile(mode):
    """A plate with a loaded hole (or driven outer edges): columns of loaded
    nodes run up the tiles, up to 64 to a tile column and so more than a lane
    lists at a time.  Every tile height gives the same fields."""
    from paper_2509_01827_gb300.cem import CEM_FP32_MIXED, Batch, Solver
    p = inputs.fragmentation(n=130, r=0.02, mode=mode, phantom_cap=8000, crack_cap=4000)
    want = None
    for rows in (0, 8, 32, 64):
        s = Solver(p, precision=CEM_FP32_MIXED)
        if rows:
            b = Batch([s])
            b.set_config(rows, 152)
            b.step(60)
        else:
            s.step(60)
        got = s.nodes()
        assert np.max(np.abs(got["vx"])) > 0
        want = want or got
        for k in ("ux", "uy", "vx", "vy", "m"):
            np.testing.assert_array_equal(got[k], want[k], err_msg=k)
        if rows:
            b.close()


def test_large_mesh_evaluation_equals_batch():
    """Above two million nodes a plate stepped alone evaluates a thread per
    surface point, a batch always a warp per candidate path: cracks and fields
    of a breaking plate are the same."""
    from paper_2509_01827_gb300.cem import CEM_FP32_MIXED, Batch, Solver
    p = inputs.fragmentation(n=1500, p0=80e6, phantom_cap=40000, crack_cap=20000)
    a, c = Solver(p, precision=CEM_FP32_MIXED), Solver(p, precision=CEM_FP32_MIXED)
    a.step(330)
    b = Batch([c])
    b.step(330)
    assert a.counts()["n_cracked"] > 0
    na, nc = a.nodes(), c.nodes()
    for k in ("ux", "uy", "vx", "vy", "m"):
        np.testing.assert_array_equal(na[k], nc[k], err_msg=k)
    ca, cc = a.cracks(), c.cracks()
    for k in ("elem", "ka", "kb", "step"):
        np.testing.assert_array_equal(ca[k], cc[k], err_msg=k)
    b.close()
