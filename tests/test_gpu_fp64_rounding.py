"""The FP64 step rounds as it always has.

On fine grids the scheme amplifies a difference of one unit in the last place by many
orders of magnitude (1e10 for a Sod tube of 8192 cells in 500 steps), so the fields of a
run, and Delta* even after a few tens of steps, are reproducible only with the same
rounding in every operation.  tests/golden/fp64_runs.txt holds digests of states recorded
from the stage kernels whose every operation ran on the FP64 pipe; the kernels that take
sums and differences on the integer pipes must give the same bits.  The inputs come from
uniform draws and constants alone (no libm), so they are the same on every host.

The shapes reach every form of the stage: a cell on one, two and 16 threads, in the
cluster, on 1-D and 2-D grids, with rows that are no multiple of a warp."""
import ctypes
import hashlib
import os

import numpy as np
import pytest

from paper_2502_16818_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fp64_runs.txt")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_16818_gb300 import _build
    _build.build()
    torch.cuda.set_device(0)


def blocks(nx, ny, bc, I=1.0, vset=W.VSET_SOUND):
    w = W.random_blocks(nx, ny, seed=nx + ny, I=I, vset=vset, bc=bc)
    w.dt = 0.2 / max(nx, ny) / 2.2
    w.tau = 4 * w.dt
    return w


def sod(nx, I):
    w = W.sod(nx, I=I)
    w.dt = min(w.dt, 0.4 * w.dx / max(w.vg))
    return w


RUNS = {                                                     # workload, integrator, steps
    "130x67": (lambda: blocks(130, 67, (0, 1)), 0, 40),
    "130x67 midpoint": (lambda: blocks(130, 67, (1, 0), I=0.0), 1, 40),
    "180x190": (lambda: blocks(180, 190, (0, 0), I=3.0), 0, 30),
    "301x260": (lambda: blocks(301, 260, (1, 1)), 0, 30),
    "33x700": (lambda: blocks(33, 700, (0, 0), I=3.0, vset=W.VSET_TGV), 0, 20),
    "sod 500": (lambda: sod(500, 0.0), 0, 200),
    "sod 8192": (lambda: sod(8192, 1.0), 0, 300),
    "tube 37": (lambda: blocks(37, 1, (1, 0)), 1, 60),
    "tube 3001": (lambda: blocks(3001, 1, (0, 0), I=3.0), 0, 40),
    "tube 9001": (lambda: blocks(9001, 1, (1, 0)), 0, 40),
    "tube 26000": (lambda: blocks(26000, 1, (0, 0)), 0, 30),
    "tube 60001": (lambda: blocks(60001, 1, (0, 0), I=0.0), 0, 20),
}


def digests(name, small=None):
    """SHA-256 of the state's and of the fields' bytes after the run."""
    from paper_2502_16818_gb300 import Solver, cdbm
    make, rk, steps = RUNS[name]
    w = make()
    s = Solver.from_workload(w, rk=rk)
    if small is not None:
        cdbm.cdbm_set_small_grid_path(s.ctx, small)
    s.init(w.rho, w.ux, w.uy, w.T)
    s.step(steps)
    s.sync()
    # + 0.0: the sign of an exact zero is left open
    out = [hashlib.sha256((a.cpu().numpy() + 0.0).tobytes()).hexdigest() for a in (s.state(), torch.stack(s.macros()))]
    s.close()
    return out


def golden():
    with open(GOLDEN) as fh:
        rows = [line.split() for line in fh if line.strip() and not line.startswith("#")]
    return {" ".join(r[:-2]): r[-2:] for r in rows}


@pytest.mark.parametrize("name", list(RUNS))
def test_state_has_the_recorded_bits(name):
    assert digests(name) == golden()[name]


@pytest.mark.parametrize("name", list(RUNS))
def test_every_form_gives_the_same_bits(name):
    assert digests(name, small=0) == digests(name, small=1)


def test_batch_has_the_bits_of_single_tubes():
    """The FP64 ensemble, with and without transverse velocity, against each tube alone."""
    from paper_2502_16818_gb300 import BatchSolver, Solver
    for uy in (False, True):
        tubes = [blocks(n, 1, (1, 0)) for n in (1, 31, 500, 2000, 8192, 9001)]
        for t in tubes:
            t.dt, t.tau, t.dx = 1e-5, 4e-5, 1.0 / 9001
            if not uy:
                t.uy = np.zeros_like(t.uy)
        b = BatchSolver(tubes)
        b.init(tubes)
        b.step(25)
        b.sync()
        out = b.macros()
        for k, t in enumerate(tubes):
            s = Solver.from_workload(t)
            s.init(t.rho, t.ux, t.uy, t.T)
            s.step(25)
            s.sync()
            for x, y in zip(b.tube(out, k), s.macros()):
                assert np.array_equal(x, y.cpu().numpy()[0]), (uy, k)
            s.close()
        b.close()


@pytest.mark.parametrize("nx,ny", [(131, 67), (500, 1), (3001, 1), (226, 220)])
def test_adjoint_is_the_same_from_every_form(nx, ny):
    """The recorded run is cdbm_step's, and its recomputed segments have its bits whatever
    form takes them: ragged grids, tubes in the cluster and beyond."""
    from paper_2502_16818_gb300 import Solver, cdbm
    w = blocks(nx, ny, (0, 0))
    got = []
    for small in (1, 0):
        s = Solver.from_workload(w)
        cdbm.cdbm_set_small_grid_path(s.ctx, small)
        s.init(w.rho, w.ux, w.uy, w.T)
        s.step(7)
        plain = s.state().clone()
        s.init(w.rho, w.ux, w.uy, w.T)
        cdbm.cdbm_adjoint_forward(s.ctx, 7, 3)
        assert torch.equal(s.state(), plain)
        fbar = torch.ones((16, ny, nx), dtype=torch.float64, device="cuda") * 0.25
        grads = [torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(4)]
        tau = cdbm.cdbm_adjoint_backward(s.ctx, fbar.data_ptr(), *(g.data_ptr() for g in grads))
        got.append((grads, tau))
        s.close()
    assert got[0][1] == got[1][1] and all(torch.equal(a, b) for a, b in zip(got[0][0], got[1][0]))


@pytest.mark.parametrize("nx,ny", [(37, 1), (500, 1), (3001, 1), (9001, 1), (131, 67)])
def test_step_noalloc_has_the_bits_of_step(nx, ny):
    from paper_2502_16818_gb300 import Solver, cdbm
    w = blocks(nx, ny, (1, 0))
    s = Solver.from_workload(w)
    s.init(w.rho, w.ux, w.uy, w.T)
    f = s.state().clone()
    s.step(9)
    grid = cdbm.cdbm_grid(w.nx, w.ny, w.dx, w.dy, w.bc_x, w.bc_y)
    vset = cdbm.cdbm_vset((ctypes.c_double * 4)(*w.vg), (ctypes.c_double * 4)(*w.eg))
    cdbm.cdbm_step_noalloc(grid, vset, w.I, w.tau, w.dt, f.data_ptr(), 9, torch.cuda.current_stream().cuda_stream)
    assert torch.equal(f, s.state())
    s.close()
