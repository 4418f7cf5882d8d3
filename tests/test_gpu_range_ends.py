"""States at the ends of the exponent range are physical: a step from densities of 2^-1010 or
2^900 raises no flag, in any form of the FP64 stage and in the ensemble."""
import numpy as np
import pytest

import oracle
from paper_2502_16818_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_16818_gb300 import _build
    _build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("nx,ny", [(500, 1), (3001, 1), (33, 40), (180, 190), (225, 220)])
@pytest.mark.parametrize("exponent", [-1010, 900])
def test_step_raises_no_flag(nx, ny, exponent):
    from paper_2502_16818_gb300 import Solver
    w = W.random_blocks(nx, ny, seed=nx, dt=0.1 / max(nx, ny), tau=0.1 / max(nx, ny))
    m = oracle.Model(w.nx, w.ny, w.dx, w.dy, w.dt, w.tau, w.I, w.vg, w.eg, w.bc_x, w.bc_y)
    f = np.asarray(oracle.init(m, w.rho, w.ux, w.uy, w.T)).reshape(16, ny, nx) * 2.0 ** exponent
    s = Solver.from_workload(w)
    s.set_state(f)
    s.step(1)
    s.sync()
    assert np.isfinite(s.state().cpu().numpy()).all()
    s.close()


@pytest.mark.parametrize("uy", [0.0, 0.05])
@pytest.mark.parametrize("exponent", [-1010, 900])
def test_batch_raises_no_flag(uy, exponent):
    from paper_2502_16818_gb300 import BatchSolver
    tubes = [W.random_blocks(n, 1, seed=n, dt=1e-5, tau=1e-3, bc=(1, 0)) for n in (100, 700, 2001)]
    for t in tubes:
        t.dx, t.rho, t.uy = 1e-3, t.rho * 2.0 ** exponent, np.full_like(t.uy, uy)
    b = BatchSolver(tubes)
    b.init(tubes)
    b.step(1)
    b.sync()
    assert all(np.isfinite(a).all() for a in b.macros())
    b.close()
