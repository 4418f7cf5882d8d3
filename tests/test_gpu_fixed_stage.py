"""FP64 stage kernels in fixed point (csrc/cdbm_stage_fx.cuh) where they can go wrong:
widths around the block sizes, values of both signs over many binades side by side,
zeros, and values outside the exponents of the integer path.  One step from a given state,
by the one-thread-per-cell kernel and by the kernels with a cell on 16 or two threads
(equal bit for bit; tubes of up to 1024 cells in the cluster kernel), against the CPU
oracle.

Bound: the oracle and the kernels each round a cell's update a few tens of times (the
oracle's linear solve included) relative to the largest value that enters it -- the cell
and its neighbours up to two away -- so they agree to 256 units of 2^-53 of it, times the
condition of the moment system (about 10 for this velocity set's blocks)."""
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


def state(kind, nx, ny, bc, seed):
    # side by side densities 60 binades apart do not stay physical: transport alone there
    w = W.random_blocks(nx, ny, seed=seed, dt=min(2e-4, 0.3 / max(nx, ny)), tau=1e30 if kind == "wide" else 1e-3, bc=(bc, bc))
    m = oracle.Model(w.nx, w.ny, w.dx, w.dy, w.dt, w.tau, w.I, w.vg, w.eg, w.bc_x, w.bc_y)
    f = np.asarray(oracle.init(m, w.rho, w.ux, w.uy, w.T)).reshape(16, ny, nx).copy()
    rng = np.random.default_rng(seed)
    if kind == "wide":                  # the density of neighbouring cells over 60 binades
        f *= np.exp2(rng.integers(-30, 31, (ny, nx)))
    elif kind == "zeros":               # the lightest group: zero, tiny and ordinary values side by side
        f[:4] *= rng.choice([0.0, 1e-300, 1e-12, 1.0], (4, ny, nx))
    elif kind == "tiny":                # below the exponents of the integer path
        f *= 2.0 ** -920
    return w, m, f


@pytest.mark.parametrize("nx,ny", [(31, 9), (33, 5), (129, 4), (257, 3), (1, 40), (130, 1), (4097, 1), (127, 110), (225, 220),
                                   (26000, 1), (65, 1030)])
@pytest.mark.parametrize("kind,bc", [("plain", 0), ("wide", 1), ("wide", 0), ("zeros", 1), ("tiny", 0)])
def test_one_step(nx, ny, kind, bc):
    from paper_2502_16818_gb300 import Solver, cdbm
    w, m, f = state(kind, nx, ny, bc, 11)
    got = []
    for small in (1, 0):
        s = Solver.from_workload(w)
        cdbm.cdbm_set_small_grid_path(s.ctx, small)
        s.set_state(f)
        s.step(1)
        got.append(s.state().cpu().numpy().reshape(16, ny, nx))
        s.close()
    assert np.array_equal(got[0], got[1])
    ref = np.asarray(oracle.step(m, f, 1)).reshape(16, ny, nx)
    mode = "wrap" if bc == 0 else "edge"
    big = np.abs(f).max(0)
    near = big.copy()                   # a step's two stages reach 4 cells
    for ax in (0, 1):
        pad = np.pad(near, [(4, 4) if a == ax else (0, 0) for a in (0, 1)], mode=mode)
        near = np.max([np.take(pad, range(k, k + near.shape[ax]), axis=ax) for k in range(9)], axis=0)
    assert np.all(np.abs(got[1] - ref) <= 10 * 256 * 2.0 ** -53 * near)
    assert np.all(np.abs(got[0] - ref) <= 10 * 256 * 2.0 ** -53 * near)
