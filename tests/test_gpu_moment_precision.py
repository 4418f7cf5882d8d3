"""Read-out of cells whose mass sits in slow velocity groups, for velocity sets whose groups
differ widely: the fast groups' tiny values must not cost the moments their precision.

The cells are symmetric (equal members per group), so u = 0 and every moment is a sum of a
few positive terms, evaluated exactly with rationals.  Bounds: the double-precision sums
round their terms up to six times; T takes six operations more (energy minus rho u^2,
1 / K and its product, the reciprocal of rho within 2 units, its product), 14 units of
2^-53 in all, held to 16.  An entry of Delta* is the difference of a raw moment (6 units)
and of p or (K + 2) p^2 / rho (two p's of 10 units and four operations: 24), held to 32
units of the sum of the two."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2502_16818_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = Fraction(1, 2 ** 53)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_16818_gb300 import _build
    _build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("vset", [((0.02, 0.02, 3.0, 3.0), (0.0, 20.0, 0.0, 2.6)), W.VSET_TGV, W.VSET_SOD, W.VSET_SOUND])
@pytest.mark.parametrize("heavy", [0, 1, 2, 3])
@pytest.mark.parametrize("light", [1e-13, 1e-6, 1.0])
def test_moments_and_tne(vset, heavy, light):
    from paper_2502_16818_gb300 import Solver
    nx, ny, I = 16, 4, 1.0
    rng = np.random.default_rng(heavy)
    q = light * rng.uniform(0.1, 1.0, (4, ny, nx))
    q[heavy] = rng.uniform(0.5, 1.0, (ny, nx))
    f = np.repeat(q, 4, axis=0)
    w = W.random_blocks(nx, ny, seed=1, I=I, dt=1e-4, tau=1e-3, vset=vset)
    s = Solver.from_workload(w)
    s.set_state(np.ascontiguousarray(f))
    rho, ux, uy, T = (a.cpu().numpy() for a in s.macros())
    tne = s.tne().cpu().numpy()
    s.close()
    assert not ux.any() and not uy.any()
    v, e = ([Fraction(x) for x in a] for a in vset)
    K = 2 + Fraction(I)
    for y in range(ny):
        for x in range(nx):
            g = [Fraction(float(a)) for a in q[:, y, x]]
            two = [2 if k % 2 == 0 else 4 for k in range(4)]                   # members with v_x != 0
            W2 = [(1 if k % 2 == 0 else 2) * v[k] ** 2 + e[k] ** 2 for k in range(4)]
            r = sum(4 * a for a in g)
            p = sum(4 * a * b for a, b in zip(g, W2)) / K
            assert abs(Fraction(float(rho[y, x])) - r) <= 6 * U * r
            assert abs(Fraction(float(T[y, x])) - p / r) <= 16 * U * p / r
            Rxx = sum(two[k] * g[k] * v[k] ** 2 for k in range(4))
            Rwxx = sum(two[k] * g[k] * W2[k] * v[k] ** 2 for k in range(4))
            for row, R, m in ((0, Rxx, p), (2, Rxx, p), (9, Rwxx, (K + 2) * p * p / r), (11, Rwxx, (K + 2) * p * p / r)):
                assert abs(Fraction(float(tne[row, y, x])) - (R - m)) <= 32 * U * (R + m), (row, y, x)
