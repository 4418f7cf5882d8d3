"""cdbm_batch_init takes device fields as they are once the work already queued on the
default stream has run, whatever stream the batch works on and wherever the other fields
live."""
import ctypes

import numpy as np
import pytest

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


@pytest.mark.parametrize("precision", [0, 1, 2, 3])
@pytest.mark.parametrize("host", [(2,), (0, 2, 3), (0, 1, 3), (), (0, 1, 2, 3)])
def test_fields_written_on_the_default_stream(precision, host):
    from paper_2502_16818_gb300 import BatchSolver, cdbm
    tubes = [W.ensemble_tube({"nx": n, "rho": (1.0, 0.4), "T": (1.0, 0.8), "I": 1.0}) for n in (300, 1000)]
    fields = [np.concatenate([getattr(t, k).reshape(-1) for t in tubes]) for k in ("rho", "ux", "uy", "T")]
    ref = BatchSolver(tubes, precision=precision)
    ref.init(tubes)
    ref.step(2)
    want = ref.macros()
    ref.close()
    b = BatchSolver(tubes, precision=precision, stream=torch.cuda.Stream())
    late = [torch.from_numpy(a).cuda() for a in fields]
    dev = [torch.full_like(a, 0.5) for a in late]
    torch.cuda.synchronize()
    torch.cuda._sleep(200_000_000)                 # 0.1 s ahead of the writes below
    for d, a in zip(dev, late):
        d.copy_(a)
    ptr = [fields[k].ctypes.data if k in host else dev[k].data_ptr() for k in range(4)]
    cdbm.cdbm_batch_init(b.b, *ptr)
    b.step(2)
    got = b.macros()
    b.close()
    for x, y in zip(got, want):
        assert np.array_equal(x, y)
