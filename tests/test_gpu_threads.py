"""Contexts of different sizes stepped at the same time from two threads (each
with a stream of its own): every step succeeds and gives, bit for bit, what the
context gives alone.  The sizes of a pair share the kernels of the coarsest
grid's inverse (702 and 693 cells, 128 and 125 cells) but not the shared memory
these need."""
import threading

import numpy as np
import pytest

from paper_1306_0645_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fld():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1306_0645_gb300 import fld as f
    f.lib()
    return f


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64).ravel()).cuda()


class Stepper:
    def __init__(self, fld, n, precision):
        self.fld = fld
        case = synth.random_case(n, seed=71, E_decades=(-16, -14))
        case.params.precision = precision
        self.stream = torch.cuda.Stream()
        with torch.cuda.stream(self.stream):
            self.E0, self.nHI, self.eta = dev(case.E), dev(case.nHI), dev(case.eta)
            self.E = self.E0.clone()
        self.stream.synchronize()
        self.ctx = fld.fld_create(case.grid, case.params, stream=self.stream)

    def step(self):
        with torch.cuda.stream(self.stream):
            self.E.copy_(self.E0)
            self.fld.fld_step(self.ctx, self.E, self.nHI, self.eta)
        self.stream.synchronize()
        return self.E


@pytest.mark.parametrize("sizes", [((52, 36, 24), (44, 36, 28)), ((16, 16, 32), (10, 10, 10))])
@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED])
def test_two_threads_with_different_coarsest_grids(fld, sizes, precision):
    steppers = [Stepper(fld, n, precision) for n in sizes]
    alone = [s.step().clone() for s in steppers]
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(steppers))

    def work(s, ref):
        try:
            start.wait()
            for q in range(300):
                if not torch.equal(s.step(), ref):
                    raise AssertionError(f"step {q} differs from the step alone")
        except Exception as e:          # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=a) for a in zip(steppers, alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s in steppers:
        s.ctx.close()
    assert not errors, errors
