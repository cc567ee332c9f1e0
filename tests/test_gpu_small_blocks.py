"""Grids whose rows and planes hold fewer than 32 of a sweep's threads: whole
steps against the oracle, with its iteration counts in FP64 (the sums <r, z>
and <p, q> are reduced over such a block's lanes)."""
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


@pytest.mark.parametrize("n,periodic", [((8, 4, 4), (0, 0, 0)), ((4, 8, 3), (0, 1, 0)), ((16, 2, 4), (1, 0, 0)),
                                        ((2, 2, 2), (0, 0, 0)), ((6, 2, 10), (0, 0, 1)), ((1, 3, 5), (0, 0, 0))])
@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED])
def test_step_on_a_few_cells(fld, oracle, n, periodic, precision):
    case = synth.random_case(n, seed=61, periodic=tuple(map(bool, periodic)), E_decades=(-16, -14))
    case.params.precision = precision
    ctx = fld.fld_create(case.grid, case.params, rtol=1e-13 if precision == synth.PREC_FP64 else 1e-8)
    E = dev(case.E)
    info = fld.fld_step(ctx, E, dev(case.nHI), dev(case.eta))
    ctx.close()
    Eref, iref = oracle.step(case.grid, case.params, {"rtol": 1e-13, "max_iter": 200}, case.E, case.nHI, case.eta)
    got = E.cpu().numpy().reshape(case.grid.shape)
    tol = 1e-10 if precision == synth.PREC_FP64 else 1e-6
    assert np.abs(got - Eref).max() < tol * np.abs(Eref).max()
    if precision == synth.PREC_FP64:
        assert abs(info["iters"] - iref["iters"]) <= 1, (info, iref)


@pytest.mark.parametrize("n", [(16, 8, 32), (16, 6, 32)])
def test_mixed_step_without_the_tail(fld, oracle, n):
    # two threads of eight cells per row
    case = synth.random_case(n, seed=62, E_decades=(-16, -14))
    case.params.precision = synth.PREC_MIXED
    ctx = fld.fld_create(case.grid, case.params, tail_cells=0)
    E = dev(case.E)
    info = fld.fld_step(ctx, E, dev(case.nHI), dev(case.eta))
    ctx.close()
    assert info["rel_res"] <= 1e-8
    Eref, _ = oracle.step(case.grid, case.params, {"rtol": 1e-13, "max_iter": 200}, case.E, case.nHI, case.eta)
    got = E.cpu().numpy().reshape(case.grid.shape)
    assert np.abs(got - Eref).max() < 1e-6 * np.abs(Eref).max()
