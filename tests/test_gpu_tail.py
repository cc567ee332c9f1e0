"""The coarse tail's ways of running a level (one CTA in shared memory, halo
slabs of the cluster, phase by phase; the coarsest grid by one CTA or by the
cluster) against the same cycle with one launch per sweep: every slab axis,
boundary mix and remainder of planes over the CTAs, both precisions, and the
sweep counts that only some of the ways take."""
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


def cycle(fld, case, **over):
    ctx = fld.fld_create(case.grid, case.params, precond_bf16=0, **over)
    fld.fld_assemble(ctx, dev(case.E), dev(case.nHI), dev(case.eta))
    r = np.random.default_rng(5).standard_normal(case.grid.cells)
    z = torch.empty(case.grid.cells, dtype=torch.float64, device="cuda")
    fld.fld_vcycle(ctx, dev(r), z)
    ctx.close()
    return z.cpu().numpy()


GRIDS = [((32, 32, 32), (0, 0, 0)), ((32, 32, 32), (1, 1, 1)), ((16, 16, 16), (0, 1, 0)), ((6, 6, 6), (0, 0, 1)),
         ((64, 20, 12), (1, 0, 1)), ((12, 40, 8), (0, 1, 0)), ((20, 28, 48), (0, 0, 1)), ((22, 18, 14), (0, 0, 0)),
         ((128, 16, 16), (1, 0, 0)), ((8, 8, 128), (0, 1, 1)), ((18, 14, 10), (1, 0, 0)), ((36, 28, 20), (0, 0, 0))]


@pytest.mark.parametrize("n,periodic", GRIDS)
@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED])
def test_tail_is_the_cycle_of_separate_launches(fld, n, periodic, precision):
    case = synth.random_case(n, seed=41, periodic=tuple(map(bool, periodic)))
    case.params.precision = precision
    got, ref = cycle(fld, case), cycle(fld, case, tail_cells=0)
    # the same operations in another order: the rounding of one cycle
    assert np.max(np.abs(got - ref)) < (1e-12 if precision == synth.PREC_FP64 else 1e-5) * np.max(np.abs(ref))


@pytest.mark.parametrize("n", [(32, 24, 20), (16, 12, 20)])
@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED])
@pytest.mark.parametrize("over", [dict(pre=2, post=2), dict(pre=1, post=2), dict(pre=0, post=1), dict(pre=1, post=0),
                                  dict(pre=3, post=1, paper_order=1), dict(paper_order=1)])
def test_tail_with_other_sweeps(fld, n, precision, over):
    case = synth.random_case(n, seed=43, periodic=(False, True, False))
    case.params.precision = precision
    got, ref = cycle(fld, case, **over), cycle(fld, case, tail_cells=0, **over)
    assert np.max(np.abs(got - ref)) < (1e-12 if precision == synth.PREC_FP64 else 1e-5) * np.max(np.abs(ref))


@pytest.mark.parametrize("n,over", [((16, 16, 16), {}), ((20, 20, 20), {}), ((16, 24, 20), {}),
                                    ((16, 16, 16), dict(pre=2, post=2)), ((12, 10, 14), dict(paper_order=1))])
def test_single_cta_solve_is_the_launched_solve(fld, n, over):
    case = synth.random_case(n, seed=44, periodic=(True, False, False), E_decades=(-16, -14))
    case.params.precision = synth.PREC_MIXED
    out = []
    for cells in (0, 8192):
        ctx = fld.fld_create(case.grid, case.params, persistent_cells=cells, **over)
        E = dev(case.E)
        info = fld.fld_step(ctx, E, dev(case.nHI), dev(case.eta))
        ctx.close()
        assert info["rel_res"] <= 1e-8
        out.append(E.cpu().numpy())
    # both meet the tolerance of the paper's solver (1e-8 in the residual)
    assert np.linalg.norm(out[0] - out[1]) < 1e-6 * np.linalg.norm(out[0])
