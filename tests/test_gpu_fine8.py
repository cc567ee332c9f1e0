"""The red/black compressed sweeps (bfloat16 coefficients, x extent a multiple
of 8): rows of two threads, of a remainder of a block, of more than one block,
one-plane and many-plane chunks, every boundary mix.  The cycle must be a
symmetric positive definite operator to FP32 rounding, which fails for any
wrong neighbour or weight, and the FP32-coefficient cycle of the one-launch-
per-sweep kernels up to the coefficients' rounding (2^-9)."""
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


@pytest.mark.parametrize("n,periodic,dirichlet", [
    ((16, 12, 20), (0, 0, 0), False), ((16, 16, 16), (1, 1, 1), False), ((24, 20, 28), (1, 0, 0), False),
    ((40, 6, 10), (0, 1, 0), False), ((272, 8, 12), (0, 0, 1), False), ((288, 12, 8), (1, 0, 0), False),
    ((48, 80, 16), (0, 1, 1), False), ((192, 96, 128), (0, 0, 0), False), ((320, 96, 80), (1, 1, 0), False), ((64, 64, 64), (0, 0, 0), True), ((128, 96, 160), (0, 0, 0), False)])
def test_compressed_cycle_is_symmetric(fld, n, periodic, dirichlet):
    case = synth.random_case(n, seed=51, periodic=tuple(map(bool, periodic)))
    if dirichlet:
        case.grid = case.grid.outflow_upper()
    case.params.precision = synth.PREC_MIXED
    rng = np.random.default_rng(6)
    x, y = rng.standard_normal((2, case.grid.cells))
    out = {}
    for bf16 in (1, 0):
        ctx = fld.fld_create(case.grid, case.params, precond_bf16=bf16, tail_cells=256,
                             coarse_cap=4096)
        fld.fld_assemble(ctx, dev(case.E), dev(case.nHI), dev(case.eta))
        z = torch.empty(case.grid.cells, dtype=torch.float64, device="cuda")
        out[bf16] = []
        for v in (x, y):
            fld.fld_vcycle(ctx, dev(v), z)
            out[bf16].append(z.cpu().numpy())
        ctx.close()
    bx, by = out[1]
    assert abs(np.dot(x, by) - np.dot(bx, y)) < 1e-5 * np.linalg.norm(x) * np.linalg.norm(by)
    assert np.dot(x, bx) > 0 and np.dot(y, by) > 0
    d = np.linalg.norm(bx - out[0][0]) / np.linalg.norm(out[0][0])
    assert d < 2e-2, d
