"""fld_autotune tunes what the V-cycle launches."""
import numpy as np
import pytest

from paper_1306_0645_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RESTRICT = 3        # kernel index of a level's records


@pytest.fixture(scope="module")
def fld():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1306_0645_gb300 import fld as f
    f.lib()
    return f


@pytest.mark.parametrize("n,tail_cells", [(64, 32768), (96, 32768), (32, 0)])
def test_levels_without_a_tuned_restriction_keep_the_default_record(fld, n, tail_cells):
    # coarse grids of at most 131072 cells below a level of eight-cell sweeps
    # are restricted one coarse cell per thread, with a shape of its own: no
    # record applies, and a step is the same before and after tuning
    case = synth.config4(n, sources=64)
    case.params.precision = synth.PREC_MIXED
    E0, nHI, eta = (torch.from_numpy(np.ascontiguousarray(v).ravel()).cuda() for v in (case.E, case.nHI, case.eta))
    ctx = fld.fld_create(case.grid, case.params, tail_cells=tail_cells)
    out = []
    for tune in (False, True):
        if tune:
            fld.fld_autotune(ctx, 1)
        E = E0.clone()
        out.append((fld.fld_step(ctx, E, nHI, eta)["rel_res"], E))
    table = fld.fld_get_tuning(ctx)
    levels = fld.fld_levels(case.grid)
    ctx.close()
    kinds = len(table) // 3 // len(levels)
    for l, (nx, ny, nz) in enumerate(levels[:-1]):
        if nx % 8 or nx < 16 or nx * ny * nz <= tail_cells:
            continue
        assert nx * ny * nz // 8 <= 131072
        q = 3 * (l * kinds + RESTRICT)
        assert table[q: q + 3] == [256, 152 * 8, 1], (l, table[q: q + 3])
    assert all(r <= 1e-8 for r, _ in out)
    assert torch.linalg.norm(out[0][1] - out[1][1]) < 1e-6 * torch.linalg.norm(out[0][1])
