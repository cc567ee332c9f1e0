"""The coarsest grid's explicit inverse: grids of one level, where a V-cycle is
z = A^-1 r, at the edges of the ranges of the elimination kernels (32, 64, 128
and 160 cells by one CTA, 32-row steps of 64 x 64 tiles beyond), against the
dense matrix formed on the host."""
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


def dense(grid, m, w):
    """The 7-point operator as a matrix; w: lower-face weights per axis."""
    n = grid.n
    idx = np.arange(grid.cells).reshape(grid.shape)
    A = np.diag(m.ravel())
    for a in range(3):
        ax = 2 - a
        lo = np.roll(idx, 1, axis=ax)
        wf = w[a].copy()
        if not grid.periodic[a]:
            sl = [slice(None)] * 3
            sl[ax] = 0
            wf[tuple(sl)] = 0.0
        for c, l, v in zip(idx.ravel(), lo.ravel(), wf.ravel()):
            A[c, c] += v
            A[l, l] += v
            A[c, l] -= v
            A[l, c] -= v
    return A


@pytest.mark.parametrize("n,periodic,stiff", [
    ((1, 1, 1), (False,) * 3, 1), ((2, 2, 2), (True,) * 3, 1), ((3, 1, 11), (True, False, True), 1),
    ((4, 4, 2), (False,) * 3, 1), ((4, 4, 4), (False, True, False), 1), ((5, 13, 1), (False,) * 3, 1),
    ((4, 8, 4), (False,) * 3, 1), ((3, 43, 1), (False,) * 3, 1), ((4, 8, 5), (True,) * 3, 1),
    ((7, 23, 1), (False,) * 3, 1), ((9, 3, 7), (False, False, True), 1), ((11, 9, 7), (False,) * 3, 1),
    ((19, 7, 3), (False, True, False), 1), ((11, 7, 7), (False,) * 3, 1),
    ((32, 32, 1), (False,) * 3, 1),
    # nearly singular: no FP32 inverse contracts the error, so the FP64
    # elimination replaces it (both its forms)
    ((4, 4, 4), (False,) * 3, 1e9), ((5, 25, 1), (False,) * 3, 1e9), ((9, 19, 1), (False,) * 3, 1e9)])
@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED])
def test_one_level_vcycle_is_the_inverse(fld, n, periodic, stiff, precision):
    c = synth.random_case(n, seed=11, periodic=periodic)
    if stiff > 1 and precision == synth.PREC_MIXED and c.grid.cells <= 160:
        pytest.skip("FP32 inverse by design")
    c.params.precision = precision
    if stiff > 1:
        c.params.dt *= stiff
        c.params.sigma = 0.0
    ctx = fld.fld_create(c.grid, c.params)
    dev = [torch.from_numpy(v.ravel().copy()).cuda() for v in (c.E, c.nHI, c.eta)]
    fld.fld_assemble(ctx, *dev)
    sysv = [torch.empty(c.grid.cells, dtype=torch.float64, device="cuda") for _ in range(4)]
    fld.fld_get_system(ctx, *sysv)
    m, wx, wy, wz = [v.cpu().numpy().reshape(c.grid.shape) for v in sysv]
    A = dense(c.grid, m, (wx, wy, wz))
    r = np.random.default_rng(3).standard_normal(c.grid.cells)
    if precision == synth.PREC_MIXED:
        r = r.astype(np.float32).astype(np.float64)
    z = torch.empty(c.grid.cells, dtype=torch.float64, device="cuda")
    fld.fld_vcycle(ctx, torch.from_numpy(r).cuda(), z)
    ctx.close()
    z = z.cpu().numpy()
    # |(A X - I)_ij| is at most a few n roundings of the products it is formed
    # from, each at most diag_i |X_ij| <= S
    N = c.grid.cells
    fp32 = precision == synth.PREC_MIXED
    X = np.linalg.inv(A)
    S = np.max(np.diag(A)[:, None] * np.abs(X))
    eps = 2.0 ** -24 if fp32 else 2.0 ** -53
    err = np.max(np.abs(A @ z - r))
    assert err <= 16 * N * eps * S * np.max(np.abs(r)), (err, S)
    if fp32 and N > 160:
        # FP64 inverse, FP32 in and out (and an FP32 operator): each entry of
        # z off by its own rounding and the operator's
        z64 = np.linalg.solve(A, r)
        bound = 2.0 ** -24 * (np.abs(z64) + np.abs(X) @ (2 * np.diag(A) * np.abs(z64) + np.abs(A) @ np.abs(z64)))
        assert np.all(np.abs(z - z64) <= 2 * bound + 1e-12 * np.max(np.abs(z64)))
