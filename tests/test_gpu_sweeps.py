"""The sweeps that take a level by parts of a row, cell by cell against the host:
the compressed FP32 sweeps (bfloat16 coefficients rounded here) and the FP64
pair sweeps, at the block shapes that launches of 2^18 threads and more choose
(32, 16 and 8 lanes along x) and at small ragged ones."""
import dataclasses

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


def make(n, periodic, outflow=False):
    case = synth.random_case(n, seed=sum(n), periodic=tuple(map(bool, periodic)), E_decades=(-20, -14))
    if outflow:
        case.grid = case.grid.outflow_upper()
    return case


def neighbours(w, u, periodic):
    """sum_f w_f u_nbr; w: lower-face weights per axis."""
    out = np.zeros_like(u)
    for a in range(3):
        ax = 2 - a
        wl = w[a].copy()
        if not periodic[a]:
            wl[tuple(0 if q == ax else slice(None) for q in range(3))] = 0.0
        out += wl * np.roll(u, 1, axis=ax)
        out += np.roll(wl, -1, axis=ax) * np.roll(u, -1, axis=ax)
    return out


def diagonal32(m, w, periodic):
    """FP32 inverse diagonal: m + (x lo + x hi + y lo + y hi + z lo + z hi)."""
    s = np.zeros_like(m)
    for a in range(3):
        ax = 2 - a
        wl = w[a].copy()
        if not periodic[a]:
            wl[tuple(0 if q == ax else slice(None) for q in range(3))] = 0.0
        s = s + wl
        s = s + np.roll(wl, -1, axis=ax)
    return np.float32(1.0) / (m + s)


def bf16(a):
    return torch.from_numpy(np.ascontiguousarray(a)).bfloat16().double().numpy()


@pytest.mark.parametrize("n,periodic,outflow", [
    ((16, 12, 20), (0, 0, 0), False), ((24, 20, 28), (1, 0, 0), False), ((40, 6, 10), (0, 1, 0), False),
    ((48, 20, 12), (1, 1, 1), False), ((48, 20, 12), (0, 0, 0), True), ((272, 8, 12), (0, 0, 1), False), ((64, 64, 64), (0, 0, 0), True),
    ((256, 96, 96), (0, 1, 0), False), ((384, 48, 128), (1, 0, 0), False), ((192, 96, 128), (0, 0, 1), False),
    ((320, 96, 80), (0, 0, 0), True)])
def test_compressed_cycle_cell_by_cell(fld, oracle, n, periodic, outflow):
    case = make(n, periodic, outflow)
    grid, per = case.grid, case.grid.periodic
    case.params.precision = synth.PREC_MIXED
    # the level below runs in FP32 (the tail), so only this one is compressed
    ctx = fld.fld_create(grid, case.params, tail_cells=grid.cells // 8, coarse_cap=4096)
    fld.fld_assemble(ctx, dev(case.E), dev(case.nHI), dev(case.eta))
    sysv = [torch.empty(grid.cells, dtype=torch.float64, device="cuda") for _ in range(4)]
    fld.fld_get_system(ctx, *sysv)
    m, wx, wy, wz = [v.cpu().numpy().reshape(grid.shape).astype(np.float32) for v in sysv]
    r = np.random.default_rng(12).standard_normal(grid.shape).astype(np.float32).astype(np.float64)
    z = torch.empty(grid.cells, dtype=torch.float64, device="cuda")
    fld.fld_vcycle(ctx, dev(r), z)
    ctx.close()
    got = z.cpu().numpy().reshape(grid.shape)

    w = [bf16(v) for v in (wx, wy, wz)]
    inv = bf16(diagonal32(m, (wx, wy, wz), per))
    k, j, i = np.indices(grid.shape)
    red = (i + j + k) % 2 == 0
    u = np.where(red, r * inv, 0.0)
    zb = np.where(red, 0.0, inv * (r + neighbours(w, u, per)))
    res = np.where(red, neighbours(w, zb, per), 0.0)
    op = {"m": m, "wx": wx, "wy": wy, "wz": wz}
    dirich = None
    if outflow:
        op["bnd"] = oracle.assemble(grid, case.params, case.E, case.nHI, case.eta)["bnd"]
        dirich = grid.dirichlet
    coarse = dataclasses.replace(grid, n=tuple(v // 2 for v in n), h=tuple(2 * v for v in grid.h))
    ec = oracle.vcycle(coarse, oracle.coarsen(n, per, op, dirich), oracle.restrict(n, per, res),
                       {"coarse_cap": 4096})
    u = np.where(red, oracle.prolong_add(n, per, ec, u), 0.0)
    zb = np.where(red, 0.0, inv * (r + neighbours(w, u, per)))
    ref = np.where(red, inv * (r + neighbours(w, zb, per)), zb)
    # the FP32 rounding of the cycle, as for the FP32-coefficient one
    assert np.abs(got - ref).max() < 1e-5 * np.abs(ref).max()
    assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("n,periodic,outflow", [((80, 96, 144), (1, 0, 1), False), ((48, 128, 176), (0, 1, 0), False),
                                                ((96, 96, 64), (0, 0, 0), True), ((96, 96, 64), (0, 0, 1), False)])
def test_fp64_cycle_on_rows_that_32_lanes_do_not_divide(fld, oracle, n, periodic, outflow):
    case = make(n, periodic, outflow)
    ctx = fld.fld_create(case.grid, case.params)
    fld.fld_assemble(ctx, dev(case.E), dev(case.nHI), dev(case.eta))
    x = np.random.default_rng(13).standard_normal(case.grid.shape)
    z = torch.empty(case.grid.cells, dtype=torch.float64, device="cuda")
    fld.fld_vcycle(ctx, dev(x), z)
    ctx.close()
    op = oracle.assemble(case.grid, case.params, case.E, case.nHI, case.eta)
    ref = oracle.vcycle(case.grid, op, x)
    got = z.cpu().numpy().reshape(case.grid.shape)
    assert np.abs(got - ref).max() < 1e-12 * np.abs(ref).max()


def test_fp64_step_on_such_rows_takes_the_oracles_iterations(fld, oracle):
    # a wrong <r, z> or <p, q> of the sweeps costs iterations
    case = make((96, 96, 64), (0, 0, 1))
    ctx = fld.fld_create(case.grid, case.params, rtol=1e-12)
    E = dev(case.E)
    info = fld.fld_step(ctx, E, dev(case.nHI), dev(case.eta))
    ctx.close()
    Eref, iref = oracle.step(case.grid, case.params, {"rtol": 1e-12, "max_iter": 200}, case.E, case.nHI, case.eta)
    got = E.cpu().numpy().reshape(case.grid.shape)
    assert np.abs(got - Eref).max() < 1e-10 * np.abs(Eref).max()
    assert info["iters"] == iref["iters"]
