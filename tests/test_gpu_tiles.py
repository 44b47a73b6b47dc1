"""The kernels' tile shapes, chunks and index maps at the sizes where they can go wrong (one cell more
or less than a tile, single-cell tiles, columns shorter than a chunk, every wall): fixed-count steps of
the solver against a plain 64-bit restatement of the same iteration on whole arrays (perf/cases.py)."""
import os
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _cases():
    sys.path.insert(0, os.path.join(ROOT, "perf"))
    try:
        import cases
    finally:
        sys.path.pop(0)
    return cases


def _worst(case, seed=3):
    import torch
    C = _cases()
    got = C.run(C.prepare(case, seed))
    torch.cuda.synchronize()
    want = C.exact(case, seed)
    off = {k: float((got[k].double() - want[k]).norm() / want[k].norm().clamp_min(1e-300)) for k in got}
    return max(off.values()), off


# tiles of 30 x 8 columns, three-slot rings, chunks chosen by size: n = 30 m + {0, 1, 2}, n < 30,
# rows 8 m + {0, 1, 7}, depths of 1-3 levels and beyond one chunk
@pytest.mark.parametrize("nx,ny,nz", [(3, 2, 1), (29, 7, 2), (30, 8, 3), (31, 9, 13), (61, 17, 4), (62, 24, 40),
                                      (90, 25, 67), (121, 33, 130)])
def test_fp32_correction_tiles(nx, ny, nz):
    """Two rounds of 20 FP32 iterations. Bound: each iteration rounds a value some 8 times in a row
    (2^-24 each), the iteration does not amplify them, and the update adds them once a round:
    2 * 20 * 8 * 2^-24 = 1.9e-5."""
    case = dict(kind="corr", nx=nx, ny=ny, nz=nz, rounds=2, iters=20, mg=0, logk=True)
    worst, off = _worst(case)
    assert worst < 2 * 20 * 8 * 2.0 ** -24, off


# 32 x 8 column blocks in chunks of levels, and index maps over the planes' points
@pytest.mark.parametrize("form", ["df64", "fp64"])
@pytest.mark.parametrize("nx,ny,nz,shear,logk", [(3, 2, 1, False, False), (31, 7, 5, True, False),
                                                 (32, 8, 17, False, True), (33, 9, 16, True, True),
                                                 (64, 15, 33, False, False), (97, 26, 40, True, False),
                                                 (130, 50, 21, False, True), (150, 147, 149, True, True)])
def test_fixed_count_steps(form, nx, ny, nz, shear, logk):
    """Three Picard intervals of PT iterations; the FP64-class bar of the oracle comparisons, 1e-10."""
    case = dict(kind="step", form=form, nx=nx, ny=ny, nz=nz, iters=45, shear=shear, logk=logk)
    worst, off = _worst(case)
    assert worst < 1e-10, off


# one cell per thread on small grids; beyond 300 k cells four: rows of 4 m + {0, 1, 3} cells, single cells and
# rows, chunks of up to 16 levels
@pytest.mark.parametrize("nx,ny,nz", [(1, 3, 5), (33, 31, 17), (1, 701, 431), (3, 2, 60001), (32, 5, 1901),
                                      (33, 31, 297), (127, 129, 19)])
def test_reactive_rows_fp32(nx, ny, nz):
    """20 FP32 iterations of some 16 roundings (2^-24 each) in a row: 20 * 16 * 2^-24 = 1.9e-5."""
    worst, off = _worst(dict(kind="rx", form="fp32", nx=nx, ny=ny, nz=nz, iters=20))
    assert worst < 20 * 16 * 2.0 ** -24, off


# coarse rows of one, odd and even numbers of cells; a coarsest grid of one block and larger ones; one cell
# per thread, four on the finest grid, four on the next one too
@pytest.mark.parametrize("nx,ny,nz", [(4, 12, 8), (20, 8, 40), (36, 28, 72), (4, 300, 256), (20, 100, 152),
                                      (132, 132, 140)])
def test_reactive_cycles_fp32(nx, ny, nz):
    """Two V-cycles on three levels against the FP64 form, which has one cell per thread: some 40 sweeps a
    cycle (30 of them coarsest) of 8 roundings in a row, 2 * 40 * 8 * 2^-24 = 3.8e-5."""
    C = _cases()
    case = dict(kind="rxmg", nx=nx, ny=ny, nz=nz, levels=3, cycles=2)
    got, want = (C.run(C.prepare(dict(case, form=f), 3)) for f in ("fp32", "fp64"))
    off = {k: float((got[k].double() - want[k]).norm() / want[k].norm().clamp_min(1e-300)) for k in got}
    assert max(off.values()) < 2 * 40 * 8 * 2.0 ** -24, off


# index maps of cells, faces and edges: full 32 x 4 tiles of cells or of edges, neither, two cells a side
@pytest.mark.parametrize("powerlaw", [False, True])
@pytest.mark.parametrize("dims", [(3, 2, 2), (31, 7, 5), (32, 8, 3), (35, 9, 4)])
def test_transposed_stencils_at_tile_edges(dims, powerlaw):
    """J^T w against the vector-Jacobian product of the CPU residual, component by component; the bar of
    the FP64 kernels against the same product, 1e-12."""
    import numpy as np
    import torch
    import pt_inputs as I
    from oracle import adjoint as A
    from paper_2207_08716_gb300.solver import PTSolver
    nx, ny, nz = dims
    p = A.adjoint_params(I.c1_params(*dims), powerlaw)
    p.update(precision=0, tol=1e-9, max_iter=400000)
    phi = I.gaussian_porosity(p, centres=((0.4, 0.55, 0.5),), width=0.2)
    theta = I.gaussian_random_field(phi.shape, seed=5, std=0.5)
    s = PTSolver(p, phi, logk=theta)
    s.step()
    UK, FK = (A.U_KEYS_PL, A.F_KEYS_PL) if powerlaw else (A.U_KEYS, A.F_KEYS)
    u = {k: A._t(s.get(k)).requires_grad_(True) for k in UK}
    rng = np.random.default_rng(11)
    shapes = I.field_shapes(nx, ny, nz)
    w = {k: rng.standard_normal(shapes.get(k, shapes["centre"])) for k in UK}
    inner = {"Vx": (slice(None), slice(None), slice(1, -1)), "Vy": (slice(None), slice(1, -1), slice(None)),
             "Vz": (slice(1, -1),)}
    for k, axis in (("Vx", 2), ("Vy", 1), ("Vz", 0)):
        np.moveaxis(w[k], axis, 0)[[0, -1]] = 0.0
    got = s.adjoint_apply(w)
    s.close()
    z = torch.zeros_like(u["Pt"])
    old = dict(Pto=z, Pfo=z, Lo=z)
    if powerlaw:
        old["mu_o"] = torch.full_like(u["Pt"], p["mu0"])
    F = A.residual(p, u, old, A._t(theta))
    rows = dict(zip(FK, UK))
    dot = sum((F[f] * A._t(w[k][inner.get(k, ())])).sum() for f, k in rows.items())
    for k, ref in zip(UK, torch.autograd.grad(dot, [u[k] for k in UK])):
        ref = ref.numpy()[inner.get(k, ())]
        assert np.abs(got[k][inner.get(k, ())] - ref).max() <= 1e-12 * max(np.abs(ref).max(), 1e-300), k
