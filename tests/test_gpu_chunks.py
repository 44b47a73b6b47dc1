"""A column's values do not depend on how it is cut into chunks of levels. Fields that vary in z alone stay
so (free-slip walls, uniform coefficients in x and y), whatever the grid's extent in x and y; with it varies
the number of columns, and with that the chunk that the marching kernels choose."""
import numpy as np
import pytest

import pt_inputs as I

pytestmark = pytest.mark.gpu

NZ = 64
FIELDS = ("Vz", "Pt", "Pf", "phi", "mu", "eta", "txx", "tyy", "tzz")


def _profile(form, nx, ny, iters):
    """Fields over z of a step's `iters` iterations on nx x ny columns of NZ cells of the same size."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_08716_gb300 import native as N
    from paper_2207_08716_gb300.solver import PTSolver
    p = I.c1_params(NZ)
    p.update(nx=nx, ny=ny, lx=nx / NZ, ly=ny / NZ, precision=getattr(N, form), tol=0.0, max_iter=iters)
    z = (np.arange(NZ) + 0.5) / NZ
    phi = p["phi0"] * (1.0 + 2.0 * np.exp(-((z - 0.45) / 0.1) ** 2) + 0.05 * np.sin(9.0 * z))
    rng = np.random.default_rng(8)
    pf = 1e-3 * rng.standard_normal(NZ)
    col = lambda v: np.ascontiguousarray(np.broadcast_to(v[:, None, None], (NZ, ny, nx)))
    s = PTSolver(p, col(phi), fields={"Pf": col(pf), "Pt": col(0.7 * pf)})
    s.step()
    out = {k: s.get(k) for k in FIELDS}
    s.close()
    for k, v in out.items():
        assert np.array_equal(v, np.broadcast_to(v[:, :1, :1], v.shape)), (form, k)
    return {k: v[:, 0, 0] for k, v in out.items()}


# on 152 SMs the double-float cells take chunks of 1 level at 32 x 8 columns and of 4, 16, 16 and 13 here
@pytest.mark.parametrize("form", ["PT_DF64", "PT_FP64"])
@pytest.mark.parametrize("nx,ny", [(64, 64), (128, 128), (256, 64), (256, 256)])
def test_columns_are_the_same_for_every_chunk(form, nx, ny):
    want, got = _profile(form, 32, 8, 30), _profile(form, nx, ny, 30)
    for k in FIELDS:
        assert np.array_equal(got[k], want[k]), (k, np.abs(got[k] - want[k]).max())
