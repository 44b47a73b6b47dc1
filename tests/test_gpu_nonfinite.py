"""Non-finite values stay non-finite: a viscosity that is NaN or infinite makes every stress that its cell
enters non-finite, and no other; a cell whose 1 / (1 - phi) is infinite does not pass for an ordinary one."""
import numpy as np
import pytest

import pt_inputs as I

pytestmark = pytest.mark.gpu

NX, NY, NZ = 9, 7, 6
STRESSES = ("txx", "tyy", "tzz", "txy", "txz", "tyz")


def _mods():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_08716_gb300 import native as N
    from paper_2207_08716_gb300.solver import PTSolver
    return N, PTSolver


def _stresses(form, shear, bad):
    """End-of-step stresses of a random state whose viscosity is replaced at the cells of `bad`."""
    N, PTSolver = _mods()
    p = I.c1_params(NX, NY, NZ)
    p.update(precision=getattr(N, form), tau_bg=0.03 if shear else 0.0, beta_n=0.1)
    st = I.random_state(p, seed=4)
    rng = np.random.default_rng(6)
    old = {k: 0.1 * rng.standard_normal(I.field_shapes(NX, NY, NZ).get(k, (NZ, NY, NX))) for k in STRESSES}
    s = PTSolver(p, I.gaussian_porosity(p), fields={**{k: st[k] for k in ("Vx", "Vy", "Vz", "Pt", "Pf")}, **old})
    s.step_begin()
    mu = s.get("mu")
    for cell, value in bad.items():
        mu[cell] = value
    s.set("mu", mu)
    s.step_end()
    out = {k: s.get(k) for k in STRESSES}
    s.close()
    return out


def _touched(cells, shear):
    """Where each stress reads one of the cells: centres, and the inner edges between four of them (with a
    background shear the xy-edges on the walls too)."""
    c = np.zeros((NZ, NY, NX), bool)
    for cell in cells:
        c[cell] = True
    out = {k: c for k in STRESSES[:3]}
    for k, (a, b) in (("txy", (1, 2)), ("txz", (0, 2)), ("tyz", (0, 1))):
        pad = np.pad(c, [(1, 1) if ax in (a, b) else (0, 0) for ax in range(3)])
        e = np.zeros([n + (ax in (a, b)) for ax, n in enumerate(c.shape)], bool)
        for da in (0, 1):
            for db in (0, 1):
                sl = [slice(None)] * 3
                sl[a] = slice(da, da + e.shape[a])
                sl[b] = slice(db, db + e.shape[b])
                e |= pad[tuple(sl)]
        if not (shear and k == "txy"):
            for ax in (a, b):
                np.moveaxis(e, ax, 0)[[0, -1]] = False   # edges on the walls carry no stress
        out[k] = e
    return out


@pytest.mark.parametrize("form", ["PT_FP64", "PT_FP32"])
@pytest.mark.parametrize("shear", [False, True])
def test_non_finite_viscosity_reaches_every_stress_it_enters(form, shear):
    bad = {(2, 3, 4): np.nan, (4, 5, 7): np.inf, (0, 0, 0): np.nan}
    got, clean = _stresses(form, shear, bad), _stresses(form, shear, {})
    touched = _touched(bad, shear)
    for k in STRESSES:
        assert np.isfinite(clean[k]).all(), k
        assert np.array_equal(~np.isfinite(got[k]), touched[k]), k
        assert np.array_equal(got[k][~touched[k]], clean[k][~touched[k]]), k


def test_zero_viscosity_leaves_the_old_stress_times_nothing():
    """mu = 0 at every cell of an edge: xi = 0 and 2 mu edot = 0, so tau = 0 (to the rounding of 1 / (1 + xi) times
    an old stress of some tenths)."""
    bad = {(2, 2, 2): 0.0, (2, 2, 3): 0.0, (2, 3, 2): 0.0, (2, 3, 3): 0.0}
    for form in ("PT_FP64", "PT_FP32"):
        got = _stresses(form, False, bad)
        assert all(np.isfinite(v).all() for v in got.values()), form
        assert abs(got["txy"][2, 3, 3]) <= 2.0 ** -52, (form, got["txy"][2, 3, 3])


def test_infinite_reciprocal_of_the_solid_fraction_is_not_finite_after_an_iteration():
    """phi = 1 in one cell, at rest and without compaction: V . grad(1 - phi) / (1 - phi) is 0 / 0 there."""
    N, PTSolver = _mods()
    p = I.c1_params(NX, NY, NZ)
    p.update(precision=N.PT_FP64, compaction_on=0)
    phi = I.gaussian_porosity(p)
    phi[3, 3, 3] = 1.0
    s = PTSolver(p, phi, fields={k: np.ones((NZ, NY, NX)) for k in ("mu", "eta")}, keep_visc=True)
    s.step_begin()
    s.iterate(0, 1, report=False)
    got = s.get("phi")
    s.close()
    assert not np.isfinite(got[3, 3, 3]), got[3, 3, 3]


def test_half_on_the_integers():
    """Routine 14: x / 2 bit for bit from 2^-1021 on, infinities and NaN included."""
    torch = pytest.importorskip("torch")
    N, _ = _mods()
    rng = np.random.default_rng(2)
    x = rng.integers(0, 2 ** 64, 1 << 16, dtype=np.uint64).view(np.float64)
    x = np.concatenate([x, [np.inf, -np.inf, np.nan, 1.0, -1.0, 2.0 ** -1021, -2.0 ** -1021,
                            np.finfo(float).max, -np.finfo(float).max]])
    x = x[(np.abs(x) >= 2.0 ** -1021) | np.isnan(x)]
    a = torch.from_numpy(x).cuda()
    out = torch.empty_like(a)
    torch.cuda.synchronize()
    assert N.load().pt_math_check(14, a.data_ptr(), None, out.data_ptr(), a.numel(), None) == N.PT_OK
    with np.errstate(invalid="ignore"):
        got, want = out.cpu().numpy(), x * 0.5
    n = np.isnan(x)
    assert np.isnan(got[n]).all()
    assert np.array_equal(got[~n].view(np.uint64), want[~n].view(np.uint64))
