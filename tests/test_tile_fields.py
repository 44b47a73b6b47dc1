"""Every field of the tile-edge cases by itself: each must be finite and within the bound. (A largest error
over the fields taken with Python's `max` passes a NaN in any field but the first.) The sizes and bounds are
those of test_gpu_tiles.py."""
import math

import pytest

import test_gpu_tiles as T


def field_errors(got, want):
    return {k: float((got[k].double() - want[k].double()).norm() / want[k].double().norm().clamp_min(1e-300))
            for k in got}


def beyond(off, bound):
    """The fields whose error is not below the bound, a NaN among them."""
    return {k: v for k, v in off.items() if not v < bound}


def _sizes(test):
    return {m.args[0]: m.args[1] for m in test.pytestmark if m.name == "parametrize"}


def _case_errors(case):
    import torch
    C = T._cases()
    got = C.run(C.prepare(case, 3))
    torch.cuda.synchronize()
    return field_errors(got, C.exact(case, 3))


def test_nan_in_the_last_field_is_beyond_every_bound():
    import torch
    want = {k: torch.ones(5, dtype=torch.float64) for k in ("a", "b", "c")}
    got = {k: v.clone() for k, v in want.items()}
    assert beyond(field_errors(got, want), 1e-12) == {}
    got["c"][3] = math.nan
    off = field_errors(got, want)
    assert max(off.values()) == 0.0          # what a plain largest error says
    assert list(beyond(off, 1e300)) == ["c"]
    got["c"][3] = math.inf
    assert list(beyond(field_errors(got, want), 1e300)) == ["c"]


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,nz", _sizes(T.test_fp32_correction_tiles)["nx,ny,nz"])
def test_fp32_correction_fields(nx, ny, nz):
    off = _case_errors(dict(kind="corr", nx=nx, ny=ny, nz=nz, rounds=2, iters=20, mg=0, logk=True))
    assert not beyond(off, 2 * 20 * 8 * 2.0 ** -24), off


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["df64", "fp64"])
@pytest.mark.parametrize("nx,ny,nz,shear,logk", _sizes(T.test_fixed_count_steps)["nx,ny,nz,shear,logk"])
def test_fixed_count_fields(form, nx, ny, nz, shear, logk):
    off = _case_errors(dict(kind="step", form=form, nx=nx, ny=ny, nz=nz, iters=45, shear=shear, logk=logk))
    assert not beyond(off, 1e-10), off


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,nz", _sizes(T.test_reactive_rows_fp32)["nx,ny,nz"])
def test_reactive_row_fields(nx, ny, nz):
    off = _case_errors(dict(kind="rx", form="fp32", nx=nx, ny=ny, nz=nz, iters=20))
    assert not beyond(off, 20 * 16 * 2.0 ** -24), off


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,nz", _sizes(T.test_reactive_cycles_fp32)["nx,ny,nz"])
def test_reactive_cycle_fields(nx, ny, nz):
    C = T._cases()
    case = dict(kind="rxmg", nx=nx, ny=ny, nz=nz, levels=3, cycles=2)
    got, want = (C.run(C.prepare(dict(case, form=f), 3)) for f in ("fp32", "fp64"))
    off = field_errors(got, want)
    assert not beyond(off, 2 * 40 * 8 * 2.0 ** -24), off
