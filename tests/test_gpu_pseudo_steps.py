"""The pseudo-time steps of the FP32 correction problem are the FP64 quotients rounded to FP32."""
import numpy as np
import pytest

import pt_inputs as I

pytestmark = pytest.mark.gpu


def test_pseudo_steps_are_rounded_quotients():
    """1 / dtau_Pt and dtau_V at 224^3 random viscosities. An FP64 reciprocal within 1.1 ulp changes the FP32
    rounding of one in 2^27 values; one of a single Newton step (good to 2^-40) changed 20 of these 11 million."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_08716_gb300 import native as N
    from paper_2207_08716_gb300.solver import PTSolver
    n = 224
    p = I.c1_params(n)
    p.update(precision=N.PT_FP32, tol=0.0, max_iter=1)
    rng = np.random.default_rng(31)
    mu = np.exp(rng.uniform(-3.0, 3.0, (n, n, n)))
    s = PTSolver(p, I.gaussian_porosity(p), fields={"mu": mu, "eta": np.ones((n, n, n))}, keep_visc=True)
    s.step_begin()
    s.iterate(0, 1)
    new = s.get("mu")
    # the workspace: 23 FP64 arrays, then FP32 ones, of which 7 is 1 / dtau_Pt, 8 mu and 9 dtau_V, each on 256 bytes
    box = (n + 1) * (n + 1) * s.px
    up = lambda b: (b + 255) // 256 * 256
    w = s.workspace.cpu().numpy()

    def slot(k):
        at = 23 * up(8 * box) + k * up(4 * box)
        return w[at:at + 4 * box].view(np.float32).reshape(n + 1, n + 1, s.px)[:n, :n, :n]
    idtp, mu32, dtv = slot(7).copy(), slot(8).copy(), slot(9).copy()
    s.close()
    assert np.array_equal(mu32, new.astype(np.float32))      # the slots are where they are taken to be
    assert not np.array_equal(new, mu)
    h = 1.0 / n
    fac_v = p["cfl_v"] * (h * h) * p["rho_i"] / (1.0 + p["beta_n"])
    fac_p = p["dtpt_scale"] * (1.0 + p["beta_n"]) / n
    for got, want in ((idtp, 1.0 / (fac_p * mu)), (dtv, fac_v / new)):
        off = np.count_nonzero(got != want.astype(np.float32))
        assert off <= 1, off
