"""The lattice friction's cosine in fixed point against numpy's, through the velocity readout and
the time step (both from v0 = tau_y cos(U13 / beta) - tau13 with unit mobility): zero, the cosine's
zeros and extrema, arguments from 1e-30 to the fixed-point range's end at 2^10 turns and beyond
it, beta that are and are not powers of two.

Tolerance: numpy's argument is off by |x| 2^-53 and its cosine by 2^-53, this one's by less; the
sum and the readout's norm add four roundings of v0 or its terms: 2^-52 (tau_y (1 + |x|) + 4 (tau_y
+ |tau13|))."""
import numpy as np
import pytest

from paper_1911_03225_gb300 import FDM, Params
from paper_1911_03225_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("beta", [0.5, 0.3, 2.0 ** -20, 1e-3, 1e3, 1e-90])
@pytest.mark.parametrize("turns", [1e-30, 0.25, 3.0, 60.0, 1023.0, 1025.0, 1e5])
def test_friction_against_numpy(beta, turns):
    n, tau_y = 32, 0.25
    u = np.random.default_rng(3).uniform(-1.0, 1.0, (n, n)) * turns * 2 * np.pi * abs(beta)
    u[0, :8] = np.arange(-4, 4) * np.pi / 2 * beta
    u[1, 0] = u[2, 0] = 0.0
    # a prescribed stress far above the field's own keeps |v0| away from cancellation of its terms
    p = Params(n1=n, n2=n, velocity_mode=B.V_STRESS, mobility=1.0, tau_y=tau_y, beta=beta,
               loading_mode=B.LOAD_STRESS, sigma_bar13=1.0, cfl=0.4, autotune=0)
    with FDM(p) as sim:
        sim.set_plastic_distortion(u)
        sim.static_solve()
        f = sim.read_fields("up13", "tau13", "v1", "v2")
        x = f["up13"] / beta
        v0 = tau_y * np.cos(x) - f["tau13"]
        tol = 2.0 ** -52 * (tau_y * (1 + np.abs(x)) + 4 * (tau_y + np.abs(f["tau13"])))
        v = np.hypot(f["v1"], f["v2"])
        moving = v > 0
        assert moving.mean() > 0.9
        assert (np.abs(v - np.abs(v0)) <= tol)[moving].all()
        vmax = np.abs(v0).max()
        info = sim.step(1)
        assert abs(0.4 * p.dx / info.dt - vmax) <= tol.max() + 2.0 ** -50 * vmax
