"""The column pass's merged scale (forward exponent plus inverse exponent) at the ends of FP64's
range, where the field and the elastic modulus are both small or both large.

Tolerance (relative L2): every scale is a power of two, so the solve is the one at unit scale but
for results below the normal range, a 2^-60 part here; 1e-14 as for the transforms at unit scale."""
import math

import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("kind", ["noise", "mode"])
@pytest.mark.parametrize("n1,n2", [(16, 16), (64, 32), (256, 128), (32, 2048)])
@pytest.mark.parametrize("field_exp,modulus_exp", [(-880, -93), (-870, -60), (-600, -300), (840, 120), (-300, 700)])
def test_static_solve_small_and_large_modulus(kind, n1, n2, field_exp, modulus_exp):
    if kind == "noise":
        u = np.random.default_rng(n1 + n2).standard_normal((n2, n1))
    else:   # its columns pass through zero: results of a few units in the last place
        u = np.sin(2 * np.pi * (np.arange(n1)[None, :] / n1 + np.arange(n2)[:, None] / n2))
    u -= u.mean()
    base = Params(n1=n1, n2=n2, nz=16, nh=4)
    K = oracle.kernel_table(n1, n2, 16, 4, base.E / (2 * (1 + base.nu)), base.nu)
    ref = oracle.static_tau(u, K, 0.0)
    p = Params(n1=n1, n2=n2, nz=16, nh=4, E=2.0 ** modulus_exp, velocity_mode=B.V_STRESS,
               loading_mode=B.LOAD_STRESS, sigma_bar13=0.0, autotune=0)
    with FDM(p) as sim:
        sim.set_plastic_distortion(np.ldexp(u, field_exp))
        sim.static_solve()
        got = sim.read_fields("tau13")["tau13"]
    got = np.ldexp(got, -(field_exp + modulus_exp))
    assert np.linalg.norm(got - ref) <= 1e-14 * np.linalg.norm(ref)


@pytest.mark.parametrize("n1", [64, 512, 2048, 4096])
@pytest.mark.parametrize("background", ["random", "constant"])
def test_mean_of_rows_of_unequal_size(n1, background):
    """The mean of U13 sets the stress under a strain: a field of equal rows, one value of 1 and positive
    ones of 2^-20 and less, in a full-depth layer (no other stress).  Bar: eight roundings of 2^-53 (a thread's
    and the row's sum, the mean, the loading law's products and difference, the way back to doubles)."""
    r = np.random.default_rng(n1).uniform(0.0, 2.0 ** -20, n1)
    if background == "constant":
        r[:] = r[0]
    r[n1 // 3] = 1.0
    p = Params(n1=n1, n2=16, nz=16, nh=16, velocity_mode=B.V_STRESS, loading_mode=B.LOAD_STRAIN_RAMP, autotune=0)
    with FDM(p) as sim:
        sim.set_plastic_distortion(np.repeat(r[None, :], 16, axis=0))
        sim.static_solve()
        tau = sim.read_fields("tau13")["tau13"]
    want = -p.E / (2 * (1 + p.nu)) * (math.fsum(r) / n1)
    assert np.abs(tau / want - 1.0).max() <= 8 * 2.0 ** -53
