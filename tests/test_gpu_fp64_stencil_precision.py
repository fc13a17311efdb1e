"""FP64 stencil nodes keep FP64's precision over the limiter parameter's whole range, where the
two axes differ in size, and over long runs.

Tolerance of one step (relative L2 of the increment): an increment is a sum of about forty rounded
products and quotients of the field's differences, on either side; on fields with no exact ties
each rounds within 2^-53 of the largest, and the fields' differences are of their own size, so 1e-14 (ninety
times 2^-53) covers both."""
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
    prev = oracle.threads()
    oracle.set_threads(0)
    yield
    oracle.set_threads(prev)


def one_step_error(u, theta, v0):
    n2, n1 = u.shape
    p = Params(n1=n1, n2=n2, nz=16, nh=4, v0=v0, theta=theta, cfl=0.45, autotune=0)
    op = oracle.Params(**{k: getattr(p, k) for k in oracle.Params.__dataclass_fields__})
    ref, rc = oracle.run(op, u, 1, K=np.zeros((n2, n1)))   # the prescribed celerity needs no stress
    assert rc == 0
    with FDM(p) as sim:
        sim.set_plastic_distortion(u)
        sim.step(1)
        got = sim.read_fields("up13")["up13"]
    return np.linalg.norm(got - ref.up13) / np.linalg.norm(ref.up13 - u)


@pytest.mark.parametrize("theta", [float(np.nextafter(2.0, 0.0)), 2.0 - 1e-10, 2.0 - 1e-9, 1.25,
                                   float(np.nextafter(1.0, 2.0))])
@pytest.mark.parametrize("n1,n2", [(64, 32), (1024, 256)])
def test_limiter_parameter_range(theta, n1, n2):
    rng = np.random.default_rng(11)
    x, y = np.arange(n1)[None, :] / 16, np.arange(n2)[:, None] / 16
    noise = rng.standard_normal((n2, n1))
    smooth = np.sin(2 * np.pi * x + 0.3) * np.cos(2 * np.pi * y + 0.1) + 0.2 * np.sin(4 * np.pi * (x + y) + 1.0)
    for u in (noise, smooth + 1e-3 * noise):
        assert one_step_error(u, theta, 1.0) <= 1e-14


@pytest.mark.parametrize("scale", [1e-3, 1e-6, 1e-9, 1e-12])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("theta,v0", [(1.0, 1.0), (1.7, -1.0), (2.0, 1.0)])
@pytest.mark.parametrize("n1,n2", [(64, 64), (1024, 256)])
def test_axes_of_different_size(scale, axis, theta, v0, n1, n2):
    """Noise of unit size with every fourth line along one axis scaled down: beside such a line the
    differences along the axis are of unit size, on it they are `scale` times that."""
    u = np.random.default_rng(12).standard_normal((n2, n1))
    if axis == 0:
        u[:, 1::4] *= scale
    else:
        u[1::4, :] *= scale
    assert one_step_error(u, theta, v0) <= 1e-14
