"""The FP64 static problem's block fixed-point transforms against the oracle, where they can go
wrong: the smallest and the longest rows and columns (one to four passes, every last radix),
fields whose sequences need every scale (noise, a single Fourier mode, a front, one spike,
constant rows, a zero field) and magnitudes near the ends of FP64's range.

Tolerance (relative L2): a transform's rounding is below 2^-52 of its sequence's norm on either
side, and the static solve chains four of them and one product: 1e-14 covers both sides' errors
four times over."""
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


def field(kind, n1, n2):
    x, y = np.arange(n1)[None, :], np.arange(n2)[:, None]
    if kind == "noise":
        return np.random.default_rng(n1 + n2).standard_normal((n2, n1))
    if kind == "mode":
        return np.sin(2 * np.pi * (x / n1 + 2 * y / n2)) + 0.5
    if kind == "front":
        return np.where((x > n1 // 4) & (x < n1 // 2) & (y > n2 // 3), 5.0, 0.0) + 0.0 * x * y
    if kind == "spike":
        u = np.zeros((n2, n1))
        u[n2 // 3, n1 // 3] = 1.0
        return u
    return np.repeat(np.random.default_rng(7).standard_normal((n2, 1)), n1, axis=1)   # constant rows


@pytest.mark.parametrize("n1,n2", [(16, 16), (32, 16), (16, 64), (64, 32), (128, 256), (256, 1024), (512, 128),
                                   (1024, 64), (2048, 512), (4096, 16), (16, 2048), (64, 4096)])
@pytest.mark.parametrize("kind", ["noise", "mode", "front", "spike", "rows"])
def test_static_solve_every_length(n1, n2, kind):
    u = field(kind, n1, n2)
    p = Params(n1=n1, n2=n2, nz=16, nh=4, velocity_mode=B.V_STRESS, loading_mode=B.LOAD_STRESS, sigma_bar13=0.25,
               autotune=0)
    K = oracle.kernel_table(n1, n2, 16, 4, p.E / (2 * (1 + p.nu)), p.nu)
    with FDM(p) as sim:
        for scale in (1.0, 2.0 ** -930, 2.0 ** 960):
            ref = oracle.static_tau(u * scale, K, 0.25 * scale)
            sim.set_loading(B.LOAD_STRESS, sigma_bar13=0.25 * scale)
            sim.set_plastic_distortion(u * scale)
            sim.static_solve()
            got = sim.read_fields("tau13")["tau13"]
            assert np.linalg.norm(got / scale - ref / scale) <= 1e-14 * np.linalg.norm(ref / scale), scale


def test_static_solve_of_zero_is_the_macroscopic_stress():
    p = Params(n1=64, n2=32, velocity_mode=B.V_STRESS, loading_mode=B.LOAD_STRESS, sigma_bar13=0.125)
    with FDM(p) as sim:
        sim.set_plastic_distortion(np.zeros((32, 64)))
        sim.static_solve()
        assert np.all(sim.read_fields("tau13")["tau13"] == 0.125)
