"""The mixed path's FP32 transforms at their smallest and longest rows and columns and over every
launch shape (rows and columns of a block beyond, equal to and below the sequences that it holds
at a time): each shape gives the same bits, and those are the oracle's field to FP32 rounding.

Tolerance (relative L2): the static solve chains four transforms of at most 12 radix-2 levels.  A
level's rounding is at most three units of 2^-24 (a product's two and a sum's one, the twiddle's
included), so 4 * 12 * 3 * 2^-24 = 8.6e-6; the field's and the symbol's rounding add two units:
9e-6."""
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


@pytest.mark.parametrize("n1,n2", [(16, 16), (32, 16), (16, 64), (64, 32), (128, 256), (256, 1024), (512, 128),
                                   (1024, 64), (2048, 512), (4096, 16), (16, 2048), (64, 4096)])
def test_static_solve_every_length_and_shape(n1, n2):
    u = np.random.default_rng(n1 + n2).standard_normal((n2, n1)).astype(np.float32)
    p = Params(n1=n1, n2=n2, nz=16, nh=4, velocity_mode=B.V_STRESS, loading_mode=B.LOAD_STRESS, sigma_bar13=0.25,
               precision=B.MIXED, autotune=0)
    K = oracle.kernel_table(n1, n2, 16, 4, p.E / (2 * (1 + p.nu)), p.nu)
    ref = oracle.static_tau(u.astype(np.float64), K, 0.25)
    first = None
    with FDM(p) as sim:
        cfg = dict(sim.launch_config())
        shapes = {(c["rows_per_block"], c["cols_per_block"]) for c in B.launch_candidates(p)}
        for rows, cols in sorted(shapes):
            sim.set_launch_config({**cfg, "rows_per_block": rows, "cols_per_block": cols})
            sim.set_plastic_distortion(u)
            sim.static_solve()
            got = sim.read_fields("tau13")["tau13"]
            first = got if first is None else first
            np.testing.assert_array_equal(got, first, err_msg=f"{rows} rows, {cols} columns")
    assert np.linalg.norm(first - ref) <= 9e-6 * np.linalg.norm(ref)
