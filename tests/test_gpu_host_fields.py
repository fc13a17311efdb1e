"""Host fields large enough to be split, merged, summed and checked on the device: what is set is
read back (exactly in FP64, to the words of the pair otherwise), in whichever state buffer it lands,
and a refused field leaves the state, its clock and the stress alone.

Tolerances: an FP32 pair or a double word holds U13 minus its mean to 2^-48 of the largest value,
read back with one FP64 rounding: 2^-46 max|U13|."""
import numpy as np
import pytest

from paper_1911_03225_gb300 import FDM, Batch, FDMError, Params
from paper_1911_03225_gb300 import binding as B

pytestmark = pytest.mark.gpu

GRIDS = [(128, 128), (16, 1024), (256, 64), (64, 128)]   # the last one stays on the host


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def close(got, u, precision):
    if precision == B.FP64:
        np.testing.assert_array_equal(got, u)
    else:
        assert np.abs(got - u).max() <= 2.0 ** -46 * np.abs(u).max()


@pytest.mark.parametrize("n1,n2", GRIDS)
@pytest.mark.parametrize("precision", [B.FP64, B.DF64, B.MIXED])
def test_set_and_read_back_in_both_buffers(n1, n2, precision):
    rng = np.random.default_rng(n1)
    p = Params(n1=n1, n2=n2, nz=16, precision=precision, cfl=0.4, autotune=0)
    with FDM(p) as sim:
        for steps in (0, 1, 2, 3):   # the state in either buffer when the next field arrives
            u = rng.standard_normal((n2, n1)) + 3.0
            sim.set_plastic_distortion(u)
            info = sim.info()
            assert info.step == 0 and info.mean_up13 == pytest.approx(u.mean(), rel=1e-14)
            close(sim.read_fields("up13")["up13"], u, precision)
            sim.step(steps)
    with Batch([p, p, p]) as b:
        us = [rng.standard_normal((n2, n1)) - i for i in range(3)]
        for rep in range(2):
            for i, u in enumerate(us):
                b.set_plastic_distortion(i, u)
                b.set_budget(i, i + rep)
            for i, u in enumerate(us):
                close(b.read_fields(i, "up13")["up13"], u, precision)
            b.enqueue_steps(2)
            b.sync()


@pytest.mark.parametrize("n1,n2", GRIDS)
@pytest.mark.parametrize("precision", [B.FP64, B.DF64, B.MIXED])
def test_refused_fields_change_nothing(n1, n2, precision):
    rng = np.random.default_rng(n2)
    u = rng.standard_normal((n2, n1))
    p = Params(n1=n1, n2=n2, nz=16, precision=precision, velocity_mode=B.V_STRESS, loading_mode=B.LOAD_STRAIN_RAMP,
               eps_bar13_rate=1e-3, cfl=0.4, autotune=0)
    with FDM(p) as sim:
        sim.set_plastic_distortion(u)
        for steps in (1, 2):
            i0 = sim.step(steps)
            before = sim.read_fields("up13", "tau13")
            for bad in (np.nan, np.inf, -np.inf):
                v = u.copy()
                v[-1, -2] = bad
                for call in (lambda: sim.set_plastic_distortion(v), lambda: sim.set_density(v, u - u.mean())):
                    with pytest.raises(FDMError) as e:
                        call()
                    assert e.value.status == B.FDM_ERR_INVALID_ARG
            with pytest.raises(FDMError) as e:
                sim.set_density(u - u.mean() + 0.5, u - u.mean())
            assert e.value.status == B.FDM_ERR_NET_BURGERS
            after = sim.read_fields("up13", "tau13")
            np.testing.assert_array_equal(after["up13"], before["up13"])
            np.testing.assert_array_equal(after["tau13"], before["tau13"])
            assert sim.info().step == i0.step and sim.info().t == i0.t


@pytest.mark.parametrize("precision", [B.FP64, B.DF64, B.MIXED])
def test_refused_modulus_keeps_the_old_field(precision):
    n = 128
    rng = np.random.default_rng(1)
    p = Params(n1=n, n2=n, nz=16, nh=16, precision=precision, velocity_mode=B.V_STRESS, sigma_bar13=0.1, autotune=0)
    f = 0.5 + rng.random((n, n))
    with FDM(p) as sim:
        sim.set_plastic_distortion(rng.standard_normal((n, n)))
        sim.set_shear_modulus_field(f, tol=0.0, max_iter=4)
        sim.static_solve()
        want = sim.read_fields("tau13")["tau13"]
        for bad in (0.0, -1.0, np.nan, np.inf):
            g = f.copy()
            g[3, 5] = bad
            for call in (lambda: sim.set_shear_modulus_field(g, tol=0.0, max_iter=4),
                         lambda: sim.static_solve_heterogeneous(g, tol=0.0, max_iter=2)):
                with pytest.raises(FDMError) as e:
                    call()
                assert e.value.status == B.FDM_ERR_INVALID_ARG
        sim.static_solve()
        np.testing.assert_array_equal(sim.read_fields("tau13")["tau13"], want)
