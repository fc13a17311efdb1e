"""FP64 stencil nodes keep FP64's precision over the limiter parameter's whole range, where the
two axes differ in size, and over long runs.

Tolerance of one step (relative L2 of the increment): an increment is a sum of about forty rounded
products and quotients of the field's differences, on either side; on fields with no exact ties
each rounds within 2^-53 of the largest, and the fields' differences are of their own size, so 1e-14 (ninety
times 2^-53) covers both."""
from math import erf, pi, sqrt

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


def one_step(u, theta, v0, level=B.T_MIDPOINT, cfl=0.45):
    n2, n1 = u.shape
    p = Params(n1=n1, n2=n2, nz=16, nh=4, v0=v0, theta=theta, time_level=level, cfl=cfl, autotune=0)
    op = oracle.Params(**{k: getattr(p, k) for k in oracle.Params.__dataclass_fields__})
    ref, rc = oracle.run(op, u, 1, K=np.zeros((n2, n1)))   # the prescribed celerity needs no stress
    assert rc == 0
    with FDM(p) as sim:
        sim.set_plastic_distortion(u)
        sim.step(1)
        return sim.read_fields("up13")["up13"], ref.up13


def one_step_error(u, theta, v0):
    got, ref = one_step(u, theta, v0)
    return np.linalg.norm(got - ref) / np.linalg.norm(ref - u)


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


@pytest.mark.parametrize("theta,level,v0", [(1.0, B.T_MIDPOINT, -1.0), (1.7, B.T_MIDPOINT, -1.0),
                                            (1.0, B.T_LITERAL, 1.0), (1.7, B.T_LITERAL, -1.0)])
@pytest.mark.parametrize("n1,n2", [(64, 32), (1024, 256)])
def test_nodes_beside_a_steep_front(theta, level, v0, n1, n2):
    """Ridges of unit slope over a floor of noise of 1e-9: nodes at their feet have outer neighbours and
    diagonals 1e9 times their own differences.  On the nodes that move by less than 1e-6 the increments
    are the floor's own.  Bar 1e-13: with these directions and limiters no term of a foot's increment
    cancels, and FP64 arithmetic stays within 1.5e-16 of 113 bits."""
    x, y = np.arange(n1)[None, :], np.arange(n2)[:, None]
    ridge = np.maximum(0.0, 3.3 - np.abs((x + 0.5 * y) % 16 - 8.2))
    u = ridge + 1e-9 * np.random.default_rng(13).standard_normal((n2, n1))
    got, ref = one_step(u, theta, v0, level)
    floor = np.abs(ref - u) < 1e-6
    assert floor.mean() > 0.2
    assert np.linalg.norm((got - ref)[floor]) <= 1e-13 * np.linalg.norm((ref - u)[floor])


@pytest.mark.parametrize("e", [2.0 ** -43, 2.0 ** -40, 2.0 ** -30])
@pytest.mark.parametrize("diagonal", [2.0 ** 20, 2.0 ** 28, 2.0 ** 33])
@pytest.mark.parametrize("v0", [1.0, -1.0])
def test_near_tie_beside_a_large_diagonal(e, diagonal, v0):
    """A node at the bottom of a kink, its one-sided derivatives the differences' own differences of a few e,
    with diagonals that dwarf them: the gradient's direction comes from the former, its size from the
    latter.  Every difference is exact in doubles, the increment is three products and a root of
    them: 1e-14 as above."""
    u = np.zeros((16, 16))
    y = x = 8
    u[y, x + 1], u[y, x - 1], u[y + 1, x], u[y - 1, x] = 1 + 3 * e, 1 + e, 1 + 5 * e, 1 + 2 * e
    u[y, x + 2] = u[y, x - 2] = u[y + 2, x] = u[y - 2, x] = 9.0
    u[y + 1, x + 1], u[y - 1, x + 1], u[y + 1, x - 1], u[y - 1, x - 1] = diagonal * 0.5 ** np.arange(4)
    got, ref = one_step(u, 1.0, v0, cfl=1.0)
    assert abs(ref[y, x]) > 0.01 * diagonal
    assert abs(got[y, x] - ref[y, x]) <= 1e-14 * abs(ref[y, x])


@pytest.mark.parametrize("power", [-990, -940, -700, -520, 520, 700, 1000])
@pytest.mark.parametrize("theta,level", [(1.0, B.T_MIDPOINT), (1.7, B.T_LITERAL)])
@pytest.mark.parametrize("n1,n2", [(64, 32), (1024, 256)])
def test_update_is_homogeneous_to_the_ends_of_the_range(power, theta, level, n1, n2):
    """Steps 1 to 4 are homogeneous in U13: a step of 2^p U is 2^p times the oracle's step of U, to the
    rounding of either (1e-14 as above; near the ends a node may take the other form)."""
    u = np.random.default_rng(14).standard_normal((n2, n1))
    u[: n2 // 2] += 4.0 * np.sin(2 * np.pi * np.arange(n1) / 16)
    _, want = one_step(u, theta, 1.0, level)
    p = Params(n1=n1, n2=n2, nz=16, nh=4, v0=1.0, theta=theta, time_level=level, cfl=0.45, autotune=0)
    with FDM(p) as sim:
        sim.set_plastic_distortion(np.ldexp(u, power))
        sim.step(1)
        got = np.ldexp(sim.read_fields("up13")["up13"], -power)
    assert np.linalg.norm(got - want) <= 1e-14 * np.linalg.norm(want - u)


def annihilation(u, steps, r):
    """The same scheme on a row that does not vary along x2 (theta = 1, v0 = 1), in the precision of u: the
    x2 weights are halves of equal values, so each side of the x1 axis has one value."""
    h = u.dtype.type(0.5)
    r = u.dtype.type(r)

    def minmod3(a, b, c):
        lo, hi = np.minimum(np.minimum(a, b), c), np.maximum(np.maximum(a, b), c)
        return np.where(lo > 0, lo, np.where(hi < 0, hi, 0 * a))

    for _ in range(steps):
        d = np.roll(u, -1) - u                     # to the next cell
        m1, m3, p3 = np.roll(d, 1), np.roll(d, 2), np.roll(d, -1)
        c = d - m1
        S = (minmod3(p3 - d, h * (p3 - m1), c), minmod3(c, h * (d - m3), m1 - m3))
        D = (d, m1)
        P = (D[0] - h * S[0], D[1] + h * S[1])
        a = np.maximum(0, np.maximum(np.sign(P[0]), np.sign(P[1])))
        b = np.minimum(0, np.minimum(np.sign(P[0]), np.sign(P[1])))
        w = np.where(a - b > 0, a - b, 1)
        weight = (np.where(a - b > 0, -b / w, h), np.where(a - b > 0, a / w, h))
        inc = 0 * u
        for s, (e, cx) in enumerate(((a * r, 1), (b * r, -1))):
            p = D[s] + S[s] * (e - h * cx)
            p = p - h * r * S[s] * np.sign(p)
            inc = inc + weight[s] * (e * (D[s] + h * S[s] * (e - cx)) - r * np.abs(p))
        u = u + inc
    return u


@pytest.mark.skipif(np.finfo(np.longdouble).eps > 2.0 ** -60, reason="needs a wider long double")
def test_long_run_does_not_drift():
    """Two walls that annihilate, 200 steps, down to 1e-40 of the start: against the same run in long
    doubles.  Rounding of the state alone is a random walk of 200 halvings (200^1/2 2^-54 = 8e-16 relative
    at one node), which the FP64 oracle's distance from that run measures; a bias of 2^-55 in each step
    would come to 5.6e-15.  Bar: four times the oracle's distance, over four wall pairs together."""
    n1, n2, steps, cfl = 128, 16, 200, 0.5
    gpu = cpu = 0.0
    x = np.arange(n1, dtype=np.float64)
    for a, b in ((-0.31, 0.12), (0.22, -0.4), (0.47, 0.35), (-0.08, -0.27)):
        s, sep = 3.0 * (1 + 0.2 * a), n1 / 4.0 * (1 + 0.1 * b)
        row = np.array([s * sqrt(pi / 2) * (erf((t - n1 / 2 + sep / 2) / (s * sqrt(2)))
                                            - erf((t - n1 / 2 - sep / 2) / (s * sqrt(2)))) for t in x])
        u = np.repeat(row[None, :], n2, axis=0)
        exact = annihilation(row.astype(np.longdouble), steps, cfl)
        p = Params(n1=n1, n2=n2, nz=16, nh=4, v0=1.0, theta=1.0, cfl=cfl, autotune=0)
        op = oracle.Params(**{k: getattr(p, k) for k in oracle.Params.__dataclass_fields__})
        ref, rc = oracle.run(op, u, steps, K=np.zeros((n2, n1)))
        assert rc == 0
        with FDM(p) as sim:
            sim.set_plastic_distortion(u)
            sim.step(steps)
            got = sim.read_fields("up13")["up13"]
        norm = np.linalg.norm(exact.astype(np.float64))
        assert 0 < norm < 1e-30

        def distance(v):
            return float(np.sqrt(np.mean([np.sum(((w.astype(np.longdouble) - exact) / norm) ** 2) for w in v])))
        gpu += distance(got) ** 2
        cpu += distance(ref.up13) ** 2
    assert gpu ** 0.5 <= 4 * cpu ** 0.5


@pytest.mark.parametrize("power", [-620, -520, 400])
@pytest.mark.parametrize("v0", [1.0, -1.0])
@pytest.mark.parametrize("n1,n2", [(64, 32), (1024, 256)])
def test_update_takes_celerities_of_any_size(power, v0, n1, n2):
    """Under the CFL rule a step depends on the celerity's sign and relative size alone: with 2^p v0 it is
    the oracle's step with v0, to the rounding of either (1e-14 as above)."""
    u = np.random.default_rng(15).standard_normal((n2, n1))
    _, want = one_step(u, 1.7, v0)
    p = Params(n1=n1, n2=n2, nz=16, nh=4, v0=float(np.ldexp(v0, power)), theta=1.7, cfl=0.45, autotune=0)
    with FDM(p) as sim:
        sim.set_plastic_distortion(u)
        sim.step(1)
        got = sim.read_fields("up13")["up13"]
    assert np.linalg.norm(got - want) <= 1e-14 * np.linalg.norm(want - u)
