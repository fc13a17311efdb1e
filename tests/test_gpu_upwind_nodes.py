"""The FP64 stencil updates nodes of one characteristic direction by a short form and collects the
others for the whole scheme: fields that send every node, none, few or whole tiles to either, on
launches of one wave and of several (where left-over nodes go through the instance's list),
against the oracle; double words, which take the whole scheme at every node, on the same fields.

Tolerance (relative L2 of the increment): 1e-11, the parity bar of both paths; the increments are
of the field's own size.  Three steps where minmod contracts rounding; one where it cannot: with
the MC limiter, and for the field that borders exact ties (derivatives that are zero in exact
arithmetic) with noise, where the oracle itself moves by 5e-3 under a perturbation of 1e-16."""
import numpy as np
import pytest

import oracle
from paper_1911_03225_gb300 import FDM, Batch, Params
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
    x, y = np.arange(n1)[None, :] / n1, np.arange(n2)[:, None] / n2
    if kind == "noise":        # every limiter and direction decision, nearly every node for the whole scheme
        return np.random.default_rng(3).standard_normal((n2, n1))
    if kind == "smooth":       # nearly every node short
        return np.sin(2 * np.pi * x) * np.cos(2 * np.pi * (y + 0.1)) + 0.3 * np.sin(4 * np.pi * (x + y))
    if kind == "walls_x":      # nothing varies along x2: its weights are halves
        return np.maximum(0.0, np.sin(2 * np.pi * x)) * 8.0 + 0.0 * y
    if kind == "walls_y":
        return np.maximum(0.0, np.sin(2 * np.pi * y)) * 8.0 + 0.0 * x
    if kind == "tents":        # kinks along lines, flat parts between
        return np.maximum(0.0, 0.2 - np.abs(x - 0.5)) * n1 / 8 + np.maximum(0.0, 0.1 - np.abs(y - 0.3)) * n2 / 8
    u = np.sin(2 * np.pi * x) + 0.0 * y   # half smooth, half noise
    u[n2 // 2:, : n1 // 2] += np.random.default_rng(4).standard_normal((n2 - n2 // 2, n1 // 2))
    return u


@pytest.mark.parametrize("kind", ["noise", "smooth", "walls_x", "walls_y", "tents", "mixed"])
@pytest.mark.parametrize("n1,n2", [(16, 16), (64, 32), (1024, 512)])
@pytest.mark.parametrize("precision", [B.FP64, B.DF64])
@pytest.mark.parametrize("v0,theta,level", [(1.0, 1.0, B.T_MIDPOINT), (-1.0, 1.7, B.T_LITERAL)])
def test_short_and_whole_nodes_match_oracle(kind, n1, n2, precision, v0, theta, level):
    u = field(kind, n1, n2)
    p = Params(n1=n1, n2=n2, nz=16, nh=4, v0=v0, theta=theta, time_level=level, cfl=0.45, precision=precision,
               autotune=0)
    op = oracle.Params(**{k: getattr(p, k) for k in oracle.Params.__dataclass_fields__})
    K = np.zeros((n2, n1))   # the prescribed celerity needs no stress
    steps = 3 if theta == 1.0 and kind != "mixed" else 1
    ref, rc = oracle.run(op, u, steps, K=K)
    assert rc == 0
    with FDM(p) as sim:
        sim.set_plastic_distortion(u)
        sim.step(steps)
        got = sim.read_fields("up13")["up13"]
    assert np.linalg.norm(got - ref.up13) <= 1e-11 * np.linalg.norm(ref.up13 - u)


def test_batch_lists_are_per_instance():
    """Several waves of blocks from several instances: each instance's left-over nodes are its own."""
    n, steps = 256, 4
    p = Params(n1=n, n2=n, nz=16, nh=4, v0=1.0, theta=1.0, cfl=0.4)
    kinds = ["tents", "smooth", "mixed", "noise", "walls_x", "tents", "mixed", "smooth"] * 2
    fields = [field(k, n, n) * (1.0 + 0.1 * i) for i, k in enumerate(kinds)]
    with Batch([p] * len(fields)) as b:
        for i, u in enumerate(fields):
            b.set_plastic_distortion(i, u)
            b.set_budget(i, steps - (i & 1))
        b.enqueue_steps(steps)
        b.sync()
        got = [b.read_fields(i, "up13")["up13"] for i in range(len(fields))]
    with FDM(p) as sim:
        for i, u in enumerate(fields):
            sim.set_plastic_distortion(u)
            sim.step(steps - (i & 1))
            np.testing.assert_array_equal(sim.read_fields("up13")["up13"], got[i])
