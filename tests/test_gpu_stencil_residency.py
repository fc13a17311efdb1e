"""The launch configuration reports the blocks per SM that the FP64 stencil is compiled for, and a
configuration saved with the figure of the time when that was two names the same shape."""
import pytest

from paper_1911_03225_gb300 import FDM, FDMError, Params
from paper_1911_03225_gb300 import binding as B

pytestmark = pytest.mark.gpu


def test_fp64_stencil_residency():
    p = Params(n1=64, n2=64, precision=B.FP64, autotune=0)
    shapes = {(c["stencil_block_rows"], c["stencil_nodes"], c["stencil_min_blocks"]) for c in B.launch_candidates(p)}
    assert shapes == {(8, 2, 4), (8, 1, 4), (16, 1, 1), (8, 4, 4)}
    with FDM(p) as sim:
        good = sim.launch_config()
        sim.set_launch_config({**good, "stencil_block_rows": 8, "stencil_nodes": 4, "stencil_min_blocks": 2})
        got = sim.launch_config()
        assert (got["stencil_block_rows"], got["stencil_nodes"], got["stencil_min_blocks"]) == (8, 4, 4)
        with pytest.raises(FDMError):
            sim.set_launch_config({**good, "stencil_min_blocks": 3})
