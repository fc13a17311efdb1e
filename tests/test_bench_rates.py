"""The benchmark compares a stencil with the arithmetic rate that bounds it: mixed and double words,
which take the whole scheme at every node; FP64, whose nodes compute in integers, has none."""
import bench


def test_stencil_rates():
    assert {p: k for p, (k, _) in bench.STENCIL_PEAK.items()} == {"mixed": "fp32", "df64": "df64"}
