"""The stacked-state solve on each of the ways its layers can run: three layers on the fused kernels with ragged lengths and F-cycles,
a serial sweep by chains, batches beyond the fused kernels' 128 rows, chains that do not fit, fp32 widths with and without the
persistent solve, repeated relaxations.  The checks are those of the stacked parity test: everything against the fp64 oracle."""
import pytest

from tests.test_gpu_stacked import test_stacked_solve as check

pytestmark = pytest.mark.gpu

CASES = [
    dict(T=61, B=8, I=16, H=64, cf=2, levels=3, nl=3, rf=1, rc=2, flags=6, op=2),
    dict(T=40, B=9, I=16, H=320, cf=4, levels=1, nl=2, rf=0, rc=0, flags=0, op=2),
    dict(T=32, B=130, I=16, H=64, cf=4, levels=2, nl=2, rf=1, rc=0, flags=0, op=2),
    dict(T=32, B=100, I=16, H=1024, cf=4, levels=2, nl=2, rf=0, rc=0, flags=1, op=2),
    dict(T=30, B=2, I=16, H=360, cf=4, levels=2, nl=2, rf=1, rc=0, flags=4, op=0),
    dict(T=50, B=5, I=8, H=136, cf=3, levels=3, nl=2, rf=2, rc=1, flags=5, op=0),
    dict(T=21, B=1, I=8, H=40, cf=20, levels=2, nl=2, rf=1, rc=0, flags=4, op=0),
]


@pytest.mark.parametrize("c", CASES, ids=lambda c: "T{T}B{B}H{H}cf{cf}L{levels}nl{nl}r{rf}{rc}f{flags}o{op}".format(**c))
def test_stacked_paths(c):
    check(c)
