"""The op graph's FP32 sweeps on rows of no multiple of four cells from the size where
a thread takes three planes, with planes left over: against the FP64 sweep (one cell a
thread) of the same step, as on the small shapes of test_gpu_sweeps.py and with their
tolerance (300 terms rounded to 2^-24, stencil weights of sum 2.5: 4.5e-5 of the norm)."""
import pytest

from test_gpu_sweeps import test_fp32_sweeps_match_fp64 as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(61, 53, 47), (99, 80, 17), (161, 137, 6), (231, 197, 3), (3, 210, 211)])
def test_three_planes_a_thread(shape):
    check(shape)
