"""How the multiply's ring of stages is filled before its activations come (host logic, no GPU)."""
import ctypes as C

import pytest

from paper_2408_08146_b200 import binding

SMEM = 232448                                            # bytes of shared memory a block may opt in to (sm_100)
STAGES = [16384 + rows * 128 for rows in range(16, 257, 16)]     # 128 weight rows and the activation rows of a tile


def _ring(stage_bytes, wide=0, pdl=1):
    lib = binding.load_library()
    v = [C.c_int(0) for _ in range(3)]
    assert lib.koala_debug_gemm_ring(stage_bytes, SMEM, wide, pdl, *(C.byref(x) for x in v)) == 0
    return tuple(x.value for x in v)


@pytest.mark.parametrize("stage_bytes", STAGES)
def test_without_programmatic_launch_the_whole_ring_is_requested_at_once(stage_bytes):
    """Nothing runs before such a launch that the pacing could spare; not more than five stages begin together."""
    stages, early, pace = _ring(stage_bytes, pdl=0)
    assert 2 <= stages <= 5 and early == stages and pace == 0
    assert stages == min(5, _ring(stage_bytes)[0])


@pytest.mark.parametrize("stage_bytes", STAGES)
def test_two_stages_at_once_and_the_others_paced(stage_bytes):
    stages, early, pace = _ring(stage_bytes)
    assert early == 2 and (pace > 0) == (stages > 2)
    assert 2 * (stages * stage_bytes + 1024) <= SMEM       # two CTAs per SM


@pytest.mark.parametrize("value", [-1600, -1, 0])
def test_no_pace_below_zero(value):
    """Two threads share the requests of the later stages, one for a pace above zero and one for zero: a negative pace would
    leave them to nobody, and every multiply would run into its wait limit."""
    lib = binding.load_library()
    lib.koala_set_tuning(24, value)
    try:
        assert all(_ring(b)[2] == 0 for b in STAGES)
    finally:
        lib.koala_set_tuning(24, 1600)
