"""How the blocks of a batch of prompts are dealt to forwards (host logic, no GPU)."""
import ctypes as C

import pytest

from paper_2408_08146_b200 import binding


def _deal(lens, rows=1024, fail_at=-1):
    lib = binding.load_library()
    n, t = C.c_int(0), C.c_int(0)
    arr = (C.c_int32 * len(lens))(*lens)
    rc = lib.koala_debug_deal_blocks(len(lens), arr, rows, fail_at, C.byref(n), C.byref(t))
    return rc, n.value, t.value


@pytest.mark.parametrize("lens", [[1], [127], [128], [129], [2048] * 8, [700, 16, 333], [50] * 64, [2000] + [20] * 63])
def test_every_token_is_dealt_once(lens):
    rc, blocks, tokens = _deal(lens)
    assert rc == 0 and tokens == sum(lens) and blocks >= len(lens)


@pytest.mark.parametrize("fail_at", [0, 1, 5])
def test_a_failed_forward_ends_the_dealing(fail_at):
    """128 blocks of 128 tokens, eight per forward: nothing is dealt after the forward that failed."""
    rc, blocks, tokens = _deal([2048] * 8, fail_at=fail_at)
    assert rc == 5
    assert (blocks, tokens) == (8 * (fail_at + 1), 1024 * (fail_at + 1))
