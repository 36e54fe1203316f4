"""How many rows a thread of the rotary kernel takes (host logic, no GPU)."""
import pytest

from paper_2408_08146_b200 import binding

CLUSTERS = 74                                            # CTA pairs that are resident at once on 148 SMs


def _rows(R, H, tile_rows, n=3, ctas=CLUSTERS):
    tiles = 3 * H // tile_rows * -(-R // 256)            # weight tiles times token tiles of at most 256 rows
    return binding.load_library().koala_debug_rope_rows(R, H, ctas, tiles, H // 64, n)


@pytest.mark.parametrize("R,H,want", [(129, 4096, 1), (257, 4096, 1), (300, 4096, 1), (360, 4096, 1), (509, 4096, 2),
                                      (1024, 4096, 2), (257, 5120, 1), (509, 5120, 2), (860, 5120, 2)])
def test_prompts_take_two_rows_where_the_launch_still_fills_the_sms(R, H, want):
    assert _rows(R, H, 256) == want
    if want == 2:
        assert (R + 1) // 2 * (H // 4) >= 148 * 1280


@pytest.mark.parametrize("R", [257, 300, 432, 512])
@pytest.mark.parametrize("H", [4096, 5120])
def test_verifications_take_one_row(R, H):
    """512 weight rows per tile: most columns have two or three partial sums, whose trips a second row would repeat."""
    assert _rows(R, H, 512) == 1


def test_whole_parts_and_many_sums_take_one_row():
    assert _rows(509, 4096, 256, ctas=0) == 1 and _rows(509, 4096, 256, n=5) == 1
