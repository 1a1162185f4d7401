"""Boxes of few long rows whose padded copies take several blocks a row: four-cell
against one-cell threads, as in test_gpu_blocks.py and with its tolerance."""
import pytest

from test_gpu_blocks import RM, test_four_cell_blocks_match_one_cell as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,kw", [((200001, 1, 1), RM), ((20002, 10, 1), {}), ((4003, 7, 8), RM),
                                      ((1021, 14, 14), RM), ((129, 1250, 2), {})])
def test_copies_of_long_rows(shape, kw):
    check(shape, kw)
