"""Pruned attention at the edges of its K/V tiles, against the oracle."""
import pytest
import torch

from test_gpu_parity import test_pruned_attention_matches_oracle as _matches_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", [2, 3, 5, 6])
@pytest.mark.parametrize("S,window,ratio", [(700, 1, 0.5), (700, 127, 0.5), (700, 128, 0.0), (700, 129, 0.3), (1000, 383, 0.7), (1290, 33, 0.0)])
def test_windows_that_start_inside_a_tile(path, S, window, ratio):
    """Masks of both ends in one tile, whole words of columns visible or not, tiles that reach past the last token."""
    _matches_oracle(torch.bfloat16, path, 1, S, 8, 2, window, ratio)


@pytest.mark.parametrize("path", [2, 3, 5, 6])
@pytest.mark.parametrize("S,window", [(514, 0), (770, 200), (1030, 0)])
def test_last_row_blocks_of_few_rows(path, S, window):
    """The rows of a tile that do not exist see everything and go nowhere, behind tiles that are cut for those that do."""
    _matches_oracle(torch.bfloat16, path, 2, S, 8, 2, window, 0.0)
