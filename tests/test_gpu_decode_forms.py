"""Decode steps at the sizes where one form of the attention gives way to another, against fp64 softmax attention."""
import pytest

from test_gpu_parity import test_decode_attention_uneven_positions_and_skips as _uneven_positions_and_skips

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("workspace", [True, False])
@pytest.mark.parametrize("B,S,Hkv,G,window", [
    (6, 30000, 4, 1, 0), (300, 200, 8, 1, 0)])                    # streaming: pieces of work items, whole ones; last tiles of 1 to 64 keys
def test_decode_attention_forms(B, S, Hkv, G, window, workspace):
    _uneven_positions_and_skips(B, S, Hkv, G, window, workspace)
