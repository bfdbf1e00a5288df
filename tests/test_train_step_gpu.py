"""The fused training step at the edges of its tiles: ragged batches (32-row
blocks, 64-row chunks), widths and outputs off
the padding, the largest network it takes and the first one beyond it."""
import pytest

import test_mlp_gpu as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,w,d_out,B", [
    (258, 256, 8, 1), (258, 256, 8, 31), (258, 256, 8, 33), (258, 256, 8, 512), (258, 256, 8, 777),
    (1, 1, 1, 5), (33, 30, 9, 65), (512, 256, 32, 300), (100, 250, 17, 129),
    (513, 64, 8, 70), (40, 264, 8, 70), (40, 64, 33, 70)])
def test_gradients(d_in, w, d_out, B):
    M.test_gradients_match_oracle(d_in, w, d_out, B)
