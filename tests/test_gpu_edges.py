"""GPU parity at the edges of the kernels' tiles and dispatch rules: the checks (and their bounds) are those of
test_gpu_parity.py, the cases are the sizes where a tile is ragged, a tile holds several images, or a variant begins or ends."""

import pytest

import test_gpu_parity as parity

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# N, n_ci, n_co, H, W, P_ci, P_co, P_0, P_1, k
CONVG_EDGES = [
    (7, 2, 9, 14, 14, 1, 1, 2, 2, 5),        # 7 x 7 shards, several images a tile, the last tile of images partly empty; 9 = 5 + 4 channels
    (19, 3, 7, 9, 17, 1, 1, 1, 1, 3),        # odd rows; 7 channels: four pairs, the last half empty
    (5, 1, 1, 3, 3, 1, 1, 1, 1, 7),          # a kernel wider than the image, one channel each way
    (2, 9, 3, 18, 40, 2, 1, 1, 1, 7),        # 16-float windows, uneven input blocks (5, 4)
    (1, 2, 17, 33, 129, 1, 2, 1, 1, 5),      # 9 and 8 channels: groups of 5, 4 and 8; one cell past tile edges
    (3, 6, 5, 20, 31, 1, 1, 3, 1, 3),        # uneven rows (7, 7, 6) beside odd columns
]


@pytest.mark.parametrize("case", CONVG_EDGES, ids=[str(c) for c in CONVG_EDGES])
@pytest.mark.parametrize("integer", [True, False], ids=["int", "normal"])
def test_generalized_conv_tiles(case, integer):
    parity.test_generalized_conv_fwd_and_adj(case, integer)
    parity.test_generalized_conv_param_gradients(case, integer)
