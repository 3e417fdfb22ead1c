"""lb_batch_config reports the tiles and blocks that a form launches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# (shape, rows of a tile) with one block per tile: 64 x 37 has 2 x ceil(37 / rows) tiles of 32 x rows;
# shape 1 launches a block for each half of a 16-row tile.
@pytest.mark.parametrize("shape,rows,blocks", [(0, 16, 2 * (3 + 2)), (1, 16, 2 * 2 * (3 + 2)), (2, 32, 2 * (2 + 1))])
def test_reported_blocks(shape, rows, blocks):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import Batch, capi

    b = Batch([np.full((37, 64), 2.0), np.full((32, 64), 2.0)], [dict(Tr=0.85, rho_ref=2.0)] * 2)
    capi.check_batch(capi.lib().lb_batch_set_config(b.b, shape, 0), b.b)
    cfg = b.config()
    assert (cfg["tile_y"], cfg["blocks_per_sm"], cfg["grid"]) == (rows, 0, blocks)
