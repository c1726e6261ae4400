"""z-MIP backward with more tiles than resident CTAs, where the tiles are
stored without the TMA unit and the last block of columns is partly past the
grid's edge (rows that are not a multiple of 16 bytes, or an output that does
not start on one): a CTA goes on to its next tile after such a block."""
import numpy as np
import pytest

import oracle as O
from gpu_util import assert_close, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# tiles of 32 columns x 8 rows x 16 planes; five CTAs run per SM
SHAPES = [(160, 320, 37, 60.0, 0.125, 0.125), (64, 112, 438, 60.0, 0.125, 0.125), (210, 333, 33, 35.0, 0.3, 0.1),
          (70, 120, 447, 45.0, 0.2, 0.25), (160, 328, 40, 35.0, 0.3, 0.1)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("offset", [0, 1])
def test_tiles_after_a_partial_block(lib, shape, offset):
    """Every sample is written (the output is pre-filled with NaN and starts
    `offset` floats into its buffer) and is the oracle's."""
    g = O.geometry(*shape)
    plan = lib.Plan(*shape)
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    assert -(-shape[2] // 32) * -(-shape[1] // 8) * -(-shape[0] // 16) > 5 * nsm
    rng = np.random.default_rng(7)
    argz = rng.integers(0, g.nz, size=(g.ny, g.nx)).astype(np.int32)
    gz = rng.standard_normal((g.ny, g.nx)).astype(np.float32)
    n = int(np.prod(plan.raw_shape))
    G = torch.full((n + offset,), np.nan, device="cuda")[offset:].view(plan.raw_shape)
    lib.opm_mip_backward(plan, to_dev(gz, torch), to_dev(argz, torch), G)
    torch.cuda.synchronize()
    assert_close(G.cpu().numpy(), O.mip_backward(gz.astype(np.float64), argz, g), what="mip backward")
