"""The fp32 CUDA-core stage kernel at the edges of its tiles: 32 rows per CTA, units of 8, 16 or 32 columns, tiles of 1, 4, 8,
16 or 32 tokens, registers for 16 or 64 envelope modes, and reductions split over a cluster of CTAs."""
import numpy as np
import pytest
import torch

from paper_2512_24545_b200 import inputs
from helpers import GpuLayer, check_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2512_24545_b200 import build
    build.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("d_out,d_in,k,l,T", [
    (1, 1, 1, 1, 1), (31, 33, 32, 3, 2), (33, 31, 65, 4, 4),      # one unit, tails of a sign word
    (64, 127, 40, 5, 5), (32, 256, 64, 16, 8), (95, 257, 33, 16, 9),
    (40, 500, 96, 17, 16), (40, 100, 30, 64, 17), (64, 64, 64, 13, 32), (33, 130, 70, 2, 33),
    (100, 2050, 60, 4, 3),                                          # two ranks, an uneven last one
    (33, 9000, 50, 7, 40), (20, 8200, 32, 20, 1)])                  # more ranks than row tiles, both mode widths
def test_alu_tiles(d_out, d_in, k, l, T):
    spec = inputs.scaled(inputs.tiny(), name="alu", d_out=d_out, d_in=d_in, k=k, l=l, seed=900 + T)
    x = inputs.make_activations(spec, T)
    with GpuLayer(spec, T) as g:
        y = g.forward(x)
        check_parity(g, x, y, averaging=k >= 32)
        np.testing.assert_array_equal(y, g.forward(x))            # ranks and warps are added in a fixed order
