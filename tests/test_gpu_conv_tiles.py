"""Channel counts and sizes at the edges of the convolutions' tiling.

The chunks of input channels (64, 32 or 16), the tiles of output channels
(halved on small levels, with a shorter last tile) and the stacked rows depend
on the layer.  In the exact regime of test_unet.py every output and gradient
has one correct value, so the comparison with the oracle is bit for bit.
"""
import numpy as np
import pytest

import test_unet as T

# widths, H, W, seed, share of pixels with a loss
CASES = [((80, 16, 112, 144), 16, 24, 5, 1 / 16),   # chunks of 16; 144 = two tiles of 64 and one of 16
         ((48, 96, 32, 64), 24, 136, 6, 1 / 32),    # one row of 128 pixels and a ragged 8; 96 channels halved to 48
         ((32, 64, 128, 128), 8, 16, 2, 1 / 2)]       # a 1x2 bottom level


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES)
def test_tiles_exact(case):
    T.test_gpu_unet_matches_oracle_bit_for_bit_in_the_exact_regime(case)
