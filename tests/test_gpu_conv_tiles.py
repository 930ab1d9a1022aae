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


@pytest.mark.gpu
@pytest.mark.parametrize("H,W", [(8, 8), (64, 64), (64, 72), (32, 128), (16, 136), (64, 256), (32, 264), (64, 512)])
def test_counted_launches_are_those_of_a_forward_pass(H, W):
    """The kernels a forward pass is counted as (ibm_profile's launches) are the
    kernel nodes of a captured one: levels of at most 64 pixels a row pool in a
    kernel of their own."""
    import ctypes as C

    import torch
    import paper_2402_17337_gb300 as ibm
    from paper_2402_17337_gb300 import build
    build.build()
    net = ibm.UNet((16, 16, 32, 32), seed=1)
    feat = torch.zeros(H, W, 4, device="cuda")
    out = torch.empty(H, W, device="cuda")
    rt = C.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    stream = torch.cuda.Stream()
    args = net._h, feat.data_ptr(), H, W, out.data_ptr(), stream.cuda_stream
    torch.cuda.synchronize()
    assert ibm.lib().ibm_unet_forward(*args) == 0  # allocates, packs the weights
    stream.synchronize()
    s, graph, n = C.c_void_p(stream.cuda_stream), C.c_void_p(), C.c_size_t(0)
    assert rt.cudaStreamBeginCapture(s, 2) == 0
    rc = ibm.lib().ibm_unet_forward(*args)
    assert rt.cudaStreamEndCapture(s, C.byref(graph)) == 0 and rc == 0
    assert rt.cudaGraphGetNodes(graph, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, C.byref(n)) == 0
    kinds = []
    for node in nodes:
        k = C.c_int(-1)
        assert rt.cudaGraphNodeGetType(C.c_void_p(node), C.byref(k)) == 0
        kinds.append(k.value)
    rt.cudaGraphDestroy(graph)
    counted = getattr(ibm.lib(), "_ZN3ibm21unet_forward_launchesEii")(H, W)
    assert kinds.count(0) == counted == 16 + sum(W >> level <= 64 for level in range(3))
    net.close()
