"""The FP32 convolution passes against the FP64 oracle (needs a GB300): output channels at each tile
width and past it, terms that leave a remainder, maps whose rows are no multiple of four, more stride
phases than a launch takes, phases without a tap, more than 32 taps in front of a narrow layer, and
the cells of 2 x 2 outputs over odd and even maps and paddings."""
import numpy as np
import pytest
import torch

from oracle import bcrown_oracle as O
from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl
from tests.helpers import RTOL, oracle_setup, rel_err

pytestmark = pytest.mark.gpu

NETS = {
    "tile16": ((5, 7, 9), [(16, 3, 1, 1), (7, 3, 2, 1)]),
    "tile32_64": ((1, 8, 8), [(17, 3, 1, 1), (33, 4, 2, 1)]),
    "tile128": ((2, 5, 6), [(65, 3, 1, 1), (70, 2, 1, 0)]),
    "two_tiles": ((3, 4, 4), [(130, 3, 1, 1), (6, 3, 1, 1)]),
    "nine_phases": ((3, 13, 10), [(5, 4, 3, 1), (6, 3, 1, 1)]),
    "empty_phases": ((4, 9, 9), [(5, 2, 3, 0), (3, 2, 1, 0)]),
    "many_taps": ((2, 9, 11), [(3, 7, 1, 3), (8, 3, 2, 0)]),
    "cells_stride_2": ((3, 13, 11), [(6, 4, 2, 1), (5, 3, 1, 1)]),   # odd maps: cells half outside
    "cells_even_padding": ((4, 9, 10), [(5, 4, 2, 0), (3, 2, 1, 0)]),
    "cells_padding_2": ((1, 8, 8), [(7, 4, 2, 2), (3, 3, 1, 1)]),
    "cells_stride_1": ((2, 7, 5), [(4, 3, 1, 0), (4, 4, 2, 1)]),
    "pointwise": ((3, 6, 6), [(8, 1, 1, 0), (20, 1, 2, 0)]),
}


@pytest.mark.parametrize("which", list(NETS))
def test_conv_passes(which):
    shape, convs = NETS[which]
    pb = wl.make_problem(which, wl.conv_layers(shape, convs, [7, 4], 3), 2, 0.1, 3, 3)
    onet, props, unst = oracle_setup(pb)
    batch = wl.random_batch(pb, unst, 21, 0, 4, 5)   # rows that end inside a tile
    a, b = wl.random_alpha_beta(batch, 6, 1.0)
    net = bc.load_net(pb.layers, pb.C)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    ref, da_ref, db_ref = O.grad(onet, props, batch, a.astype(np.float64), b.astype(np.float64))
    out = bc.bound_grad(net, dom, bc.DeviceBatch.from_host(batch), torch.from_numpy(a).cuda(),
                        torch.from_numpy(b).cuda(), bc.FP32)
    assert bc.status(net) == 0
    assert np.max(rel_err(out[0].cpu().numpy(), ref)) <= RTOL
    for g, gr in zip(out[1:], (da_ref, db_ref)):   # the gradient bar of the other convolutional nets
        scale = max(np.abs(gr).max(initial=0), 1e-6)
        assert np.max(np.abs(g.cpu().numpy() - gr), initial=0) <= 1e-4 * scale
