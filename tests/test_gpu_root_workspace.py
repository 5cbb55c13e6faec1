"""The workspace that root bounds of many properties take (needs a GB300): bounded, since the net keeps it and
captured graphs depend on its address, and without effect on the bounds."""
import numpy as np
import pytest
import torch

from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_many_properties_in_bounded_workspace():
    P = 40   # 40 x 512 rows of 15.6 KB: 320 MB, more than two chunks
    pb = wl.make_problem("root_ws", wl.mlp_layers([784] + [256] * 6 + [10], 3), P, 0.01, 2, 4)
    net = bc.load_net(pb.layers, pb.C)
    lo, hi = (torch.as_tensor(np.ascontiguousarray(x)).cuda() for x in (pb.x_lo, pb.x_hi))
    l, u, n = bc.root_bounds(net, lo, hi)
    assert bc.workspace(net)[1] <= 192 << 20
    for p in (0, 16, 17, 39):   # (the first chunk ends inside property 16)
        l1, u1, n1 = bc.root_bounds(net, lo[p:p + 1].contiguous(), hi[p:p + 1].contiguous())
        assert torch.equal(l1[0], l[p]) and torch.equal(u1[0], u[p]) and n1[0] == n[p]
