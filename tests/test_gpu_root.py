"""Root bounds of convolutional networks over patches against the FP64 oracle (needs a GB300):
strides, paddings, kernels and map sizes where the patches touch the border, cover a map's odd
remainder, fit only some layers' maps, or run through three convolutions; several properties at once.
The oracle works on explicit matrices of the whole maps."""
import numpy as np
import pytest
import torch

from oracle import bcrown_oracle as O
from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl
from tests.helpers import rel_err

pytestmark = pytest.mark.gpu

NETS = {
    "two_strided": ((2, 13, 11), [(3, 4, 2, 1), (4, 4, 2, 1)]),
    "three_3x3": ((1, 15, 17), [(2, 3, 1, 1), (3, 3, 2, 1), (2, 3, 1, 1)]),
    "no_padding": ((2, 12, 9), [(3, 3, 1, 0), (3, 2, 2, 0)]),
    "stride_over_kernel": ((1, 16, 16), [(3, 3, 1, 1), (2, 2, 3, 0)]),
    "last_layer_dense": ((1, 9, 9), [(2, 3, 2, 1), (2, 3, 1, 1), (2, 3, 1, 1)]),   # the last patch outgrows its maps
    "pointwise": ((3, 8, 8), [(4, 1, 1, 0), (3, 3, 1, 1)]),
}


@pytest.mark.parametrize("which", list(NETS))
@pytest.mark.parametrize("n_props", [1, 3])
def test_conv_root_bounds(which, n_props):
    shape, convs = NETS[which]
    pb = wl.make_problem(which, wl.conv_layers(shape, convs, [7, 4], 3), n_props, 0.1, 3, 3)
    net = bc.load_net(pb.layers, pb.C)
    x_lo, x_hi = torch.as_tensor(pb.x_lo).cuda(), torch.as_tensor(pb.x_hi).cuda()
    onet = O.OracleNet(pb.layers, pb.C)
    l_ref, u_ref = O.root_bounds(onet, pb.x_lo, pb.x_hi)
    l, u, cnt = bc.root_bounds(net, x_lo, x_hi, precision=bc.FP32)
    assert bc.status(net) == 0
    assert rel_err(l.cpu().numpy(), l_ref).max() <= 1e-5 and rel_err(u.cpu().numpy(), u_ref).max() <= 1e-5
    assert np.array_equal(cnt.cpu().numpy(), ((l < 0) & (u > 0)).sum(1).cpu().numpy())
    # certified: sound against sampled pre-activations of the exact network, and as close as the a
    # priori terms allow (the bar of the other nets)
    lc, uc, _ = (x.cpu().numpy() for x in bc.root_bounds(net, x_lo, x_hi, precision=bc.CERTIFY))
    rng = np.random.default_rng(0)
    for p in range(n_props):
        xs = rng.uniform(pb.x_lo[p].astype(np.float64), pb.x_hi[p].astype(np.float64), size=(500, pb.x_lo.shape[1]))
        z = np.concatenate([zi for zi in onet.preacts(xs)[1:]], axis=1)
        assert np.all(z >= lc[p] - 1e-9) and np.all(z <= uc[p] + 1e-9)
    assert rel_err(lc, l_ref).max() <= 2e-2 and rel_err(uc, u_ref).max() <= 2e-2
    # the fixed rule reaches the same code with another slope
    lf, uf, _ = bc.root_bounds(net, x_lo, x_hi, bc.ALPHA_FIXED, 0.25, bc.FP32)
    l_fix, u_fix = O.root_bounds(onet, pb.x_lo, pb.x_hi, O.ALPHA_FIXED, 0.25)
    assert rel_err(lf.cpu().numpy(), l_fix).max() <= 1e-5 and rel_err(uf.cpu().numpy(), u_fix).max() <= 1e-5


def test_root_bounds_of_a_fully_connected_net_do_not_depend_on_the_other_properties():
    """All properties' rows run together: each property's bounds equal those of its own call."""
    pb = wl.make_problem("fc", wl.mlp_layers([9, 33, 20, 65, 4], 2), 5, 0.1, 3, 2)
    net = bc.load_net(pb.layers, pb.C)
    x_lo, x_hi = torch.as_tensor(pb.x_lo).cuda(), torch.as_tensor(pb.x_hi).cuda()
    for precision in (bc.FP32, bc.CERTIFY):
        l, u, cnt = bc.root_bounds(net, x_lo, x_hi, precision=precision)
        for p in range(5):
            l1, u1, c1 = bc.root_bounds(net, x_lo[p:p + 1].contiguous(), x_hi[p:p + 1].contiguous(), precision=precision)
            assert torch.equal(l[p:p + 1], l1) and torch.equal(u[p:p + 1], u1) and torch.equal(cnt[p:p + 1], c1)
