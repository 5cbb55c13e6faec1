"""What a row's bits depend on: its own data only (needs a GB300).  A small network's rows
have the same bits whichever kernel the batch's size takes and in bcrown_bound_static; a property's place
among the others, which moves its tables off the 16-byte boundaries, changes nothing either."""
import numpy as np
import pytest
import torch

from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl
from tests.helpers import oracle_setup

pytestmark = pytest.mark.gpu


def _t(x):
    return torch.as_tensor(np.ascontiguousarray(x, np.float32)).cuda()


def _problem(widths, n_props, eps=0.2):
    pb = wl.make_problem("bits", wl.mlp_layers(widths, 3), n_props, eps, 2, 4)
    _, props, unst = oracle_setup(pb)
    return pb, unst, bc.load_net(pb.layers, pb.C), bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])


@pytest.mark.parametrize("widths", [
    [3, 1, 2], [16, 32, 32, 4], [33, 31, 64, 62, 2], [64, 64, 7, 3], [31, 33, 2],     # a warp per row
    [33, 31, 64, 65, 2], [65, 9, 3], [37, 300, 260, 5], [257, 255, 256, 2], [784, 20, 512, 3],   # a block
    [9, 8, 8, 8, 8, 8, 8, 2],
])
def test_one_launch_and_layers_have_the_same_bits(widths):
    pb, unst, net, dom = _problem(widths, 3)
    most = min(6, min(len(u) for u in unst))
    batch = wl.random_batch(pb, unst, 50, most // 2, most, 5)
    a, b = (_t(x) for x in wl.random_alpha_beta(batch, 6, 1.0))
    db = bc.DeviceBatch.from_host(batch)
    n0 = bc.kernel_launches()
    lb = bc.bound(net, dom, db, a, b, bc.FP32)
    assert bc.kernel_launches() - n0 == 1
    assert torch.equal(lb, bc.bound_static(net, dom, db, a, b))
    assert bc.status(net) == 0


@pytest.mark.parametrize("widths,B", [([40, 96, 80, 4], 9000), ([37, 300, 260, 5], 1600), ([300, 30, 3], 40000)])
def test_a_row_does_not_depend_on_the_batch(widths, B):
    """Bound, gradient and minimising corner of a batch's first subdomains, alone and among many."""
    pb, unst, net, dom = _problem(widths, 2, 0.1)
    U = np.array([len(u) for u in unst])
    big = wl.random_batch(pb, unst, B, 0, 6, 3)
    n = 50
    na, ns = int((U[big.prop_of[:n]] * pb.K).sum()), int(big.split_cnt[:n].sum())
    small = wl.Batch(big.prop_of[:n], big.split_off[:n], big.split_cnt[:n], big.split_layer[:ns], big.split_idx[:ns],
                     big.split_sign[:ns], big.alpha_off[:n], na, ns * pb.K)
    a, b = (_t(x) for x in wl.random_alpha_beta(big, 5, 0.5))
    got = []
    for batch, x, y in ((small, a[:na], b[:ns * pb.K]), (big, a, b)):
        db = bc.DeviceBatch.from_host(batch)
        n0 = bc.kernel_launches()
        out = bc.bound_grad(net, dom, db, x, y, bc.FP32)
        assert (bc.kernel_launches() - n0 == 1) == (batch is small)
        got.append(list(out) + [v.reshape(-1) for v in bc.bound_xstar(net, dom, db, x, y)])
        assert torch.equal(got[-1][0], got[-1][3])
        assert bc.status(net) == 0
    for s, l in zip(*got):
        assert torch.equal(s, l[:s.numel()])


@pytest.mark.parametrize("which", ["mlp", "mlp_odd", "wide"])
@pytest.mark.parametrize("precision", [bc.FP32, bc.CERTIFY])
def test_a_row_does_not_depend_on_its_property_s_place(which, precision):
    """The same property four times, its hidden neurons no multiple of 4."""
    layers = {"mlp": lambda: wl.mlp_layers([20, 640, 128, 30, 4], 3), "mlp_odd": lambda: wl.mlp_layers([20, 636, 129, 64, 4], 3),
              "wide": lambda: wl.conv_layers((3, 24, 24), [(8, 3, 1, 1)], [30, 4], 3)}[which]()
    pb = wl.make_problem("place", layers, 1, 0.05, 3, 4)
    _, props, unst = oracle_setup(pb)
    assert props["l"].shape[1] % 4
    net = bc.load_net(pb.layers, pb.C)
    dom = bc.domain_from_host(*(np.repeat(props[k], 4, 0) for k in ("x_lo", "x_hi", "l", "u")))
    one = wl.random_batch(pb, unst, 600, 1, 6, 5)
    a, b = (_t(x) for x in wl.random_alpha_beta(one, 6, 1.0))
    got = []
    for p in range(4):
        one.prop_of[:] = p
        db = bc.DeviceBatch.from_host(one)
        got.append(bc.bound(net, dom, db, a, b, precision))
        if precision == bc.FP32:
            assert torch.equal(bc.bound_static(net, dom, db, a, b), got[-1])
    assert bc.status(net) == 0
    for g in got[1:]:
        assert torch.equal(g, got[0])


@pytest.mark.parametrize("which", ["mlp", "odd_maps"])
def test_a_bf16_layer_path_row_does_not_depend_on_the_batch(which):
    """Subdomains of a property with few unstable neurons, alone in a ragged tile and among those of one with
    many: bound and gradient.  Both networks have warps that hold several rows."""
    layers = {"mlp": lambda: wl.mlp_layers([37, 300, 260, 5], 11),
              "odd_maps": lambda: wl.conv_layers((4, 7, 7), [(24, 3, 1, 1), (72, 3, 2, 1)], [40, 4], 3)}[which]()
    pb = wl.make_problem("bits", layers, 2, 0.02, 3, 4)
    pb.x_lo[1] -= 0.5
    pb.x_hi[1] += 0.5
    _, props, unst = oracle_setup(pb)
    U = np.array([len(u) for u in unst])
    assert U[0] < 0.25 * props["l"].shape[1] < 0.5 * U[1]
    net = bc.load_net(pb.layers, pb.C)
    bc.set_launch(net, bc.N.PATH_LAYER_EPI)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    n = 7
    big = wl.random_batch(pb, unst, 150, 1, 8, 5, props=np.where(np.arange(150) < n, 0, np.arange(150) % 2))
    na, ns = int((U[big.prop_of[:n]] * pb.K).sum()), int(big.split_cnt[:n].sum())
    small = wl.Batch(big.prop_of[:n], big.split_off[:n], big.split_cnt[:n], big.split_layer[:ns], big.split_idx[:ns],
                     big.split_sign[:ns], big.alpha_off[:n], na, ns * pb.K)
    a, b = (_t(x) for x in wl.random_alpha_beta(big, 6, 1.0))
    got = [bc.bound_grad(net, dom, bc.DeviceBatch.from_host(x), y, z, bc.BF16)
           for x, y, z in ((small, a[:na], b[:ns * pb.K]), (big, a, b))]
    assert bc.status(net) == 0
    for s, l in zip(*got):
        assert torch.equal(s, l[:s.numel()])
