"""The one-launch FP32 kernel of small fully connected networks against the FP64 oracle and against the
layer-by-layer path (needs a GB300): a warp and a block per row, widths around its 32, 64 and 256
threads, one hidden layer and several, one and more properties, split lists from none to the longest."""
import numpy as np
import pytest
import torch

from oracle import bcrown_oracle as O
from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl
from tests.helpers import RTOL, oracle_setup, rel_err

pytestmark = pytest.mark.gpu


def _t(x):
    return torch.as_tensor(np.ascontiguousarray(x, np.float32)).cuda()


@pytest.mark.parametrize("widths", [
    [3, 1, 2], [16, 32, 32, 4], [33, 31, 64, 65, 2], [64, 64, 7, 3],     # the second is a block's (65 outputs)
    [65, 9, 3], [37, 300, 260, 5], [257, 255, 256, 2], [2048, 20, 512, 3], [9, 8, 8, 8, 8, 8, 8, 2],
])
@pytest.mark.parametrize("n_props,max_splits", [(1, 0), (3, 5), (2, 64)])
def test_rows(widths, n_props, max_splits):
    pb = wl.make_problem("rows", wl.mlp_layers(widths, 3), n_props, 0.2, 2, 4)
    onet, props, unst = oracle_setup(pb)
    most = min(max_splits, min(len(u) for u in unst))
    batch = wl.random_batch(pb, unst, 11, most // 2, most, 5)   # 22 rows: a block of four rows half empty
    a, b = wl.random_alpha_beta(batch, 6, 1.0)
    net = bc.load_net(pb.layers, pb.C)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    db = bc.DeviceBatch.from_host(batch)
    n0 = bc.kernel_launches()
    lb, da, dbeta = bc.bound_grad(net, dom, db, _t(a), _t(b), bc.FP32)
    assert bc.kernel_launches() - n0 == 1
    assert bc.status(net) == 0
    ref, da_ref, db_ref = O.grad(onet, props, batch, a.astype(np.float64), b.astype(np.float64))
    assert np.max(rel_err(lb.cpu().numpy(), ref)) <= RTOL
    for g, gr in ((da, da_ref), (dbeta, db_ref)):
        scale = max(np.abs(gr).max(initial=0), 1e-6)
        assert np.max(np.abs(g.cpu().numpy() - gr), initial=0) <= 1e-4 * scale
    assert torch.equal(bc.bound(net, dom, db, _t(a), _t(b), bc.FP32), lb)
    lb_x, x = bc.bound_xstar(net, dom, db, _t(a), _t(b))
    assert torch.equal(lb_x, lb)
    x = x.reshape(batch.B, pb.K, -1).cpu().numpy()
    lo, hi = pb.x_lo[batch.prop_of][:, None], pb.x_hi[batch.prop_of][:, None]
    assert np.all((x == lo) | (x == hi))


def test_rows_and_layers_agree():
    """The subdomains of a batch past the rule's work go layer by layer: the same values up to the order of
    the bound's sum (RTOL), the same corner and gradients up to a sum's rounding."""
    pb = wl.make_problem("rows", wl.mlp_layers([40, 96, 80, 4], 3), 2, 0.1, 2, 4)
    onet, props, unst = oracle_setup(pb)
    net = bc.load_net(pb.layers, pb.C)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    U = np.array([len(u) for u in unst])
    big = wl.random_batch(pb, unst, 9000, 0, 6, 3)
    n = 50
    na, ns = int((U[big.prop_of[:n]] * pb.K).sum()), int(big.split_cnt[:n].sum())
    small = wl.Batch(big.prop_of[:n], big.split_off[:n], big.split_cnt[:n], big.split_layer[:ns], big.split_idx[:ns],
                     big.split_sign[:ns], big.alpha_off[:n], na, ns * pb.K)
    a, b = wl.random_alpha_beta(big, 5, 0.5)
    got = []
    for batch, x, y in ((small, a[:na], b[:ns * pb.K]), (big, a, b)):
        n0 = bc.kernel_launches()
        out = bc.bound_grad(net, dom, bc.DeviceBatch.from_host(batch), _t(x), _t(y), bc.FP32)
        assert (bc.kernel_launches() - n0 == 1) == (batch is small)
        assert bc.status(net) == 0
        got.append([v.cpu().numpy() for v in out])
    for s, l in zip(*got):
        l = l[:s.size]
        assert np.abs(s - l).max() <= RTOL * max(np.abs(l).max(), 1.0)


def test_rows_refuse_what_the_layers_refuse():
    pb = wl.make_problem("rows", wl.mlp_layers([8, 24, 3], 3), 1, 0.3, 2, 4)
    onet, props, unst = oracle_setup(pb)
    batch = wl.random_batch(pb, unst, 4, 2, 2, 5)
    a, b = wl.random_alpha_beta(batch, 6, 1.0)
    net = bc.load_net(pb.layers, pb.C)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    for field, value in (("prop_of", 1), ("split_idx", 24), ("split_sign", 0), ("split_cnt", 65)):
        arrays = {f: getattr(batch, f).copy() for f in ("prop_of", "split_off", "split_cnt", "split_layer", "split_idx",
                                                       "split_sign", "alpha_off")}
        arrays[field][1] = value
        db = bc.DeviceBatch.from_host(wl.Batch(*arrays.values(), batch.n_alpha, batch.n_beta))
        bc.bound(net, dom, db, _t(a), _t(b), bc.FP32)
        assert bc.status(net) != 0
    lb = bc.bound(net, dom, bc.DeviceBatch.from_host(batch), _t(a), _t(b), bc.FP32)
    assert bc.status(net) == 0 and torch.isfinite(lb).all()


@pytest.mark.parametrize("widths,B,bound,grad", [
    ([2048, 512, 4], 4, False, False),    # long chains of one layer
    ([2048, 256, 4], 4, False, True),     # long in the bound, made up for in the gradient
    ([784, 20, 10], 4000, False, False),  # many rows of one layer
    ([784, 20, 10], 1000, True, True),
    ([64] * 9 + [10], 9000, False, False),   # a warp per row, few of them resident
    ([64] * 9 + [10], 4, True, True),
])
def test_which_calls_take_the_one_launch(widths, B, bound, grad):
    """Shapes that the layers' kernels do faster go to them, the bound and the gradient each by its own time."""
    pb = wl.make_problem("rows", wl.mlp_layers(widths, 3), 1, 0.02, 2, 4)
    onet = O.OracleNet(pb.layers, pb.C)
    l, u = (x.astype(np.float32) for x in O.interval_bounds(onet, pb.x_lo, pb.x_hi))
    batch = wl.random_batch(pb, [np.nonzero(O.unstable_mask(l[0], u[0]))[0]], B, 0, 2, 5)
    a, b = (_t(x) for x in wl.random_alpha_beta(batch, 6, 1.0))
    net, dom, db = bc.load_net(pb.layers, pb.C), bc.domain_from_host(pb.x_lo, pb.x_hi, l, u), bc.DeviceBatch.from_host(batch)
    n0 = bc.kernel_launches()
    lb = bc.bound(net, dom, db, a, b, bc.FP32)
    n1 = bc.kernel_launches()
    lb_g, _, _ = bc.bound_grad(net, dom, db, a, b, bc.FP32)
    assert (n1 - n0 == 1, bc.kernel_launches() - n1 == 1) == (bound, grad)
    assert torch.equal(lb, lb_g)
    assert bc.status(net) == 0
