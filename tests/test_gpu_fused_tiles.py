"""The fused kernel's row tiles (needs a GB300): a batch takes tiles of 16, 32 or 64 rows by its size,
and a row's bound and gradient are one column of every contraction, so the subdomains of a batch get
the same values bit for bit whatever batch they are part of.  Widths leave odd K blocks (the last pair
of a layer half empty), partial chunks and a box that needs one, several and all eight input chunks;
the bound is checked against the oracle's at the 784 net's BF16 tolerance."""
import numpy as np
import pytest
import torch

from oracle import bcrown_oracle as O
from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl
from tests.helpers import oracle_setup

pytestmark = pytest.mark.gpu

# rows per tile 16 (up to 152 tiles), 32, 64 on a 152-SM GPU
SMALL, MIDDLE, LARGE = 40, 1100, 2600


@pytest.mark.parametrize("widths,n_props", [
    ([70, 200, 130, 60, 5], 1),
    ([300, 100, 256, 40, 4], 3),        # 5 input blocks; a 100-wide layer ends inside a block
    ([1024, 256, 256, 3], 1),           # the widest box: 8 input chunks
    ([9, 33, 4], 2),                    # one hidden layer, one block everywhere
])
def test_rows_do_not_depend_on_the_tile(widths, n_props):
    pb = wl.make_problem("tiles", wl.mlp_layers(widths, 4), n_props, 0.02, 2, 4)
    onet, props, unst = oracle_setup(pb)
    batch = wl.random_batch(pb, unst, LARGE, 0, 6, 3)
    a, b = wl.random_alpha_beta(batch, 5, 0.5)
    net = bc.load_net(pb.layers, pb.C)
    assert bc.path_supported(net, 1)   # the fused kernel
    bc.set_launch(net, 1)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    U = np.array([len(u) for u in unst])
    got = {}
    for n in (SMALL, MIDDLE, LARGE):
        na = int((U[batch.prop_of[:n]] * pb.K).sum())
        ns = int(batch.split_cnt[:n].sum())
        part = wl.Batch(batch.prop_of[:n], batch.split_off[:n], batch.split_cnt[:n], batch.split_layer[:ns],
                        batch.split_idx[:ns], batch.split_sign[:ns], batch.alpha_off[:n], na, ns * pb.K)
        db = bc.DeviceBatch.from_host(part)
        ta, tb = torch.from_numpy(a[:na]).cuda(), torch.from_numpy(b[:ns * pb.K]).cuda()
        out = bc.bound_grad(net, dom, db, ta, tb, bc.BF16)
        assert bc.status(net) == 0
        assert torch.equal(bc.bound(net, dom, db, ta, tb, bc.BF16), out[0])
        got[n] = [x.cpu() for x in out]
    for n in (MIDDLE, LARGE):
        for small, large in zip(got[SMALL], got[n]):
            assert torch.equal(small, large[:small.numel()])
    n = SMALL
    ns = int(batch.split_cnt[:n].sum())
    part = wl.Batch(batch.prop_of[:n], batch.split_off[:n], batch.split_cnt[:n], batch.split_layer[:ns],
                    batch.split_idx[:ns], batch.split_sign[:ns], batch.alpha_off[:n],
                    int((U[batch.prop_of[:n]] * pb.K).sum()), ns * pb.K)
    ref = O.bound(onet, props, part, a[:part.n_alpha].astype(np.float64), b[:part.n_beta].astype(np.float64))
    # BF16 operands move a bound by a few units of 2^-9 of the magnitudes it sums
    scale = np.maximum(np.abs(ref).max(), 1.0)
    assert np.abs(got[n][0].numpy() - ref).max() <= 2e-2 * scale


@pytest.mark.parametrize("B", [5, 700])   # one tile and several
def test_one_property_needs_no_plan_and_still_refuses_another(B):
    """With one property the rows stand in the batch's order; a subdomain that names another property is
    reported and leaves the others' values as they are."""
    pb = wl.make_problem("single", wl.mlp_layers([30, 96, 64, 3], 4), 1, 0.05, 2, 4)
    onet, props, unst = oracle_setup(pb)
    batch = wl.random_batch(pb, unst, B, 0, 6, 3)
    a, b = wl.random_alpha_beta(batch, 5, 0.5)
    net = bc.load_net(pb.layers, pb.C)
    assert bc.path_supported(net, 1)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    lb = bc.bound(net, dom, bc.DeviceBatch.from_host(batch), ta, tb, bc.BF16).reshape(B, -1)
    assert bc.status(net) == 0
    prop_of = batch.prop_of.copy()
    prop_of[B // 2] = 1
    bad = wl.Batch(prop_of, batch.split_off, batch.split_cnt, batch.split_layer, batch.split_idx, batch.split_sign,
                   batch.alpha_off, batch.n_alpha, batch.n_beta)
    got = bc.bound(net, dom, bc.DeviceBatch.from_host(bad), ta, tb, bc.BF16).reshape(B, -1)
    assert bc.status(net) != 0
    keep = torch.arange(B) != B // 2
    assert torch.equal(got[keep.cuda()], lb[keep.cuda()])
