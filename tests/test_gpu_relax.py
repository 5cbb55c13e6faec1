"""The FP32 path's relaxation passes and optimiser step at the edges of their forms (needs a GB300):
layers that are and are not a multiple of four neurons, one warp and a block per row, properties
whose first neuron is off a 16-byte boundary, split lists from none to the longest."""
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


@pytest.mark.parametrize("widths,n_props", [
    ([6, 4, 8, 3], 2),            # one group of four, two groups
    ([6, 132, 2048, 3], 1),       # a remainder of the warp's 128; the widest row of one warp
    ([6, 2052, 16, 3], 1),        # a block per row, one group past two rounds
    ([6, 2052, 6, 3], 2),         # 2,058 neurons: the second property starts off a boundary
    ([6, 2051, 30, 3], 1),        # no multiple of four
])
@pytest.mark.parametrize("max_splits", [0, 3, 60])
def test_relaxation(widths, n_props, max_splits):
    pb = wl.make_problem("relax", wl.mlp_layers(widths, 3), n_props, 0.3, 2, 4)
    onet, props, unst = oracle_setup(pb)
    most = min(max_splits, min(len(u) for u in unst))
    batch = wl.random_batch(pb, unst, 7, most, most, 5)
    a, b = wl.random_alpha_beta(batch, 6, 1.0)
    net = bc.load_net(pb.layers, pb.C)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    db = bc.DeviceBatch.from_host(batch)
    ref = O.bound(onet, props, batch, a.astype(np.float64), b.astype(np.float64)).reshape(-1)
    lb = bc.bound(net, dom, db, _t(a), _t(b), bc.FP32).cpu().numpy()
    assert np.max(rel_err(lb, ref)) <= RTOL
    certified = bc.bound(net, dom, db, _t(a), _t(b), bc.CERTIFY).cpu().numpy()
    assert bc.status(net) == 0
    assert np.all(certified <= ref + 1e-12 * np.abs(ref))
    # gamma of the widest sum (2,052 terms, 2^-24 each) times the sums of magnitudes of each layer, which
    # are up to a few hundred times the bound
    assert np.abs(certified - ref).max() <= 0.1 * max(np.abs(ref).max(), 1.0)


def test_adam_of_a_block_and_of_a_warp_per_row_agree():
    """A batch whose rows have 2,048 alphas or more on average takes a block per row; the same subdomains
    next to many without an alpha take a warp: the same values bit for bit."""
    pb = wl.make_problem("wide", wl.mlp_layers([6, 3000, 3], 3), 2, 0.5, 2, 4)
    onet, props, unst = oracle_setup(pb)
    l, u = props["l"].copy(), props["u"].copy()
    l[0], u[0] = -np.abs(l[0]) - 0.1, np.abs(u[0]) + 0.1       # every neuron unstable
    l[1], u[1] = np.abs(l[1]) + 0.1, np.abs(u[1]) + 0.2 + np.abs(l[1])   # none
    U = np.array([pb.hidden_widths[0], 0])
    rng = np.random.default_rng(3)
    subs = []
    for n in (0, 3, 17):
        g = np.sort(rng.choice(pb.hidden_widths[0], n, replace=False)).astype(np.int64)
        subs.append((0, g, rng.choice([-1, 1], n).astype(np.int8)))
    none = (1, np.zeros(0, np.int64), np.zeros(0, np.int8))
    net = bc.load_net(pb.layers, pb.C)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], l, u)
    got = []
    for extra in (0, 9):
        batch = wl.pack_batch(pb.hidden_widths, pb.K, U, subs + [none] * extra)
        assert (batch.n_alpha >= 2048 * batch.B * pb.K) == (extra == 0)
        alpha, beta = torch.full((batch.n_alpha,), 0.4).cuda(), torch.full((batch.n_beta,), 0.1).cuda()
        lb = bc.optimize(net, dom, bc.DeviceBatch.from_host(batch), alpha, beta,
                         bc.OptCfg(iters=3, precision=bc.FP32, certify=False))
        assert bc.status(net) == 0
        got.append((lb[:3 * pb.K].cpu(), alpha.cpu(), beta.cpu()))
    for x, y in zip(*got):
        assert torch.equal(x, y)
    assert not torch.equal(got[0][1], torch.full_like(got[0][1], 0.4))
