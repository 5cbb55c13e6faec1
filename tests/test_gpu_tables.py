"""The per-property tables of unstable neurons (needs a GB300) at the edges of a thread's 4 neurons and of
a 4096-neuron segment, one and several properties: a neuron's rank is its alpha's place, so the
gradient with respect to alpha against the FP64 oracle shows every one."""
import numpy as np
import pytest
import torch

from oracle import bcrown_oracle as O
from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl
from tests.helpers import RTOL, oracle_setup, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [[3, 1, 2], [4, 3, 2, 3], [6, 127, 130, 2], [5, 4096, 2], [5, 4095, 6, 2],
                                    [4, 8193, 2]])
@pytest.mark.parametrize("n_props", [1, 3])
def test_tables(widths, n_props):
    pb = wl.make_problem("tables", wl.mlp_layers(widths, 3), n_props, 0.2, 2, 4)
    onet, props, unst = oracle_setup(pb)
    batch = wl.random_batch(pb, unst, 4, 0, 3, 5)
    a, b = wl.random_alpha_beta(batch, 6, 1.0)
    net = bc.load_net(pb.layers, pb.C)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    ref, da_ref, _ = O.grad(onet, props, batch, a.astype(np.float64), b.astype(np.float64))
    lb, da, _ = bc.bound_grad(net, dom, bc.DeviceBatch.from_host(batch), torch.from_numpy(a).cuda(),
                              torch.from_numpy(b).cuda(), bc.FP32)
    assert bc.status(net) == 0
    assert np.max(rel_err(lb.cpu().numpy(), ref)) <= RTOL
    scale = max(np.abs(da_ref).max(initial=0), 1e-6)
    assert np.max(np.abs(da.cpu().numpy() - da_ref), initial=0) <= 1e-4 * scale
