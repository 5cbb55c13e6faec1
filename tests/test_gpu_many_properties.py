"""The BF16 layer path over so many properties that their hidden neurons pass 2^31 (needs a GB300 with 100 GB
free): a subdomain of the last property is bounded as in a domain that holds its property alone."""
import numpy as np
import pytest
import torch

from oracle import bcrown_oracle as O
from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl
from tests.helpers import oracle_setup

pytestmark = pytest.mark.gpu


def test_neuron_tables_past_31_bits():
    if torch.cuda.mem_get_info()[0] < 100 << 30:
        pytest.skip("needs 100 GB of device memory")
    pb = wl.make_problem("many", wl.conv_layers((4, 8, 8), [(16, 3, 1, 1)], [24, 4], 3), 1, 0.1, 3, 4)
    onet, props, unst = oracle_setup(pb)
    H = props["l"].shape[1]
    P = 2 ** 31 // H + 2   # the last property's neurons begin past 2^31
    batch = wl.random_batch(pb, unst, 16, 0, 4, 5)
    a, b = wl.random_alpha_beta(batch, 6, 1.0)
    ref = O.bound(onet, props, batch, a, b)
    at, bt = (torch.as_tensor(np.ascontiguousarray(x, np.float32)).cuda() for x in (a, b))
    net = bc.load_net(pb.layers, pb.C)
    bc.set_launch(net, bc.N.PATH_LAYER_EPI)
    one = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    want = bc.bound_grad(net, one, bc.DeviceBatch.from_host(batch), at, bt, bc.BF16)
    many = bc.Domain(*(v.repeat(P, 1) for v in (one.x_lo, one.x_hi, one.l, one.u)))
    many.l[:-1] = 1.0   # (every other property all active)
    many.u[:-1] = 2.0
    batch.prop_of[:] = P - 1
    got = bc.bound_grad(net, many, bc.DeviceBatch.from_host(batch), at, bt, bc.BF16)
    assert bc.status(net) == 0
    for g, w in zip(got, want):
        assert torch.equal(g, w)
    assert np.abs(got[0].cpu().numpy() - ref).max() <= 3e-2 * max(np.median(np.abs(ref)), 1.0)
    del net, many
    torch.cuda.empty_cache()
