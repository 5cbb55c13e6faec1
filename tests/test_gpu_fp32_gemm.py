"""The FP32 GEMM of the CUDA-core path at the edges of its tiles (needs a GB300): fully connected nets
whose widths and row counts leave remainders of the 32 x 64 and 64 x 128 tiles and of the K step of 32,
aligned rows (widths a multiple of 4: 16-byte copies) and unaligned ones, and row counts on both sides
of the rule that chooses the tile.  Bounds and gradients against the FP64 oracle at the FP32 bar."""
import numpy as np
import pytest
import torch

from oracle import bcrown_oracle as O
from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl
from tests.helpers import RTOL, oracle_setup, rel_err, repack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,B", [
    ([7, 33, 31, 3], 1),            # less than one tile each way, odd rows
    ([33, 65, 63, 5], 11),          # one past and one short of a tile, unaligned
    ([32, 64, 128, 4], 32),         # whole tiles
    ([36, 68, 132, 4], 43),         # aligned remainders of 4
    ([8, 129, 4, 3], 7600),         # 15,200 rows: 476 large tiles of a 129-wide layer, small ones elsewhere
    ([12, 128, 64, 3], 7681),       # 15,362 rows: 241 large tiles for every layer
])
def test_gemm_tiles(widths, B):
    pb = wl.make_problem("gemm", wl.mlp_layers(widths, 5), 1, 0.08, 2, 5)
    onet, props, unst = oracle_setup(pb)
    batch = wl.random_batch(pb, unst, B, 0, 3, 9)
    a, b = wl.random_alpha_beta(batch, 4, 0.5)
    net = bc.load_net(pb.layers, pb.C)
    dom = bc.domain_from_host(props["x_lo"], props["x_hi"], props["l"], props["u"])
    db = bc.DeviceBatch.from_host(batch)
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    lb, da, dbeta = (x.cpu().numpy() for x in bc.bound_grad(net, dom, db, ta, tb, bc.FP32))
    assert bc.status(net) == 0
    assert np.array_equal(bc.bound(net, dom, db, ta, tb).cpu().numpy(), lb)
    # the oracle on a sample of subdomains, the first and the last among them
    idx = np.unique(np.concatenate([[0, B - 1], np.linspace(0, B - 1, min(B, 40)).astype(int)]))
    U = [len(u) for u in unst]
    sb, sa, sbeta = repack(pb, batch, U, idx, a, b)
    ref, ra, rb = O.grad(onet, props, sb, sa.astype(np.float64), sbeta.astype(np.float64))
    rows = (idx[:, None] * pb.K + np.arange(pb.K)).reshape(-1)
    assert rel_err(lb[rows], np.asarray(ref).reshape(-1)).max() <= RTOL
    got_a = np.concatenate([da[batch.alpha_off[i]:batch.alpha_off[i] + U[0] * pb.K] for i in idx])
    got_b = np.concatenate([dbeta[batch.split_off[i] * pb.K:(batch.split_off[i] + batch.split_cnt[i]) * pb.K]
                            for i in idx])
    for got, want in ((got_a, ra), (got_b, rb)):
        want = np.asarray(want).reshape(-1)
        if want.size:   # entry by entry within 1e-3 of |g| + 1e-3 max |g|, as the gradient tests hold it
            assert (np.abs(got - want) <= 1e-3 * (np.abs(want) + 1e-3 * np.abs(want).max())).all()


@pytest.mark.parametrize("widths", [[7, 33, 31, 3], [33, 65, 63, 5], [32, 64, 128, 4], [36, 68, 132, 4], [8, 129, 4, 3]])
@pytest.mark.parametrize("n", [1, 31, 33, 192])
def test_gemm_tiles_forward(widths, n):
    """The plain forward pass takes the GEMM at every size (bounds of small networks do not)."""
    pb = wl.make_problem("gemm", wl.mlp_layers(widths, 5), 1, 0.08, 2, 5)
    net = bc.load_net(pb.layers, pb.C)
    x = np.random.default_rng(n).uniform(0, 1, (n, widths[0])).astype(np.float32)
    ref = O.OracleNet(pb.layers, pb.C).forward(x)
    got = bc.forward(net, torch.from_numpy(x).cuda()).cpu().numpy()
    assert got.shape == ref.shape and np.max(rel_err(got, ref)) <= RTOL
