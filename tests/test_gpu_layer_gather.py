"""The fused-epilogue BF16 layer path where its operand is gathered and a tile is wider than 128 columns
(needs a GB300): 129, 160, 192 and 256 channels, forward and backward, on maps that are no box of 128
positions and from channels that are neither 8 nor a multiple of 64, with several tiles and rounds of the
ring per SM, a ragged last tile, and few or most neurons unstable."""
import numpy as np
import pytest
import torch

from oracle import bcrown_oracle as O
from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl
from tests.helpers import grad_agreement, grad_groups, repack
from tests.test_gpu_tc import GRAD_COS, GRAD_SHARE, GRAD_TOL

pytestmark = pytest.mark.gpu

NETS = {
    "129": ((16, 10, 10), [(129, 3, 1, 1), (24, 3, 1, 1)]),
    "160": ((16, 14, 14), [(160, 3, 1, 1), (32, 3, 2, 1)]),
    "192": ((64, 14, 14), [(192, 3, 2, 1), (24, 3, 1, 1)]),
    "256": ((24, 13, 13), [(256, 3, 2, 1), (40, 2, 1, 0)]),     # 7 x 7, 6 x 6: three stages
}


def _t(x):
    return torch.as_tensor(np.ascontiguousarray(x, np.float32)).cuda()


def _tolerance(onet, props, batch, a, b):
    """Per row, 8 standard deviations of what rounding the contractions' operands to BF16 does to the bound
    to first order, the roundings taken as independent: an operand is off by up to 2^-9 of itself, 0.6 times
    that in the root mean square, and dlb/dA is the primal path's h.  (Emulated in 64 bits with rounded
    operands, the cases here are off by at most half of it.)"""
    _, tr = O.bound(onet, props, batch, a, b, trace=True)
    rows = O.expand_rows(onet, batch, props["l"], props["u"])
    lo, hi = (np.asarray(props[k], np.float64)[rows.prop] for k in ("x_lo", "x_hi"))
    h = np.where(tr.A[0] >= 0, lo, hi)
    var = 0.0
    for i in range(1, onet.L):
        W = onet.W[i]
        zw = O._mv(W, h)
        var = var + (tr.Lam[i] ** 2 * zw ** 2).sum(1)                            # Lambda's rounding
        var = var + (O._mm(tr.Lam[i] ** 2, W.multiply(W)) * h ** 2).sum(1)       # the weights'
        h = tr.D[i] * (zw + onet.b[i]) + tr.lam[i]
    return 8 * 0.6 * 2.0 ** -9 * np.sqrt(var)


@pytest.mark.parametrize("which", list(NETS))
@pytest.mark.parametrize("eps", [0.004, 0.1])
def test_gathered_wide_tiles_match_oracle(which, eps):
    shape, convs = NETS[which]
    layers = wl.conv_layers(shape, convs, [4], 7)
    pb = wl.make_problem("gather_" + which, layers, 2, eps, 3, 8)
    onet = O.OracleNet(pb.layers, pb.C)
    l, u = (x.astype(np.float32) for x in O.interval_bounds(onet, pb.x_lo, pb.x_hi))
    unst = [np.nonzero(O.unstable_mask(l[p], u[p]))[0] for p in range(pb.P)]
    props = dict(x_lo=pb.x_lo, x_hi=pb.x_hi, l=l, u=u)
    share = np.mean([len(x) for x in unst]) / l.shape[1]
    batch = wl.random_batch(pb, unst, 211, 0, 8, 9, props=np.arange(211) % 2)   # 633 rows
    a, b = wl.random_alpha_beta(batch, 3, 1.0)
    net = bc.load_net(pb.layers, pb.C)
    dom = bc.domain_from_host(pb.x_lo, pb.x_hi, l, u)
    bc.set_launch(net, bc.N.PATH_LAYER_EPI)
    db, at, bt = bc.DeviceBatch.from_host(batch), _t(a), _t(b)
    lb, da, dbeta = bc.bound_grad(net, dom, db, at, bt, bc.BF16)
    assert bc.status(net) == 0
    again = bc.bound(net, dom, db, at, bt, bc.BF16)
    assert torch.equal(lb, again)
    idx = np.array([0, 1, 57, 104, 150, 209, 210])
    U = [len(x) for x in unst]
    sb, sa, sbeta = repack(pb, batch, U, idx, a, b)
    ref, da_ref, db_ref = O.grad(onet, props, sb, sa.astype(np.float64), sbeta.astype(np.float64))
    tol = _tolerance(onet, props, sb, sa.astype(np.float64), sbeta.astype(np.float64))
    err = np.abs(lb.cpu().numpy().reshape(batch.B, pb.K)[idx].reshape(-1) - ref)
    print("%s eps %g: %.0f %% unstable, max err / tolerance %.3f, tolerance / |bound| %.1e"
          % (which, eps, 100 * share, (err / tol).max(), (tol / np.abs(ref)).max()))
    assert np.all(err <= tol)
    _, ga, gb = repack(pb, batch, U, idx, da.cpu().numpy(), dbeta.cpu().numpy())
    la, lbeta = grad_groups(onet, sb, props)
    for g, gr, lay in ((ga, da_ref, la), (gb, db_ref, lbeta)):
        for i, (part, cos, n) in grad_agreement(g, gr, lay, GRAD_TOL).items():
            print("layer %d: %d entries, share within tolerance %.4f, cosine %.6f" % (i, n, part, cos))
            if n >= 20:
                assert cos >= GRAD_COS and (n < 100 or part >= GRAD_SHARE), (i, part, cos)
