"""The work this library is used for, as cases that can be timed and compared.

A case names an entry point of `paper_2103_06624_gb300.bcrown`, a network, a number of subdomains
B (and properties P) and the options of the call.  Networks, boxes, split lists, slopes and
multipliers are drawn from the seed; the root bounds l, u that a caller holds are CROWN bounds
(Lemma 2.2, adaptive slopes) computed here with torch.  The arrays of a case have one size for
every seed: the neurons nearest to stability are moved across it until each layer's usual
number is unstable, and the split lists' lengths and the properties' shares depend on the case alone.

The networks and their boxes are the repository's own: the 16-32-32-4 and 784-256x6-10 MLPs, the
two CIFAR-shaped convolutional networks, and (drawn cases) a 37-300-260-5 MLP, which the fused
tensor-core kernel does not take, and a small strided convolutional network.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2103_06624_gb300 import bcrown as bc
from paper_2103_06624_gb300 import workloads as wl

# in_shape, convolutions (channels, kernel, stride, padding), widths after flattening, half-width
# of the box, specifications, depth of the split lists, unstable neurons per hidden layer
NETS = {
    "mlp16": dict(shape=(16, 1, 1), convs=[], fcs=[32, 32, 4], eps=0.05, K=3, depth=4, unstable=(8, 12)),
    "mlp37": dict(shape=(37, 1, 1), convs=[], fcs=[300, 260, 5], eps=0.03, K=4, depth=10, unstable=(60, 90)),
    "mlp784": dict(shape=(784, 1, 1), convs=[], fcs=[256] * 6 + [10], eps=0.015, K=9, depth=12, unstable=(110, 194, 256, 256, 256, 256)),
    "conv_tiny": dict(shape=(2, 6, 6), convs=[(3, 3, 2, 1), (4, 3, 1, 1)], fcs=[8, 4], eps=0.05, K=3, depth=4,
                      unstable=(5, 14, 3)),
    "conv_small": dict(shape=(3, 32, 32), convs=[(32, 4, 2, 1), (64, 4, 2, 1)], fcs=[512, 512, 10], eps=2 / 255, K=9,
                       depth=16, unstable=(484, 534, 302, 500)),
    "conv_big": dict(shape=(3, 32, 32), convs=[(64, 3, 1, 1), (64, 3, 2, 1), (128, 3, 1, 1), (128, 3, 2, 1)],
                     fcs=[512, 10], eps=2 / 255, K=9, depth=24, unstable=(3000, 1300, 5000, 2800, 511)),
}


def listed():
    return [
        # the smallest call: one bound and gradient of a small property's first subdomains, FP32
        dict(name="grad_fp32_mlp16_b64", kind="grad", net="mlp16", B=64, P=1, precision="fp32"),
        # the first rounds of a branch and bound on the MLP: few subdomains, latency
        dict(name="grad_bf16_mlp784_b16", kind="grad", net="mlp784", B=16, P=1, precision="bf16"),
        # one optimiser iteration's bound and gradient at the paper's batch size
        dict(name="grad_bf16_mlp784_b1024", kind="grad", net="mlp784", B=1024, P=1, precision="bf16"),
        # a pool shared by 64 properties, uneven shares, every property's last tile ragged
        dict(name="grad_bf16_mlp784_p64_b11173", kind="grad", net="mlp784", B=11173, P=64, precision="bf16"),
        # the whole call a verifier makes per batch: 20 Adam iterations, then the certified bound
        dict(name="optimize_mlp784_b1024", kind="optimize", net="mlp784", B=1024, P=1, iters=20, warm=False),
        # the upper bound of Algorithm 1: FP32 bounds with their minimisers x*, and the network there
        dict(name="xstar_mlp784_b512", kind="xstar", net="mlp784", B=512, P=1),
        # bound and gradient on the convolutional networks: an odd batch of the small one, the
        # paper's batch size on the big one (the largest case)
        dict(name="grad_bf16_conv_small_b509", kind="grad", net="conv_small", B=509, P=1, precision="bf16"),
        dict(name="grad_bf16_conv_big_b1024", kind="grad", net="conv_big", B=1024, P=1, precision="bf16"),
        # an ascent continued from a kept optimiser state (children of a batch keep stepping), certified
        dict(name="optimize_conv_big_b64", kind="optimize", net="conv_big", B=64, P=1, iters=4, warm=True),
        # certified bounds of finished subdomains (outward rounding), an odd batch
        dict(name="certify_conv_small_b333", kind="bound", net="conv_small", B=333, P=1, precision="certify"),
        # what every property pays before branching: its certified root bounds
        dict(name="root_conv_small", kind="root", net="conv_small", B=1, P=1, precision="certify"),
        # joint optimisation of the intermediate bounds (Section 3.3): bound and all four gradients
        dict(name="joint_grad_mlp784_b16", kind="joint", net="mlp784", B=16, P=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grad", "grad", "grad", "grad", "bound", "bound", "optimize", "optimize", "xstar", "root",
                       "joint", "split"])
    if kind == "grad":
        precision = rng.choice(["bf16", "bf16", "bf16", "fp32"])
        net = rng.choice(["mlp784", "mlp784", "conv_small", "conv_big", "mlp37", "conv_tiny", "mlp16"])
        hi = {"mlp784": 11173, "conv_small": 1024, "conv_big": 1024, "mlp37": 4096, "conv_tiny": 4096, "mlp16": 4096}
        if precision == "fp32":
            hi.update(mlp784=2048, conv_small=256, conv_big=48)
        B = _log_int(rng, 1, hi[net])
        P = min(B, _log_int(rng, 1, 64)) if net.startswith("mlp") and rng.random() < 0.5 else 1
        return dict(kind=kind, net=net, B=B, P=P, precision=precision)
    if kind == "bound":
        precision = rng.choice(["certify", "certify", "fp32", "bf16"])
        net = rng.choice(["mlp784", "mlp784", "conv_small", "conv_big", "mlp37", "conv_tiny"])
        hi = {"mlp784": 4096, "conv_small": 512, "conv_big": 96, "mlp37": 4096, "conv_tiny": 4096}
        return dict(kind=kind, net=net, B=_log_int(rng, 1, hi[net]), P=1, precision=precision)
    if kind == "optimize":
        net = rng.choice(["mlp784", "mlp784", "conv_small", "conv_big"])
        if net == "mlp784":
            return dict(kind=kind, net=net, B=_log_int(rng, 4, 1024), P=1, iters=20, warm=False)
        hi = {"conv_small": 200, "conv_big": 64}[net]
        return dict(kind=kind, net=net, B=_log_int(rng, 2, hi), P=1, iters=rng.randint(2, 4), warm=True)
    if kind == "xstar":
        net = rng.choice(["mlp784", "mlp784", "conv_small", "mlp37"])
        return dict(kind=kind, net=net, B=_log_int(rng, 1, 1500 if net != "conv_small" else 200), P=1)
    if kind == "root":
        net = rng.choice(["mlp784", "mlp784", "conv_small", "mlp37", "mlp16"])
        P = 1 if net == "conv_small" else _log_int(rng, 1, 12)
        return dict(kind=kind, net=net, B=1, P=P, precision=rng.choice(["certify", "certify", "fp32"]))
    if kind == "joint":
        net = rng.choice(["mlp784", "mlp16"])
        return dict(kind=kind, net=net, B=_log_int(rng, 1, 24 if net == "mlp784" else 512), P=1)
    net = rng.choice(["mlp784", "conv_small"])
    return dict(kind="split", net=net, B=_log_int(rng, 1, 1024), P=1)


# --------------------------------------------------------------------------------------------
# Networks and root bounds (torch)
# --------------------------------------------------------------------------------------------

class _Layer:
    """One linear layer on the GPU: its weights and the two directions of its contraction."""

    def __init__(self, kind, W, b, in_shape, out_shape, stride=1, pad=0):
        self.kind, self.W, self.b = kind, W, b
        self.in_shape, self.out_shape, self.stride, self.pad = in_shape, out_shape, stride, pad
        self.d_in, self.d_out = math.prod(in_shape), math.prod(out_shape)

    def to(self, dtype):
        return _Layer(self.kind, self.W.to(dtype), self.b.to(dtype), self.in_shape, self.out_shape, self.stride, self.pad)

    def bias(self):
        """The bias of every output neuron."""
        return self.b if self.kind == "fc" else self.b.repeat_interleave(self.out_shape[1] * self.out_shape[2])

    def macs(self):
        return self.W.numel() * (self.out_shape[1] * self.out_shape[2] if self.kind == "conv" else 1)

    def fwd(self, x, W=None):
        W = self.W if W is None else W
        if self.kind == "fc":
            return x @ W.T
        return F.conv2d(x.reshape((-1,) + self.in_shape), W, stride=self.stride, padding=self.pad).reshape(len(x), -1)

    def bwd(self, A):
        if self.kind == "fc":
            return A @ self.W
        k, s = self.W.shape[-1], self.stride
        left = [self.in_shape[i + 1] - ((self.out_shape[i + 1] - 1) * s - 2 * self.pad + k) for i in (0, 1)]
        return F.conv_transpose2d(A.reshape((-1,) + self.out_shape), self.W, stride=s, padding=self.pad,
                                  output_padding=left).reshape(len(A), -1)


def _conv_exactly():
    return torch.backends.cudnn.flags(enabled=True, benchmark=False, deterministic=True, allow_tf32=False)


def _geometry(name):
    """(kind, weight shape, in_shape, out_shape, stride, pad) of each layer."""
    spec, out = NETS[name], []
    shape = spec["shape"]
    for co, k, s, p in spec["convs"]:
        o = (co, (shape[1] + 2 * p - k) // s + 1, (shape[2] + 2 * p - k) // s + 1)
        out.append(("conv", (co, shape[0], k, k), shape, o, s, p))
        shape = o
    for w in spec["fcs"]:
        out.append(("fc", (w, math.prod(shape)), shape, (w, 1, 1), 1, 0))
        shape = (w, 1, 1)
    return out


def _layers(name, seed):
    """He-normal weights, biases N(0, 0.01), as the repository's generators draw them."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    made = []
    for kind, ws, i, o, s, p in _geometry(name):
        fan = math.prod(ws[1:])
        W = torch.randn(ws, device="cuda", generator=g) * math.sqrt(2.0 / fan)
        b = torch.randn(ws[0], device="cuda", generator=g) * 0.1
        made.append(_Layer(kind, W, b, i, o, s, p))
    return made


def _chords(l, u):
    """Masks (active, unstable) and the upper chord of every neuron."""
    act, uns = l >= 0, (l < 0) & (u > 0)
    s = torch.where(uns, u / torch.where(uns, u - l, torch.ones_like(u)), torch.zeros_like(u))
    return act, uns, s, torch.where(uns, -s * l, torch.zeros_like(l))


def _root_bounds(layers, x_lo, x_hi, rows_at_once=1 << 27):
    """CROWN bounds [P, H] of the hidden neurons in the layers' precision (adaptive lower slopes)."""
    P, dt = len(x_lo), layers[0].W.dtype
    mid, rad = (x_hi + x_lo) / 2, (x_hi - x_lo) / 2
    first = layers[0]
    z = first.fwd(mid) + first.bias()
    r = first.fwd(rad, first.W.abs())
    ls, us = [z - r], [z + r]
    for T in range(1, len(layers) - 1):
        top, d = layers[T], layers[T].d_out
        lo, hi = torch.empty((P, d), device="cuda", dtype=dt), torch.empty((P, d), device="cuda", dtype=dt)
        widest = max(max(ly.d_in, ly.d_out) for ly in layers[:T + 1])
        step = max(1, min(d, rows_at_once // (widest * P)))
        bias = top.bias()
        for j0 in range(0, d, step):
            n = min(step, d - j0)
            E = torch.zeros((n, d), device="cuda", dtype=dt)
            E[torch.arange(n), torch.arange(j0, j0 + n)] = 1
            for sign, out in ((1.0, lo), (-1.0, hi)):
                A = (sign * top.bwd(E)).expand(P, n, -1)
                c = (sign * bias[j0:j0 + n]).expand(P, n)
                for m in range(T - 1, -1, -1):
                    act, uns, s, t = (v[:, None] for v in _chords(ls[m], us[m]))
                    up = torch.where(uns & (us[m] >= -ls[m])[:, None], torch.ones_like(s), torch.zeros_like(s))
                    pos = A >= 0
                    L = A * torch.where(act, torch.ones_like(s), torch.where(pos, up, s))
                    c = c + (L * layers[m].bias()).sum(-1) + torch.where(pos, torch.zeros_like(A), A * t).sum(-1)
                    A = layers[m].bwd(L.reshape(P * n, -1)).reshape(P, n, -1)
                c = c + (A * mid[:, None]).sum(-1) - (A.abs() * rad[:, None]).sum(-1)
                out[:, j0:j0 + n] = sign * c
        ls.append(lo)
        us.append(hi)
    return ls, us


def _usual_unstable(name, ls, us):
    """l, u [P, H] with the network's number of unstable neurons per layer (a few fewer in the first
    layer of some properties): the stable ones nearest to instability get a small negative l or
    positive u, the unstable ones nearest to stability a zero."""
    for m, want in enumerate(NETS[name]["unstable"]):
        l, u = ls[m], us[m]
        score = torch.minimum(u, -l)   # > 0: unstable
        for p in range(len(l)):
            order = torch.argsort(score[p], descending=True, stable=True)
            n = want - (p % 8) * (want // 20) if m == 0 else want
            more, less = order[:n], order[n:]
            more, less = more[score[p, more] <= 0], less[score[p, less] > 0]
            gap = 1e-3 * (u[p] - l[p]) + 1e-6
            act = l[p, more] >= 0
            l[p, more[act]], u[p, more[~act]] = -gap[more[act]], gap[more[~act]]
            act = u[p, less] >= -l[p, less]
            l[p, less[act]], u[p, less[~act]] = 0.0, 0.0
    return torch.cat(ls, 1), torch.cat(us, 1)


def _problem(case, seed):
    """Layers, merged specification matrix, boxes and root bounds of a case (all on the GPU)."""
    spec = NETS[case["net"]]
    layers = _layers(case["net"], seed)
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    x0 = torch.rand((case["P"], layers[0].d_in), device="cuda", generator=g)
    x_lo, x_hi = x0 - spec["eps"], x0 + spec["eps"]
    C = torch.zeros((spec["K"], layers[-1].d_out), device="cuda")
    C[:, 0] = 1
    C[torch.arange(spec["K"]), torch.arange(1, spec["K"] + 1)] = -1
    with _conv_exactly():
        ls, us = _root_bounds(layers, x_lo, x_hi) if case["kind"] != "root" else (None, None)
    return layers, C, x_lo, x_hi, ls, us


def _splits(case, seed, widths, l, u):
    """Subdomains in the C-ABI layout: properties in uneven shares and mixed order, each subdomain
    with 1 .. depth distinct unstable neurons of its property split either way."""
    rng, fixed = np.random.default_rng(seed + 2), np.random.default_rng(case["B"] * 64 + case["P"])
    B, P, K, depth = case["B"], case["P"], NETS[case["net"]]["K"], NETS[case["net"]]["depth"]
    unst = [np.flatnonzero(m) for m in ((l < 0) & (u > 0)).cpu().numpy()]
    U = np.array([len(x) for x in unst], np.int64)
    w = np.exp(fixed.uniform(0, math.log(64), P))
    share = np.floor(np.cumsum(w) / w.sum() * B).astype(np.int64)
    prop = rng.permutation(np.searchsorted(share, np.arange(B), side="right").clip(0, P - 1))
    cnt = rng.permutation(np.arange(B) % depth + 1)
    pick = np.floor(rng.random((B, depth)) * U[prop][:, None]).astype(np.int64)
    while True:   # draw again where a subdomain would split one neuron twice
        order = np.argsort(pick, axis=1, kind="stable")
        srt = np.take_along_axis(pick, order, 1)
        dup = np.zeros_like(pick, bool)
        np.put_along_axis(dup[:, :], order[:, 1:], srt[:, 1:] == srt[:, :-1], 1)
        dup &= np.arange(depth)[None] < cnt[:, None]
        if not dup.any():
            break
        again = np.floor(rng.random((B, depth)) * U[prop][:, None]).astype(np.int64)
        pick = np.where(dup, again, pick)
    used = np.arange(depth)[None] < cnt[:, None]
    offs = np.concatenate([[0], np.cumsum(U)[:-1]])
    flat = np.concatenate(unst) if U.sum() else np.zeros(0, np.int64)
    g = flat[(offs[prop][:, None] + pick)[used]]
    edge = np.concatenate([[0], np.cumsum(widths)])
    layer = np.searchsorted(edge, g, side="right")
    sign = rng.choice(np.array([-1, 1], np.int8), len(g))
    per = U[prop] * K
    aoff = np.concatenate([[0], np.cumsum(per)[:-1]]).astype(np.int64)
    off = np.concatenate([[0], np.cumsum(cnt)[:-1]]).astype(np.int32)
    hb = wl.Batch(prop.astype(np.int32), off, cnt.astype(np.int32), layer.astype(np.uint8),
                  (g - edge[layer - 1]).astype(np.uint32), sign, aoff, int(per.sum()), int(cnt.sum()) * K)
    return hb, U


def _slopes(n, g):
    """Slopes in [0, 1], a tenth of them at either end, as the projection leaves them."""
    return (torch.rand(n, device="cuda", generator=g) * 1.25 - 0.125).clamp_(0, 1)


def _multipliers(n, g):
    return (torch.randn(n, device="cuda", generator=g) * 0.2).clamp_(min=0)


def _opt_cfg(case):
    return bc.OptCfg(iters=case["iters"], precision=bc.BF16, certify=True)


def _state_of(case, hb, K, g):
    """Optimiser state after 7 iterations: the iterate, moments of matching size, no bound kept yet."""
    def moments(n, size):
        v = (torch.rand(n, device="cuda", generator=g) + 0.1) * size ** 2 * 0.007
        return torch.randn(n, device="cuda", generator=g) * size * 0.5, v
    ma, va = moments(hb.n_alpha, 0.02)
    mb, vb = moments(hb.n_beta, 0.5)
    return dict(alpha_cur=_slopes(hb.n_alpha, g), m_alpha=ma, v_alpha=va, beta_cur=_multipliers(hb.n_beta, g),
                m_beta=mb, v_beta=vb, best_lb=torch.full((hb.B * K,), -math.inf, device="cuda"))


def _inputs(case, seed):
    layers, C, x_lo, x_hi, ls, us = _problem(case, seed)
    d = dict(layers=layers, C=C, x_lo=x_lo, x_hi=x_hi)
    if case["kind"] == "root":
        return d
    l, u = _usual_unstable(case["net"], ls, us)
    hb, U = _splits(case, seed, [ly.d_out for ly in layers[:-1]], l, u)
    g = torch.Generator(device="cuda").manual_seed(seed + 3)
    fresh = case["kind"] == "optimize" and not case["warm"]
    alpha = torch.full((hb.n_alpha,), 0.5, device="cuda") if fresh else _slopes(hb.n_alpha, g)
    beta = torch.zeros(hb.n_beta, device="cuda") if fresh else _multipliers(hb.n_beta, g)
    d.update(l=l, u=u, hb=hb, U=U, alpha=alpha, beta=beta)
    if case["kind"] == "optimize" and case["warm"]:
        d["opt"] = _state_of(case, hb, len(C), g)
    if case["kind"] == "joint":
        n_ap, n_bp = _joint_sizes(layers, d)
        d.update(alpha_p=_slopes(n_ap, g), beta_p=_multipliers(n_bp, g))
    if case["kind"] == "split":
        rng = np.random.default_rng(seed + 4)   # the neuron each subdomain is split on
        widths = [ly.d_out for ly in layers[:-1]]
        pl = rng.integers(1, len(widths) + 1, hb.B)
        d["pick"] = (pl.astype(np.uint8), np.floor(rng.random(hb.B) * np.array(widths)[pl - 1]).astype(np.int32))
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    host = [wl.Layer(ly.kind, ly.W.cpu().numpy(), ly.b.cpu().numpy(), ly.in_shape if ly.kind == "conv" else (ly.d_in,),
                     ly.out_shape if ly.kind == "conv" else (ly.d_out,), ly.stride, ly.pad) for ly in d["layers"]]
    st = dict(case=case, net=bc.load_net(host, d["C"].cpu().numpy()), x_lo=d["x_lo"].contiguous(),
              x_hi=d["x_hi"].contiguous())
    if case["kind"] != "root":
        st.update(dom=bc.Domain(st["x_lo"], st["x_hi"], d["l"], d["u"]), batch=bc.DeviceBatch.from_host(d["hb"]),
                  U=d["U"], alpha=d["alpha"], beta=d["beta"])
    if "opt" in d:
        st["opt"] = d["opt"]
    if case["kind"] == "joint":
        st.update(alpha_p=d["alpha_p"], beta_p=d["beta_p"])
    if case["kind"] == "split":
        st["pick"] = tuple(torch.from_numpy(x).cuda() for x in d["pick"])
    return st


_PRECISION = {"fp32": bc.FP32, "bf16": bc.BF16, "certify": bc.CERTIFY}


def run(state):
    case, net = state["case"], state["net"]
    kind = case["kind"]
    if kind == "root":
        return bc.root_bounds(net, state["x_lo"], state["x_hi"], precision=_PRECISION[case["precision"]])
    args = (net, state["dom"], state["batch"])
    if kind == "grad":
        return bc.bound_grad(*args, state["alpha"], state["beta"], _PRECISION[case["precision"]])
    if kind == "bound":
        return bc.bound(*args, state["alpha"], state["beta"], _PRECISION[case["precision"]])
    if kind == "xstar":
        lb, xs = bc.bound_xstar(*args, state["alpha"], state["beta"])
        return lb, xs, bc.forward(net, xs)
    if kind == "joint":
        return bc.bound_joint_grad(*args, state["alpha"], state["beta"], state["alpha_p"], state["beta_p"])
    if kind == "split":
        child, a, b = bc.batch_split(*args, *state["pick"], state["alpha"], state["beta"], state["U"])
        return (child.prop_of, child.split_off, child.split_cnt, child.split_layer, child.split_idx, child.split_sign,
                child.alpha_off, a, b)
    # the ascent overwrites its inputs, and the parents' slopes and multipliers are kept
    a, b = state["alpha"].clone(), state["beta"].clone()
    if not case["warm"]:
        return bc.optimize(*args, a, b, _opt_cfg(case)), a, b
    opt = bc.OptState(state["batch"], net.K)
    for k, v in state["opt"].items():
        getattr(opt, k).copy_(v)
    opt.t = 7
    lb = bc.optimize(*args, a, b, _opt_cfg(case), state=opt)
    return lb, a, b, opt.alpha_cur, opt.beta_cur, opt.m_alpha, opt.v_alpha, opt.m_beta, opt.v_beta, opt.best_lb


def work(case):
    spec, geo = NETS[case["net"]], _geometry(case["net"])
    K, B, P, U = spec["K"], case["B"], case["P"], sum(spec["unstable"])
    macs = [math.prod(ws) * (o[1] * o[2] if kind == "conv" else 1) for kind, ws, i, o, s, p in geo[:-1]]
    weights = 4 * sum(math.prod(ws) + ws[0] for kind, ws, i, o, s, p in geo)
    d0, widths = math.prod(spec["shape"]), [math.prod(g[3]) for g in geo[:-1]]
    H, R, S = sum(widths), B * K, B * (spec["depth"] + 1) / 2
    props = 4 * P * (2 * d0 + 2 * H)
    lists = B * 20 + S * 6
    na, nb = R * U, S * K
    base = weights + props + lists + 4 * (na + nb) + 4 * R
    per_row = 2 * sum(macs)
    kind = case["kind"]
    if kind == "grad":
        return {"bytes": base + 4 * (na + nb), "flops": 2 * per_row * R}
    if kind == "bound":
        return {"bytes": base, "flops": per_row * R}
    if kind == "xstar":
        return {"bytes": base + 4 * R * d0 + 4 * R * K, "flops": (2 * per_row + 2 * K * widths[-1]) * R}
    if kind == "split":
        return {"bytes": lists + 3 * 4 * (na + nb) + 2 * (lists + 6 * B), "flops": 0}
    if kind == "optimize":
        state = 4 * R + 24 * (na + nb) if case["warm"] else 0
        return {"bytes": base + 4 * (na + nb) + 2 * state, "flops": (2 * case["iters"] + 1) * per_row * R}
    # rows +-z_j of the hidden layers T >= 2, each through the layers below (the top's own
    # weights are its rows, so they need no contraction)
    below = [2 * sum(macs[:t]) for t in range(len(macs))]
    rows = sum(2 * widths[t] * below[t] for t in range(1, len(widths)))
    if kind == "root":
        return {"bytes": weights + props, "flops": P * (rows + 2 * macs[0])}
    first = [sum(spec["unstable"][:t]) for t in range(1, len(widths))]
    na_p, nb_p = B * 2 * sum(first), 2 * (len(widths) - 1) * S
    return {"bytes": base + 4 * (na + nb) + 8 * (na_p + nb_p), "flops": 2 * (per_row * R + B * rows)}


# --------------------------------------------------------------------------------------------
# The same results in 64 bits with torch
# --------------------------------------------------------------------------------------------

def _split_tables(d, bs, dev):
    """Signs and list positions [len(bs), H] of the subdomains' splits."""
    hb = d["hb"]
    edge = np.concatenate([[0], np.cumsum([ly.d_out for ly in d["layers"][:-1]])])
    sign = np.zeros((len(bs), edge[-1]), np.int8)
    slot = np.zeros((len(bs), edge[-1]), np.int64)
    for q, b in enumerate(bs):
        o, c = int(hb.split_off[b]), int(hb.split_cnt[b])
        g = edge[hb.split_layer[o:o + c].astype(np.int64) - 1] + hb.split_idx[o:o + c].astype(np.int64)
        sign[q, g] = hb.split_sign[o:o + c]
        slot[q, g] = np.arange(c)
    return torch.from_numpy(sign).to(dev), torch.from_numpy(slot).to(dev)


def _back(layers, T, A, c, x_lo, x_hi, bounds, sign, shift, slope):
    """Theorem 3.1 for rows [n, rows]: A [n, rows, d_T] over the post-activations of layer T, c
    [n, rows]; bounds[m] = (l, u), sign[m], shift[m] (beta S) and slope[m] of hidden layer m,
    each broadcast to [n, rows, d_m].  Returns lb [n, rows] and A^(0)."""
    n, rows = A.shape[:2]
    for m in range(T, -1, -1):
        l, u = bounds[m]
        act, uns, s, t = _chords(l, u)
        sg = sign[m]
        pos = A >= 0
        D = torch.where(act, 1.0, torch.where(uns, torch.where(pos, slope[m].clamp(0, 1), s), 0.0))
        D = torch.where(sg == 0, D, (sg < 0).to(A.dtype))
        L = A * D + shift[m]
        c = c + (L * layers[m].bias()).sum(-1) + torch.where(pos | (sg != 0), torch.zeros_like(A), A * t).sum(-1)
        A = layers[m].bwd(L.reshape(n * rows, -1)).reshape(n, rows, -1)
    x = torch.where(A >= 0, x_lo[:, None], x_hi[:, None])
    return c + (A * x).sum(-1), A


def _rows64(d, layers, bs, alpha, beta, want_x=False):
    """lb [len(bs), K] (and x*) of subdomains bs of one property, at alpha [n, K, U] and beta [n, K, depth]."""
    hb, dev = d["hb"], "cuda"
    p = int(hb.prop_of[bs[0]])
    l, u = d["l"][p].double(), d["u"][p].double()
    uns = torch.nonzero((l < 0) & (u > 0))[:, 0]
    sign, slot = _split_tables(d, bs, dev)
    full = torch.zeros(alpha.shape[:2] + (len(l),), device=dev, dtype=torch.float64)
    full = full.index_copy(2, uns, alpha)
    shift = torch.gather(beta.clamp(min=0), 2, slot[:, None].expand(-1, alpha.shape[1], -1)) * sign[:, None]
    edge = np.concatenate([[0], np.cumsum([ly.d_out for ly in layers[:-1]])])

    def cut(v):
        return [v[..., edge[m]:edge[m + 1]] for m in range(len(layers) - 1)]
    Wb, bb = d["C"].double() @ layers[-1].W, d["C"].double() @ layers[-1].b
    n, K = alpha.shape[:2]
    lb, A = _back(layers, len(layers) - 2, Wb.expand(n, -1, -1), bb.expand(n, K), d["x_lo"][p].double()[None],
                  d["x_hi"][p].double()[None], list(zip(cut(l), cut(u))), cut(sign[:, None]), cut(shift), cut(full))
    return (lb, torch.where(A >= 0, d["x_lo"][p].double(), d["x_hi"][p].double())) if want_x else lb


def _groups(d, layers, rows_bytes=1 << 28):
    """Subdomains of one property each, at most a memory's worth at once."""
    hb, K = d["hb"], len(d["C"])
    most = max(1, int(rows_bytes // (K * 8 * max(ly.d_in for ly in layers))))
    for p in range(len(d["x_lo"])):
        bs = np.flatnonzero(hb.prop_of == p)
        for q in range(0, len(bs), most):
            yield bs[q:q + most]


def _gather(d, bs, v, per):
    """The values of subdomains bs out of a flat array, padded to [n, K, most], and their indices."""
    hb, K = d["hb"], len(d["C"])
    if per == "alpha":
        cnt = d["U"][hb.prop_of[bs]]
        start = hb.alpha_off[bs]
    else:
        cnt, start = hb.split_cnt[bs].astype(np.int64), hb.split_off[bs].astype(np.int64) * K
    most = max(1, int(cnt.max(initial=0)))
    i = start[:, None, None] + np.arange(K)[None, :, None] * cnt[:, None, None] + np.arange(most)[None, None]
    used = torch.from_numpy(np.broadcast_to(np.arange(most)[None, None] < cnt[:, None, None], i.shape).copy()).cuda()
    i = torch.from_numpy(i).cuda().clamp_(max=max(0, v.numel() - 1))
    got = v[i] * used if v.numel() else torch.zeros(i.shape, device="cuda", dtype=v.dtype)
    return got, i, used


def _grad64(d, layers, alpha, beta):
    K = len(d["C"])
    lb = torch.empty(d["hb"].B * K, device="cuda", dtype=torch.float64)
    da, db = torch.zeros_like(alpha), torch.zeros_like(beta)
    rows = torch.arange(K, device="cuda")
    for bs in _groups(d, layers):
        a, ia, ua = _gather(d, bs, alpha, "alpha")
        b, ib, ub = _gather(d, bs, beta, "beta")
        a.requires_grad_(True)
        b.requires_grad_(True)
        out = _rows64(d, layers, bs, a, b)
        ga, gb = torch.autograd.grad(out.sum(), (a, b), allow_unused=True)
        lb[torch.from_numpy(bs).cuda()[:, None] * K + rows] = out.detach()
        da[ia[ua]] = ga[ua]
        if beta.numel() and gb is not None:
            db[ib[ub]] = gb[ub]
    return lb, da, db


def _bound64(d, layers, alpha, beta, want_x=False):
    K = len(d["C"])
    lb = torch.empty(d["hb"].B * K, device="cuda", dtype=torch.float64)
    xs = torch.empty((d["hb"].B * K, layers[0].d_in), device="cuda", dtype=torch.float64) if want_x else None
    for bs in _groups(d, layers):
        out = _rows64(d, layers, bs, _gather(d, bs, alpha, "alpha")[0], _gather(d, bs, beta, "beta")[0], want_x)
        at = torch.from_numpy(bs).cuda()[:, None] * K + torch.arange(K, device="cuda")
        lb[at] = out[0] if want_x else out
        if want_x:
            xs[at] = out[1]
    return (lb, xs) if want_x else lb


def _forward64(d, layers, x):
    for ly in layers[:-1]:
        x = torch.relu(ly.fwd(x) + ly.bias())
    return (x @ layers[-1].W.T + layers[-1].b) @ d["C"].double().T


def _owners(d):
    """Row of every alpha and every beta entry."""
    hb, K = d["hb"], len(d["C"])
    row = np.arange(hb.B)[:, None] * K + np.arange(K)
    ra = np.repeat(row.reshape(-1), np.repeat(d["U"][hb.prop_of], K))
    rb = np.repeat(row.reshape(-1), np.repeat(hb.split_cnt.astype(np.int64), K))
    return torch.from_numpy(ra).cuda(), torch.from_numpy(rb).cuda()


def _ascent64(case, d, layers):
    """The projected Adam ascent (Appendix C.1) in 64 bits: the final bound and the state."""
    cfg = _opt_cfg(case)
    ra, rb = _owners(d)
    best = [d["alpha"].double(), d["beta"].double()]
    t0 = 7 if case["warm"] else 0
    if case["warm"]:
        o = {k: v.double() for k, v in d["opt"].items()}
        th, m, v, top = [o["alpha_cur"], o["beta_cur"]], [o["m_alpha"], o["m_beta"]], [o["v_alpha"], o["v_beta"]], o["best_lb"]
    else:
        th = [x.clone() for x in best]
        m, v = [torch.zeros_like(x) for x in th], [torch.zeros_like(x) for x in th]
        top = torch.full((d["hb"].B * len(d["C"]),), -math.inf, device="cuda", dtype=torch.float64)
    for t in range(t0, t0 + cfg.iters):
        lb, *g = _grad64(d, layers, *th)
        up = lb > top
        top = torch.where(up, lb, top)
        best = [torch.where(up[r], x, b) for r, x, b in zip((ra, rb), th, best)]
        for q, lr in ((0, cfg.lr_alpha), (1, cfg.lr_beta)):
            m[q] = cfg.adam_beta1 * m[q] + (1 - cfg.adam_beta1) * g[q]
            v[q] = cfg.adam_beta2 * v[q] + (1 - cfg.adam_beta2) * g[q] ** 2
            step = m[q] / (1 - cfg.adam_beta1 ** (t + 1)) / ((v[q] / (1 - cfg.adam_beta2 ** (t + 1))).sqrt() + cfg.adam_eps)
            th[q] = (th[q] + lr * cfg.decay ** t * step).clamp(0, 1 if q == 0 else math.inf)
    lb = _bound64(d, layers, *best)
    # which iterate a row keeps turns on differences below the BF16 rounding: no value for those
    if not case["warm"]:
        return lb, None, None
    return lb, None, None, th[0], th[1], m[0], v[0], m[1], v[1], top


def _joint_sizes(layers, d):
    hb, uns = d["hb"], ((d["l"] < 0) & (d["u"] > 0)).cpu().numpy()
    edge = np.cumsum([ly.d_out for ly in layers[:-1]])
    first = np.stack([uns[:, :edge[t - 1]].sum(1) for t in range(1, len(edge))], 1) if len(edge) > 1 else np.zeros((len(uns), 0))
    return int(2 * first.sum(1)[hb.prop_of].sum()), int(2 * (len(edge) - 1) * hb.split_cnt.sum())


def _joint64(d, layers):
    """lb and the four gradients with the intermediate bounds recomputed (Section 3.3)."""
    hb, K, dev = d["hb"], len(d["C"]), "cuda"
    v = {k: d[k].double().requires_grad_(True) for k in ("alpha", "beta", "alpha_p", "beta_p")}
    edge = np.concatenate([[0], np.cumsum([ly.d_out for ly in layers[:-1]])])
    L = len(layers)
    lbs, at_p = [], 0
    for b in range(hb.B):
        p, off, cnt = int(hb.prop_of[b]), int(hb.split_off[b]), int(hb.split_cnt[b])
        lr, ur = d["l"][p].double(), d["u"][p].double()
        root_uns = (lr < 0) & (ur > 0)
        sign, slot = (x[0] for x in _split_tables(d, [b], dev))
        x_lo, x_hi = d["x_lo"][p].double()[None], d["x_hi"][p].double()[None]

        def tables(upto, slopes, betas):
            """Per layer < upto: signs, shifts, slopes from vectors by rank and by list position."""
            uns = torch.nonzero(root_uns[:edge[upto]])[:, 0]
            full = torch.zeros(slopes.shape[:-1] + (int(edge[upto]),), device=dev, dtype=torch.float64).index_copy(-1, uns, slopes)
            shift = betas.clamp(min=0)[..., slot[:edge[upto]]] * sign[:edge[upto]] if cnt else torch.zeros_like(full)
            cut = lambda x: [x[..., edge[m]:edge[m + 1]] for m in range(upto)]  # noqa: E731
            return cut(sign[:edge[upto]].expand_as(full)), cut(shift), cut(full)

        bounds = [(lr[:edge[1]], ur[:edge[1]])]
        for T in range(1, L - 1):
            f = int(root_uns[:edge[T]].sum())
            made = []
            for way in (0, 1):
                sl = v["alpha_p"][at_p:at_p + f]
                at_p += f
                b0 = 2 * (L - 2) * off + (2 * (T - 1) + way) * cnt
                sg, sh, fu = tables(T, sl, v["beta_p"][b0:b0 + cnt])
                s = 1.0 if way == 0 else -1.0
                lb, _ = _back(layers, T - 1, (s * layers[T].W)[None], (s * layers[T].bias())[None], x_lo, x_hi, bounds, sg, sh, fu)
                made.append(s * lb[0])
            l0, u0 = lr[edge[T]:edge[T + 1]], ur[edge[T]:edge[T + 1]]
            bounds.append((torch.where(made[0] > l0, made[0], l0), torch.where(made[1] < u0, made[1], u0)))
        U = int(d["U"][p])
        a0 = int(hb.alpha_off[b])
        sg, sh, fu = tables(L - 1, v["alpha"][a0:a0 + K * U].reshape(K, U), v["beta"][off * K:(off + cnt) * K].reshape(K, cnt))
        Wb, bb = d["C"].double() @ layers[-1].W, d["C"].double() @ layers[-1].b
        lb, _ = _back(layers, L - 2, Wb[None], bb[None], x_lo, x_hi, bounds, sg, sh, fu)
        lbs.append(lb[0])
    lb = torch.cat(lbs)
    g = torch.autograd.grad(lb.sum(), list(v.values()), allow_unused=True)
    return (lb.detach(), *[torch.zeros_like(x) if y is None else y for x, y in zip(v.values(), g)])


def exact(case, seed):
    if case["kind"] == "split":
        return None   # whole numbers, and copies
    if work(case)["flops"] > 6e12:
        return None
    d = _inputs(case, seed)
    with _conv_exactly():
        layers = [ly.to(torch.float64) for ly in d["layers"]]
        if case["kind"] == "root":
            ls, us = _root_bounds(layers, d["x_lo"].double(), d["x_hi"].double())
            return torch.cat(ls, 1), torch.cat(us, 1), None
        if case["kind"] == "joint":
            return _joint64(d, layers)
        if case["kind"] == "optimize":
            return _ascent64(case, d, layers)
        a, b = d["alpha"].double(), d["beta"].double()
        if case["kind"] == "grad":
            return _grad64(d, layers, a, b)
        if case["kind"] == "bound":
            return _bound64(d, layers, a, b)
        lb, xs = _bound64(d, layers, a, b, want_x=True)
        return lb, xs, _forward64(d, layers, xs)
