"""The work this framework is asked to do, as a list of measured cases.

A case names a network of `paper_2101_05844_gb300.synth`, a number of subproblems S and a kind:

  solve         a whole bounding call on a new batch: reset (interval bounds), Big-M and Active Set
                iterations from zero (or a parent's) duals, optionally Saddle Point after them, bound
  iterate       a stretch of Big-M / Active Set iterations of a solve under way, `cuts` masks per
                neuron in use, and the bound at its end; `precision` 16 is the BF16 form
  saddle        a stretch of Saddle Point iterations of a solve under way, and the bound at its end
  intervals     a new batch on a context: its intermediate bounds by interval propagation
  gradient      the differentiable bound and its gradient (weights, biases, input box)
  intermediate  intermediate bounds by batched dual solves over sub-networks

The networks' weights are the same for every seed (a user verifies one network on many inputs); boxes,
properties, splits and the duals of a solve under way come from the seed.

Duals and primal iterates are returned where a pass starts from drawn ones. A whole solve starts from
zero duals, where the iterates follow every decision of the first steps; it returns what its caller asks
for, the bounds. `bound_into(32, ...)` sums the per-neuron terms in float32, so the float64 buffer it
fills holds float32 numbers, and they are returned as such.
"""
import math

import torch
import torch.nn.functional as F

from paper_2101_05844_gb300 import autograd, binding, synth

PLANNED = 400_000   # iterations a solve under way has planned; it is met three quarters in
STARTED = 300_000
SADDLE_STARTED = 6000   # Saddle Point is run for thousands of iterations: step 1 / (t + 10)

_NETS = {}


def listed():
    return [
        # one property of a small MLP on one box, a whole solve: nothing but latency and launches
        dict(name="mlp_one_box_solve", kind="solve", net="mlp_8_16_16_1", S=1, bigm=20, act=80, sp=0, cuts=5,
             splits=0, warm=False),
        # one image against its nine other classes: the smallest batch of a verification query
        dict(name="wide_nine_properties", kind="iterate", net="wide_conv", S=9, cuts=5, iters=25, precision=32),
        dict(name="wide_nine_saddle", kind="saddle", net="wide_conv", S=9, iters=25),
        # a batch of branch and bound: 250 children of one box, warm-started, the inexpensive solver
        dict(name="bab_children", kind="solve", net="wide_conv", S=250, bigm=60, act=0, sp=0, cuts=3, splits=20,
             warm=True),
        # thousands of subdomains with one to five masks each, the tighter solver
        dict(name="bab_subdomains", kind="iterate", net="wide_conv", S=2048, cuts=5, iters=8, precision=32, splits=20),
        # the deeper conv net at 8/255, float32 and the BF16 form, and Saddle Point
        dict(name="conv4_float32", kind="iterate", net="conv4", S=64, cuts=5, iters=8, precision=32),
        dict(name="conv4_bf16", kind="iterate", net="conv4", S=1024, cuts=5, iters=8, precision=16),
        dict(name="conv4_saddle", kind="saddle", net="conv4", S=64, iters=4),
        # a new batch of boxes on an existing context
        dict(name="conv4_intervals", kind="intervals", net="conv4", S=256),
        # the dense MLP: the BF16 form, the gradient for training, the hidden layers' tightened bounds
        dict(name="mlp_wide_bf16", kind="iterate", net="mlp_784_1024x3_10", S=256, cuts=5, iters=16, precision=16),
        dict(name="mlp_wide_gradient", kind="gradient", net="mlp_784_1024x3_10", S=256, cuts=3, chain=False),
        dict(name="mlp_intermediate", kind="intermediate", net="mlp_784_256_256_10", S=1, bigm=16, act=0, cuts=2),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))

    kind = rng.choice(["solve", "iterate", "iterate", "iterate", "saddle", "intervals", "gradient", "intermediate"])
    net = rng.choice(["wide_conv", "wide_conv", "conv4", "mlp_784_1024x3_10", "mlp_100_75_33_7", "small_conv"])
    heavy = {"conv4": 16, "mlp_784_1024x3_10": 4, "wide_conv": 1}.get(net, 0.1)
    if kind == "solve":
        return dict(kind=kind, net=net, S=spread(1, max(2, int(256 / max(1, heavy)))), bigm=rng.randint(10, 30),
                    act=rng.randint(0, 20), sp=rng.choice([0, 0, 8]), cuts=rng.randint(1, 7),
                    splits=rng.choice([0, 5, 20]), warm=rng.choice([False, True]))
    if kind == "iterate":
        return dict(kind=kind, net=net, S=spread(1, int(2048 / max(1, heavy))), cuts=rng.randint(0, 7),
                    iters=rng.randint(1, 16), precision=rng.choice([32, 32, 16]), splits=rng.choice([0, 0, 20]))
    if kind == "saddle":
        return dict(kind=kind, net=net, S=spread(1, int(512 / max(1, heavy))), iters=rng.randint(1, 8))
    if kind == "intervals":
        return dict(kind=kind, net=net, S=spread(1, int(4096 / max(1, heavy))))
    if kind == "gradient":
        return dict(kind=kind, net=net, S=spread(1, int(128 / max(1, heavy / 4))), cuts=rng.randint(0, 5),
                    chain=rng.choice([False, True]))
    net = "mlp_%d_%d_%d_10" % (spread(50, 784), spread(40, 300), spread(20, 300))
    return dict(kind=kind, net=net, S=rng.randint(1, 2), bigm=rng.randint(5, 16), act=0, cuts=2)


# ------------------------------------------------------------------------------------ inputs
def _net(name):
    if name not in _NETS:
        layers = synth.small_convnet() if name == "small_conv" else synth.arch(name)
        _NETS[name] = synth.make_net(layers, 1)
    return _NETS[name]


def _eps(name):
    return {"wide_conv": 2 / 255, "conv4": 8 / 255}.get(name, 0.1)


def _boxes(case, seed, gen):
    """Boxes around U[0, 1] centres and one property row each: y against the runner-up at the centre."""
    net, S = _net(case["net"]), case["S"]
    shared = case["kind"] == "solve" or case.get("splits", 0) > 0   # subdomains or properties of one box
    c = torch.rand((1 if shared else S, net[0]["n_in"]), generator=gen, device="cuda")
    e = _eps(case["net"])
    lo, hi = (c - e).expand(S, -1).contiguous(), (c + e).expand(S, -1).contiguous()
    n_out = net[-1]["n_out"]
    if n_out == 1:
        C = torch.ones((S, 1), device="cuda")
    else:
        h = c
        for q, L in enumerate(net):
            W, b = torch.from_numpy(L["W"]).cuda(), torch.from_numpy(L["b"]).cuda()
            if L["kind"] == "linear":
                h = h @ W.T + b
            else:
                h = F.conv2d(h.view(-1, *L["in_shape"]), W, b, stride=L["stride"], padding=L["pad"]).flatten(1)
            h = torch.relu(h) if q + 1 < len(net) else h
        order = h.argsort(1, descending=True).expand(S, -1)
        other = 1 + (torch.arange(S, device="cuda") % (n_out - 1) if shared else torch.zeros(S, dtype=torch.long, device="cuda"))
        C = torch.zeros((S, n_out), device="cuda")
        C[torch.arange(S), order[:, 0]] = 1.0
        C[torch.arange(S), order.gather(1, other[:, None])[:, 0]] = -1.0
    return lo, hi, C


def _splits(case, gen, NH):
    """Up to `splits` split neurons per subdomain, active or inactive; None without splits."""
    k = case.get("splits", 0)
    if not k:
        return None
    S, k = case["S"], min(k, NH)
    out = torch.zeros((S, NH), dtype=torch.int8, device="cuda")
    at = torch.randint(0, NH // k, (S, k), generator=gen, device="cuda") + torch.arange(k, device="cuda") * (NH // k)
    sign = torch.randint(0, 2, (S, k), generator=gen, device="cuda") * 2 - 1
    keep = torch.arange(k, device="cuda") < torch.randint(0, k + 1, (S, 1), generator=gen, device="cuda")
    out.scatter_(1, at, (sign * keep).to(torch.int8))
    return out


def _caps(case, gen):
    if not case.get("splits", 0) or case["kind"] != "iterate":
        return None
    return torch.randint(1, max(1, case["cuts"]) + 1, (case["S"],), generator=gen, device="cuda", dtype=torch.int32)


def _dual(gen, *shape):
    v = torch.rand(shape, generator=gen, device="cuda") * 0.3
    return v * (torch.rand(shape, generator=gen, device="cuda") >= 0.3)


def _duals(case, gen, lhat, uhat, NT):
    """Duals, moments and snapshots of an Active Set solve under way; Adam's moments at the scale of
    the supergradients, whose entries span the neurons' pre-activation intervals."""
    S, NH = lhat.shape
    cuts, cap = case["cuts"], max(1, case["cuts"])
    width = (0.25 * (uhat - lhat) + 1e-3).float()

    def moments(w):
        m = torch.randn(w.shape, generator=gen, device="cuda") * w
        v = (0.5 + torch.rand(w.shape, generator=gen, device="cuda")) * w * w
        return m, v

    d = dict(alpha=_dual(gen, S, NH), beta0=_dual(gen, S, NH), beta1=_dual(gen, S, NH))
    d["adam"] = torch.stack([t for _ in range(3) for t in moments(width)])
    d["slot"] = _dual(gen, S, cap, NH) if cuts else torch.zeros((S, cap, NH), device="cuda")
    d["slot_adam"] = torch.stack(moments(width[:, None].expand(S, cap, NH)))
    bits = (1 << cuts) - 1
    d["xsnap"] = torch.randint(0, 256, (S, NT), generator=gen, device="cuda", dtype=torch.uint8) & bits
    d["zsnap"] = torch.randint(0, 256, (S, NH), generator=gen, device="cuda", dtype=torch.uint8) & bits
    if case.get("caps") is not None:
        on = torch.arange(cap, device="cuda")[None, :] < case["caps"][:, None]
        d["slot"] = d["slot"] * on[..., None]
    return d


def _saddle_state(case, gen, lo, hi, lhat, uhat):
    """Primal iterate, duals and statistics of a Saddle Point solve under way."""
    S, NH = lhat.shape
    NT = lo.shape[1]
    d = dict(alpha=_dual(gen, S, NH))
    d["x"] = lo + torch.rand(lo.shape, generator=gen, device="cuda") * (hi - lo)
    d["z"] = torch.rand((S, NH), generator=gen, device="cuda")
    Sb = _dual(gen, S, NH)
    share = torch.rand((S, NH), generator=gen, device="cuda")
    G = Sb * (share * uhat + (1 - share) * lhat)
    C = Sb * (1 - share) * lhat
    P = torch.randn((S, NT), generator=gen, device="cuda") * 0.1
    P[:, NT - _net(case["net"])[-1]["n_in"]:] = 0.0   # the last hidden layer feeds no masked product
    d.update(Sb=Sb, G=G, C=C, P=P)
    d["mua"] = torch.where(d["alpha"] > 0, d["alpha"], 1e-3) * 1.5
    d["mub"] = torch.where(Sb > 0, Sb, 1e-3) * 1.5
    return d


def _options(case):
    if case["kind"] == "saddle":
        return binding.default_options(bigm_iters=1, as_iters=0, max_cuts=1, graph_chunk=case["iters"])
    if case["kind"] in ("iterate", "gradient"):
        cuts, n = case["cuts"], case.get("iters", 0)
        kw = dict(max_cuts=max(1, cuts), graph_chunk=n, precision=case.get("precision", 32))
        kw.update(bigm_lr0=4e-5, bigm_lr1=1e-6, as_lr0=4e-5, as_lr1=1e-6)   # a solve's last, small steps
        if cuts:   # every mask was added in the first `cuts` Active Set iterations
            return binding.default_options(bigm_iters=100, as_iters=PLANNED, omega=0, vars_per_add=cuts, **kw)
        return binding.default_options(bigm_iters=PLANNED, as_iters=0, **kw)
    if case["kind"] == "intervals":
        return binding.default_options()
    kw = dict(bigm_iters=case["bigm"], as_iters=case["act"], max_cuts=case["cuts"])
    if case["kind"] == "solve":   # small steps: children refine their parent's duals
        kw.update(bigm_lr0=1e-4, bigm_lr1=1e-6, as_lr0=1e-4, as_lr1=1e-6)
    else:
        kw.update(bigm_lr0=1e-3, bigm_lr1=1e-4)
    return binding.default_options(omega=max(2, int(0.3 * case["act"])), sp_init_steps=10, **kw)


def _set(ctx, which, t):
    """as_set_state from a device tensor."""
    r = binding.lib().as_set_state(ctx.h, which, t.contiguous().data_ptr())
    if r != binding.AS_OK:
        raise binding.CBError(r, "as_set_state")


def _get(ctx, which, t):
    """as_get_state into a device tensor."""
    r = binding.lib().as_get_state(ctx.h, which, t.data_ptr())
    if r != binding.AS_OK:
        raise binding.CBError(r, "as_get_state")
    return t


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def prepare(case, seed):
    gen = _gen(seed)
    net = _net(case["net"])
    kind, S = case["kind"], case["S"]
    NT = sum(L["n_in"] for L in net)
    NH = NT - net[0]["n_in"]
    lo, hi, C = _boxes(case, seed, gen)
    if kind == "intermediate":
        return dict(kind=kind, net=net, lo=lo, hi=hi, options=_options(case))
    if kind == "gradient":
        net = [dict(L, W=torch.from_numpy(L["W"]).cuda(), b=torch.from_numpy(L["b"]).cuda()) for L in net]
    splits, caps = _splits(case, gen, NH), _caps(case, gen)
    ctx = binding.Context(net, lo, hi, C, None, None, splits, caps, _options(case))
    st = dict(kind=kind, ctx=ctx, lo=lo, hi=hi, C=C, splits=splits, caps=caps, case=dict(case),
              out=torch.zeros(S, dtype=torch.float64, device="cuda"))
    hidden = lambda: torch.empty((S, NH), device="cuda")  # noqa: E731
    if kind == "solve":
        if case["warm"]:
            st["parent"] = [_dual(gen, S, NH) for _ in range(3)]
        return st
    if kind == "intervals":
        st.update(lhat=hidden(), uhat=hidden())
        return st
    lhat, uhat = _get(ctx, binding.ST_LHAT, hidden()), _get(ctx, binding.ST_UHAT, hidden())
    if kind == "saddle":
        plo, phi = (_get(ctx, w, torch.empty((S, NT), device="cuda")) for w in (binding.ST_LO, binding.ST_HI))
        d = _saddle_state(case, gen, plo, phi, lhat, uhat)
        _set(ctx, binding.ST_ITER, torch.tensor([0, SADDLE_STARTED, 1], dtype=torch.int32, device="cuda"))
        stats = torch.zeros((4, S, NT), device="cuda")
        for q, key in enumerate(("Sb", "G", "C")):
            stats[q, :, NT - NH:] = d[key]
        stats[3] = d["P"]
        _set(ctx, binding.ST_SP_STATS, stats)
        _set(ctx, binding.ST_SP_CAPS, torch.stack([d["mua"], d["mub"]]))
        _set(ctx, binding.ST_SP_X, d["x"])
        _set(ctx, binding.ST_SP_Z, d["z"])
        _set(ctx, binding.ST_ALPHA, d["alpha"])
        st.update(alpha=hidden(), z=hidden(), x=torch.empty((S, NT), device="cuda"))
        return st
    d = _duals(dict(case, caps=caps), gen, lhat, uhat, NT)
    _set(ctx, binding.ST_ITER, torch.tensor([STARTED, 0, 0], dtype=torch.int32, device="cuda"))
    _set(ctx, binding.ST_BETA0, d["beta0"])
    _set(ctx, binding.ST_BETA1, d["beta1"])
    _set(ctx, binding.ST_ADAM, d["adam"])
    _set(ctx, binding.ST_SLOT_ADAM, d["slot_adam"])
    if case["cuts"]:
        _set(ctx, binding.ST_XSNAP, d["xsnap"])
        _set(ctx, binding.ST_ZSNAP, d["zsnap"])
        _set(ctx, binding.ST_SLOT_BETA, d["slot"])
    _set(ctx, binding.ST_ALPHA, d["alpha"])
    if kind == "gradient":
        st["leaves"] = [t.detach().clone().requires_grad_(True)
                        for t in (lo, hi, *[L[k] for L in net for k in ("W", "b")])]
        st["seed_grad"] = torch.rand(S, generator=gen, device="cuda", dtype=torch.float64)
        if case["chain"]:
            st["grads"] = [torch.zeros_like(t) for t in st["leaves"]]
        return st
    st.update(alpha=hidden(), beta0=hidden(), beta1=hidden())
    st["slot"] = torch.empty((S, max(1, case["cuts"]), NH), device="cuda") if case["cuts"] else None
    return st


def run(state):
    kind = state["kind"]
    if kind == "intermediate":
        return dict(zip(("lhat", "uhat"), binding.intermediate_bounds(state["net"], state["lo"], state["hi"],
                                                                      options=state["options"])))
    ctx, case = state["ctx"], state["case"]
    if kind == "intervals":
        ctx.reset(state["lo"], state["hi"], state["C"])
        return {"lhat": _get(ctx, binding.ST_LHAT, state["lhat"]), "uhat": _get(ctx, binding.ST_UHAT, state["uhat"])}
    if kind == "gradient":
        if case["chain"]:   # through the interval bounds, gradients accumulated into the caller's buffers
            g = state["grads"]
            for t in g:
                t.zero_()
            ctx.bound_into(32, state["out"])
            ctx.backward(state["seed_grad"], g[2::2], g[3::2], g[0], g[1], through_bounds=True)
            return {"bound": state["out"].float(), "grads": g}
        leaves = state["leaves"]
        bound = autograd.bound(ctx, leaves[0], leaves[1], leaves[2:])
        return {"bound": bound.detach().float(), "grads": list(torch.autograd.grad(bound, leaves, state["seed_grad"]))}
    if kind == "solve":
        ctx.reset(state["lo"], state["hi"], state["C"], None, None, state["splits"])
        if case["warm"]:
            for which, t in zip((binding.ST_ALPHA, binding.ST_BETA0, binding.ST_BETA1), state["parent"]):
                _set(ctx, which, t)
        ctx.as_step(case["bigm"] + case["act"])
        if case["sp"]:
            ctx.sp_step(case["sp"])
        ctx.bound_into(32, state["out"])
        return {"bound": state["out"].float()}
    if kind == "saddle":
        ctx.sp_step(case["iters"])
        ctx.bound_into(32, state["out"])
        return {"bound": state["out"].float(), "alpha": _get(ctx, binding.ST_ALPHA, state["alpha"]),
                "x": _get(ctx, binding.ST_SP_X, state["x"]), "z": _get(ctx, binding.ST_SP_Z, state["z"])}
    ctx.as_step(case["iters"])
    ctx.bound_into(32, state["out"])
    got = {"bound": state["out"].float()}
    for key, which in (("alpha", binding.ST_ALPHA), ("beta0", binding.ST_BETA0), ("beta1", binding.ST_BETA1),
                       ("slot", binding.ST_SLOT_BETA)):
        if state[key] is not None:
            got[key] = _get(ctx, which, state[key])
    return got


# ------------------------------------------------------------------------------------ work
def _sizes(net):
    nnz = 0
    for L in net[:-1]:
        if L["kind"] == "linear":
            nnz += L["n_in"] * L["n_out"]
        else:
            (c, h, w), (_, oh, ow) = L["in_shape"], L["out_shape"]
            rows = sum(1 for o in range(oh) for k in range(L["kh"]) if 0 <= o * L["stride"] - L["pad"] + k < h)
            cols = sum(1 for o in range(ow) for k in range(L["kw"]) if 0 <= o * L["stride"] - L["pad"] + k < w)
            nnz += L["out_c"] * c * rows * cols
    NT = sum(L["n_in"] for L in net)
    return nnz, NT, NT - net[0]["n_in"], sum(L["W"].size + L["b"].size for L in net)


def work(case):
    net = _net(case["net"])
    nnz, NT, NH, weights = _sizes(net)
    S, kind = case["S"], case["kind"]
    # an iteration reads and writes the duals and both moments of alpha, beta_0, beta_1 and every slot,
    # and reads the neurons' boxes and pre-activation bounds; its products are one multiply-add per
    # nonzero weight, forward and backward, for the unmasked operand and for every slot
    def iteration(cuts):
        return (S * (NH * (72 + 24 * cuts + 8 * cuts + 8) + NT * 8) + 4 * weights, 4.0 * S * nnz * (1 + cuts))

    def saddle():   # alpha, Sb, G, C, P, x, z read and written, caps and boxes read; three row, two col sums
        return S * (NH * (4 * 10 + 8 + 8) + NT * (4 * 4 + 8)) + 4 * weights, 10.0 * S * nnz

    batch = S * (8 * net[0]["n_in"] + 8 * NH) + 4 * weights, 4.0 * S * nnz
    if kind == "iterate":
        b, f = iteration(case["cuts"])
        return {"bytes": case["iters"] * b, "flops": case["iters"] * f}
    if kind == "saddle":
        b, f = saddle()
        return {"bytes": case["iters"] * b, "flops": case["iters"] * f}
    if kind == "intervals":
        return {"bytes": batch[0], "flops": batch[1]}
    if kind == "gradient":   # the bound's evaluation, then one product per weight, slot and subproblem
        b, f = iteration(case["cuts"])
        return {"bytes": S * (NH * (20 + 12 * case["cuts"]) + NT * 8) + 12 * weights, "flops": f}
    if kind == "solve":
        total = [batch[0], batch[1]]
        for t in range(case["bigm"] + case["act"]):
            cuts = 0 if t < case["bigm"] else min(case["cuts"], 2)
            b, f = iteration(cuts)
            total = [total[0] + b, total[1] + f]
        return {"bytes": total[0], "flops": total[1]}
    total = [0.0, 0.0]   # intermediate: 2 n_k solves per box over layers 1 .. k-1
    for k in range(1, len(net) - 1):
        sub = net[:k + 1]
        sn, sNT, sNH, sw = _sizes(sub)
        rows = 2 * net[k]["n_out"] * S
        n = case["bigm"] + case["act"]
        total[0] += n * (rows * (sNH * 72 + sNT * 8) + 4 * sw)
        total[1] += n * 4.0 * rows * sn
    return {"bytes": total[0], "flops": total[1]}


# ------------------------------------------------------------------------------------ 64 bits
class _Net64:
    """The network's layers in float64 and plain torch: W x, W^T y, W+ and W- products."""

    def __init__(self, net, leaves=None):
        self.net = net
        par = leaves or [torch.from_numpy(L[k]).cuda().double() for L in net for k in ("W", "b")]
        self.W, self.b = par[0::2], []
        for L, b in zip(net, par[1::2]):
            self.b.append(b if L["kind"] == "linear" else b.repeat_interleave(L["n_out"] // L["out_c"]))
        self.pos = [torch.where(W >= 0, W, 0.0) for W in self.W]
        self.neg = [torch.where(W >= 0, 0.0, W) for W in self.W]
        self.n = len(net)
        self.widths = [L["n_in"] for L in net]

    def fwd(self, k, W, x):
        L = self.net[k]
        if L["kind"] == "linear":
            return x @ W.T
        return F.conv2d(x.view(-1, *L["in_shape"]), W, stride=L["stride"], padding=L["pad"]).flatten(1)

    def bwd(self, k, W, y):
        L = self.net[k]
        if L["kind"] == "linear":
            return y @ W
        (_, h, w), (_, oh, ow) = L["in_shape"], L["out_shape"]
        st, pd = L["stride"], L["pad"]
        extra = (h - ((oh - 1) * st - 2 * pd + L["kh"]), w - ((ow - 1) * st - 2 * pd + L["kw"]))
        return F.conv_transpose2d(y.view(-1, *L["out_shape"]), W, stride=st, padding=pd, output_padding=extra).flatten(1)

    def intervals(self, lo, hi, splits=None):
        los, his, lh, uh, at = [lo], [hi], [], [], 0
        for k in range(self.n - 1):
            a = self.fwd(k, self.pos[k], los[-1]) + self.fwd(k, self.neg[k], his[-1]) + self.b[k]
            c = self.fwd(k, self.pos[k], his[-1]) + self.fwd(k, self.neg[k], los[-1]) + self.b[k]
            if splits is not None:
                sp = splits[:, at:at + a.shape[1]]
                amb = (a < 0) & (c > 0)
                a, c = torch.where(amb & (sp > 0), 0.0, a), torch.where(amb & (sp < 0), 0.0, c)
            at += a.shape[1]
            lh.append(a)
            uh.append(c)
            los.append(a.clamp(min=0))
            his.append(c.clamp(min=0))
        return lh, uh, los, his


def _cut(t, widths):
    """A hidden vector's (last dimension's) layers."""
    return list(torch.split(t, widths[1:], -1))


class _Active64:
    """The dual function and Adam iterations of the Active Set solver (Alg. 1) in float64."""

    def __init__(self, N, lo, hi, C, bounds, d, cuts, caps=None):
        self.N, self.cuts = N, cuts
        self.lh, self.uh, self.lo, self.hi = bounds
        n, w = N.n, N.widths
        self.wout, self.bout = C @ N.W[n - 1], C @ N.b[n - 1]
        D = lambda t: t.double()  # noqa: E731
        self.a, self.b0, self.b1 = (_cut(D(d[k]), w) for k in ("alpha", "beta0", "beta1"))
        self.m = [_cut(D(t), w) for t in d["adam"]]
        self.s = [[t[:, b] for t in _cut(D(d["slot"]), w)] for b in range(cuts)]
        self.sm = [[[t[:, b] for t in _cut(D(q), w)] for b in range(cuts)] for q in d["slot_adam"]]
        self.on = [torch.ones(lo.shape[0], 1, dtype=torch.bool, device="cuda") if caps is None else (b < caps)[:, None]
                   for b in range(cuts)]
        xs, zs = list(torch.split(d["xsnap"].int(), w, -1)), _cut(d["zsnap"].int(), w)
        fixed = [a == c for a, c in zip(self.lo, self.hi)]
        self.p = [[((xs[k] >> b) & 1 == 0) | fixed[k] for k in range(n - 1)] for b in range(cuts)]
        self.q = [[((xs[k] >> b) & 1 == 1) | fixed[k] for k in range(n - 1)] for b in range(cuts)]
        self.zb = [[(zs[k] >> b) & 1 == 1 for k in range(n - 1)] for b in range(cuts)]
        self.sums()

    def masked(self, b, k, xp, xn, whole):
        """(W o I_b) applied to xp under positive and xn under negative weights; `whole`: rows of all ones."""
        N = self.N
        part = N.fwd(k, N.pos[k], xp * self.p[b][k]) + N.fwd(k, N.neg[k], xn * self.q[b][k])
        return torch.where(self.zb[b][k], whole, part)

    def sums(self):
        N = self.N
        self.lam, self.mu = [], []
        for b in range(self.cuts):
            la, mu = [], []
            for k in range(N.n - 1):
                l, u = self.lo[k], self.hi[k]
                la.append(self.masked(b, k, l, u, N.fwd(k, N.pos[k], l) + N.fwd(k, N.neg[k], u)))
                rest = N.fwd(k, N.pos[k], u * ~self.p[b][k]) + N.fwd(k, N.neg[k], l * ~self.q[b][k])
                mu.append(torch.where(self.zb[b][k], 0.0, rest))
            self.lam.append(la)
            self.mu.append(mu)

    def minimise(self):
        N, f, g = self.N, [], []
        for k in range(N.n):
            if k == N.n - 1:
                v = -self.wout
            else:
                row = -(self.a[k] - self.b1[k])
                for b in range(self.cuts):
                    row = row + torch.where(self.zb[b][k], self.s[b][k], 0.0)
                v = N.bwd(k, N.W[k], row)
                for b in range(self.cuts):
                    part = torch.where(self.zb[b][k], 0.0, self.s[b][k])
                    v = v + N.bwd(k, N.pos[k], part) * self.p[b][k] + N.bwd(k, N.neg[k], part) * self.q[b][k]
            if k:
                h = k - 1
                v = v + self.a[h] - self.b0[h] - self.b1[h] - sum(self.s[b][h] for b in range(self.cuts))
                gk = self.b0[h] * self.uh[h] + self.b1[h] * self.lh[h]
                for b in range(self.cuts):
                    gk = gk + self.s[b][h] * (self.lam[b][h] + self.mu[b][h] + N.b[h])
                g.append(gk)
            f.append(v)
        self.f = f
        self.up = [v >= 0 for v in f]
        self.x = [torch.where(u, h, l) for u, h, l in zip(self.up, self.hi, self.lo)]
        self.z = [(v >= 0).double() for v in g]

    def value(self):
        """The Lagrangian at (x*, z*), constraint by constraint."""
        N = self.N
        val = (self.wout * self.x[-1]).sum(1) + self.bout
        for k in range(N.n - 1):
            x, z = self.x[k + 1], self.z[k]
            wx = N.fwd(k, N.W[k], self.x[k])
            hat = wx + N.b[k]
            t = self.a[k] * (hat - x) + self.b0[k] * (x - z * self.uh[k]) + self.b1[k] * (x - hat + (1 - z) * self.lh[k])
            for b in range(self.cuts):
                row = self.masked(b, k, self.x[k], self.x[k], wx)
                t = t + self.s[b][k] * (self.lam[b][k] * (1 - z) - row - N.b[k] * z - self.mu[b][k] * z + x)
            val = val + t.sum(1)
        return val

    def iterate(self, it, opt):
        N = self.N
        act = it - opt.bigm_iters
        t, T = (act, opt.as_iters) if opt.as_iters else (it, opt.bigm_iters)
        l0, l1 = (opt.as_lr0, opt.as_lr1) if opt.as_iters else (opt.bigm_lr0, opt.bigm_lr1)
        lr = l0 + (l1 - l0) * t / max(1, T - 1)

        def adam(th, m, v, g, step):
            m = opt.adam_b1 * m + (1 - opt.adam_b1) * g
            v = opt.adam_b2 * v + (1 - opt.adam_b2) * g * g
            mh, vh = m / (1 - opt.adam_b1 ** step), v / (1 - opt.adam_b2 ** step)
            return (th + lr * mh / (vh.sqrt() + opt.adam_eps)).clamp(min=0), m, v

        self.minimise()
        for k in range(N.n - 1):
            x, z = self.x[k + 1], self.z[k]
            wx = N.fwd(k, N.W[k], self.x[k])
            hat = wx + N.b[k]
            gs = (hat - x, x - z * self.uh[k], x - hat + (1 - z) * self.lh[k])
            for q, (th, g) in enumerate(zip((self.a, self.b0, self.b1), gs)):
                th[k], self.m[2 * q][k], self.m[2 * q + 1][k] = adam(th[k], self.m[2 * q][k], self.m[2 * q + 1][k], g, it + 1)
            for b in range(self.cuts):
                row = self.masked(b, k, self.x[k], self.x[k], wx)
                g = x - row + self.lam[b][k] * (1 - z) - z * (N.b[k] + self.mu[b][k])
                new = adam(self.s[b][k], self.sm[0][b][k], self.sm[1][b][k], g, act - b + 1)
                for box, v in zip((self.s[b], self.sm[0][b], self.sm[1][b]), new):
                    box[k] = torch.where(self.on[b], v, box[k])


class _Saddle64:
    """Saddle Point iterations (Alg. 2) in float64, the oracle masks of eq. (3) formed per weight."""

    def __init__(self, N, C, bounds, d):
        self.N = N
        self.lh, self.uh, self.lo, self.hi = bounds
        self.wout, self.bout = C @ N.W[N.n - 1], C @ N.b[N.n - 1]
        w = N.widths
        cut = lambda key: _cut(d[key].double(), w)  # noqa: E731
        self.a, self.Sb, self.G, self.C, self.z, self.mua, self.mub = map(cut, ("alpha", "Sb", "G", "C", "z", "mua", "mub"))
        self.x, self.P = (list(torch.split(d[k].double(), w, -1)) for k in ("x", "P"))

    def phase_a(self):
        N, self.f = self.N, []
        for k in range(N.n):
            v = -self.wout if k == N.n - 1 else self.P[k] - N.bwd(k, N.W[k], self.a[k])
            self.f.append(v + self.a[k - 1] - self.Sb[k - 1] if k else v)
        self.xbar = [torch.where(v >= 0, h, l) for v, h, l in zip(self.f, self.hi, self.lo)]
        self.zbar = [(g >= 0).double() for g in self.G]

    def value(self):
        self.phase_a()
        val = self.bout - sum((f * x).sum(1) for f, x in zip(self.f, self.xbar))
        for k in range(self.N.n - 1):
            val = val + (self.N.b[k] * self.a[k] + self.C[k] - self.G[k].clamp(min=0)).sum(1)
        return val

    def rows(self, k):
        """The layer's inputs as a matrix per subproblem, [S, K, positions], and its weights [rows, K]."""
        L = self.N.net[k]
        if L["kind"] == "linear":
            return lambda t: t[:, :, None], lambda t: t[:, :, 0], self.N.W[k]
        fold = dict(kernel_size=(L["kh"], L["kw"]), stride=L["stride"], padding=L["pad"])
        return (lambda t: F.unfold(t.view(-1, *L["in_shape"]), **fold),
                lambda t: F.fold(t, L["in_shape"][1:], **fold).flatten(1), self.N.W[k].flatten(1))

    def iterate(self, t):
        N, gamma = self.N, 1.0 / (t + 10)
        mix = lambda old, new: (1 - gamma) * old + gamma * new  # noqa: E731
        self.phase_a()
        S = self.x[0].shape[0]
        for k in range(N.n - 1):
            unfold, fold, W = self.rows(k)
            l, u, x = self.lo[k], self.hi[k], self.x[k]
            free = (u != l).double()
            wide = torch.where(u != l, u - l, 1.0)
            X, Lo, Hi, Fr = map(unfold, (x, l, u, free))
            Tp, Tn = unfold(torch.where(u != l, (x - l) / wide, -1.0)), unfold(torch.where(u != l, (u - x) / wide, -1.0))
            there = unfold(torch.ones_like(x))
            pos = X.shape[2]
            R = W.shape[0]
            grid = lambda v: v.view(S, R, pos)  # noqa: E731
            z, xo, uh, lh, mua, mub = map(grid, (self.z[k], self.x[k + 1], self.uh[k], self.lh[k], self.mua[k], self.mub[k]))
            bias = grid(N.b[k].expand(S, -1))
            back = torch.zeros_like(X)
            new = {key: torch.empty_like(z) for key in ("a", "Sb", "G", "C")}
            for r in range(R):
                w = W[r][None, :, None]
                plus = w > 0
                I = (z[:, r:r + 1] >= torch.where(plus, Tp, Tn)) | (there == 0) | (w == 0)
                wx = w * X
                hat = wx.sum(1) + bias[:, r]
                A = torch.where(I, wx, 0.0).sum(1)
                lam = torch.where(I, w * torch.where(plus, Lo, Hi), 0.0).sum(1)
                mu = torch.where(I, 0.0, w * torch.where(plus, Hi, Lo)).sum(1)
                nout, nfree = (~I).sum(1), ((w != 0) & (Fr > 0)).sum(1)
                zr, xr = z[:, r], xo[:, r]
                v0 = xr - zr * uh[:, r]
                v1 = xr - hat + (1 - zr) * lh[:, r]
                vI = xr - A + (1 - zr) * lam - zr * (bias[:, r] + mu)
                vI = torch.where((nout == 0) | (nout == nfree), -math.inf, vI)
                one = v1 > v0
                best = torch.where(one, v1, v0)
                two = vI > best
                bb = torch.where(torch.where(two, vI, best) >= 0, mub[:, r], 0.0)
                gs = torch.where(two, lam + mu + bias[:, r], torch.where(one, lh[:, r], uh[:, r]))
                cs = torch.where(two, lam, torch.where(one, lh[:, r] - bias[:, r], 0.0))
                new["a"][:, r] = torch.where(hat - xr >= 0, mua[:, r], 0.0)
                new["Sb"][:, r], new["G"][:, r], new["C"][:, r] = bb, bb * gs, bb * cs
                b1, bI = torch.where(one & ~two, bb, 0.0), torch.where(two, bb, 0.0)
                back += w * (b1[:, None] + torch.where(I, bI[:, None], 0.0))
            self.P[k] = mix(self.P[k], fold(back))
            for key, box in (("a", self.a), ("Sb", self.Sb), ("G", self.G), ("C", self.C)):
                box[k] = mix(box[k], new[key].reshape(S, -1))
        self.x_next = [mix(a, b) for a, b in zip(self.x, self.xbar)]
        self.z = [mix(a, b) for a, b in zip(self.z, self.zbar)]
        self.x = self.x_next


def _subset(d, a, c, dims):
    return {k: (v[a:c] if dims.get(k, 0) == 0 else v[:, a:c]) for k, v in d.items()}


def exact(case, seed):
    kind, S = case["kind"], case["S"]
    if kind in ("solve", "intermediate"):
        return None   # whole solves from zero duals: float64 takes other decisions on the way
    net = _net(case["net"])
    nnz, NT, NH, _ = _sizes(net)
    cost = 4.0 * S * nnz * (1 + 2 * case.get("cuts", 0)) * max(1, case.get("iters", 1))
    if kind == "saddle":
        cost *= 8
    if cost > 6e12:
        return None
    gen = _gen(seed)
    lo, hi, C = _boxes(case, seed, gen)
    splits, caps = _splits(case, gen, NH), _caps(case, gen)
    N = _Net64(net)
    lo64, hi64, C64 = lo.double(), hi.double(), C.double()
    step = S if kind == "gradient" else max(1, int((2e7 if kind == "saddle" else 4e7) / (4 * NT)))
    bounds = [N.intervals(lo64[a:a + step], hi64[a:a + step], None if splits is None else splits[a:a + step])
              for a in range(0, S, step)]
    lhat, uhat = (torch.cat([torch.cat(b[q], 1) for b in bounds]) for q in (0, 1))
    if kind == "intervals":
        return {"lhat": lhat, "uhat": uhat}
    opt = _options(case)
    if kind == "saddle":
        plo, phi = (torch.cat([torch.cat(b[q], 1) for b in bounds]) for q in (2, 3))
        d = _saddle_state(case, gen, plo.float(), phi.float(), lhat.float(), uhat.float())
        parts = []
        for q, a in enumerate(range(0, S, step)):
            s = _Saddle64(N, C64[a:a + step], bounds[q], _subset(d, a, a + step, {}))
            for t in range(case["iters"]):
                s.iterate(SADDLE_STARTED + t)
            parts.append([s.value(), torch.cat(s.a, 1), torch.cat(s.x, 1), torch.cat(s.z, 1)])
        return dict(zip(("bound", "alpha", "x", "z"), (torch.cat(p) for p in zip(*parts))))
    d = _duals(dict(case, caps=caps), gen, lhat.float(), uhat.float(), NT)
    if kind == "iterate":
        parts = []
        for q, a in enumerate(range(0, S, step)):
            sub = _subset(d, a, a + step, {"adam": 1, "slot_adam": 1})
            s = _Active64(N, lo64[a:a + step], hi64[a:a + step], C64[a:a + step], bounds[q], sub, case["cuts"],
                          None if caps is None else caps[a:a + step])
            for t in range(case["iters"]):
                s.iterate(STARTED + t, opt)
            s.minimise()
            slots = [torch.stack([torch.cat(v, 1) for v in s.s], 1)] if case["cuts"] else []
            parts.append([s.value(), torch.cat(s.a, 1), torch.cat(s.b0, 1), torch.cat(s.b1, 1)] + slots)
        return dict(zip(("bound", "alpha", "beta0", "beta1", "slot"), (torch.cat(p) for p in zip(*parts))))
    # gradient: the Lagrangian as a function of weights, biases and box at fixed duals, masks, x*'s ends and z*
    weight = torch.rand(S, generator=gen, device="cuda", dtype=torch.float64)
    leaves = [t.clone().requires_grad_(True) for t in (lo64, hi64, *[torch.from_numpy(L[k]).cuda().double() for L in net
                                                                     for k in ("W", "b")])]
    M = _Net64(net, leaves[2:])
    lh, uh, los, his = M.intervals(leaves[0], leaves[1])
    if not case["chain"]:
        lh, uh = [t.detach() for t in lh], [t.detach() for t in uh]
        los, his = ([leaves[q]] + [t.detach() for t in v[1:]] for q, v in ((0, los), (1, his)))
    s = _Active64(M, leaves[0], leaves[1], C64, (lh, uh, los, his), d, case["cuts"])
    s.minimise()
    value = s.value()
    grads = torch.autograd.grad((value * weight).sum(), leaves)
    return {"bound": value.detach(), "grads": list(grads)}
