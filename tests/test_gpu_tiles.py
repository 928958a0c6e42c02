"""The float32 Active Set passes on tiles (csrc/cb_tile.cuh) against the lane teams' walks: the same
subproblems in a large batch (tiles) and in small ones (teams), one iteration from the same drawn state.
Sizes at the edges of tiles: positions that do not fill a tile, planes smaller and larger than one,
stride phases of unequal size, channels that are no multiple of a thread's, wide linear layers whose
taps are split over blocks, every count of slots, additions, caps and the ellipsoid."""
import numpy as np
import pytest

from paper_2101_05844_gb300 import binding, synth

pytestmark = pytest.mark.gpu

NETS = {
    "odd planes": synth._convnet((3, 13, 11), [(5, 3, 1, 1), (9, 3, 2, 1), (12, 4, 3, 2)], [33, 3]),
    "wide": synth._convnet((3, 32, 32), [(16, 4, 2, 1), (32, 4, 2, 1)], [100, 10]),
    "tall kernel": synth._convnet((2, 20, 70), [(10, 5, 2, 0)], [17, 2]),
    "linear": synth._mlp([300, 65, 7, 130, 4]),
    "long linear": synth._mlp([3000, 40, 2]),
}
# float32 sums of n terms in another order: 2^-24 (2 sqrt(n) + 8) of the sum of the terms' magnitudes
# (n <= 3000 here), and an Adam step moves a dual by its gradient's relative error times the step size
RTOL = 2.0 ** -24 * (2 * np.sqrt(3000) + 8) * 8


def _draw(ctx, rng, S, nslots, it, cap):
    NH, NT = ctx.NH, ctx.NT
    lh, uh = (ctx.get_state(w).reshape(S, NH) for w in (binding.ST_LHAT, binding.ST_UHAT))
    w = (0.25 * (uh - lh) + 1e-3).astype(np.float32)
    dual = lambda *s: (rng.random(s) * 0.3 * (rng.random(s) > 0.3)).astype(np.float32)  # noqa: E731
    mom = lambda w: ((rng.standard_normal(w.shape) * w).astype(np.float32),  # noqa: E731
                     ((0.5 + rng.random(w.shape)) * w * w).astype(np.float32))
    d = {binding.ST_ITER: np.array([it, 0, 0], np.int32), binding.ST_BETA0: dual(S, NH), binding.ST_BETA1: dual(S, NH)}
    m = [mom(w) for _ in range(3)]
    d[binding.ST_ADAM] = np.stack([t for p in m for t in p])
    ws = np.repeat(w[:, None], cap, 1)
    ws[:, nslots:] = 0
    d[binding.ST_SLOT_ADAM] = np.stack(mom(ws))
    bits = (1 << nslots) - 1
    d[binding.ST_XSNAP] = (rng.integers(0, 256, (S, NT)) & bits).astype(np.uint8)
    d[binding.ST_ZSNAP] = (rng.integers(0, 256, (S, NH)) & bits).astype(np.uint8)
    sb = dual(S, cap, NH)
    sb[:, nslots:] = 0
    d[binding.ST_SLOT_BETA] = sb
    d[binding.ST_ALPHA] = dual(S, NH)
    return d


def _axis(which):
    return 1 if which in (binding.ST_ADAM, binding.ST_SLOT_ADAM) else 0


CASES = [("odd planes", 700, 0, False, 0), ("odd planes", 701, 3, True, 0), ("odd planes", 699, 8, False, 0),
         ("odd planes", 640, 6, True, 1), ("wide", 40, 5, False, 0), ("wide", 33, 7, True, 0), ("tall kernel", 200, 2, False, 0),
         ("linear", 1500, 4, True, 0), ("linear", 1537, 1, False, 1), ("long linear", 300, 5, False, 0)]


@pytest.mark.parametrize("name,S,nslots,add,ball", CASES)
def test_tiles_agree_with_lane_teams(name, S, nslots, add, ball):
    layers = NETS[name]
    net = synth.make_net(layers, 3)
    work = S * sum(L["W"].size * (L["out_shape"][1] * L["out_shape"][2] if L["kind"] == "conv" else 1) for L in net[:-1])
    assert work >= 3e7, "the batch must be large enough for tiles"
    c, lo, hi = synth.make_boxes(net[0]["n_in"], S, 0.05, 4)
    C = synth.properties_runner_up(synth.forward(net, c))
    cap = nslots + (1 if add else 0) if nslots < 8 else 8
    cap = max(cap, 1)
    rng = np.random.default_rng(5)
    caps = rng.integers(max(1, cap - 2), cap + 1, S).astype(np.int32)
    kw = dict(bigm_iters=10, as_iters=1000, omega=0, vars_per_add=cap, max_cuts=cap, graph_chunk=0, input_l2=ball,
              as_lr0=1e-3, as_lr1=1e-3, sp_init_steps=3)
    it = 10 + nslots if add else 10 + 100 if nslots else 3
    big = binding.Context(net, lo, hi, C, caps=caps, options=binding.default_options(**kw))
    d = _draw(big, rng, S, nslots, it, cap)
    for w, v in d.items():
        big.set_state(w, v)
    big.as_step(1)
    outs = [binding.ST_ALPHA, binding.ST_BETA0, binding.ST_BETA1, binding.ST_SLOT_BETA, binding.ST_ADAM]
    got = {w: big.get_state(w) for w in outs}
    bound = big.bound(64)
    pick = sorted(set([0, 1, S // 2, S - 2, S - 1]))
    one = binding.Context(net, lo[pick], hi[pick], C[pick], caps=caps[pick], options=binding.default_options(**kw))
    n = len(pick)
    for w, v in d.items():
        one.set_state(w, v if w == binding.ST_ITER else np.take(v, pick, _axis(w)))
    # interval bounds: float64-accurate sums in either order, rounded outward to float32
    for w in (binding.ST_LHAT, binding.ST_UHAT):
        a, b = big.get_state(w).reshape(S, -1)[pick], one.get_state(w).reshape(len(pick), -1)
        assert (np.abs(a - b) <= 2.0 ** -22 * np.abs(b) + 1e-9).all(), (name, w)
    one.as_step(1)
    for w in outs:
        shape = d[w].shape
        a = np.take(got[w].reshape(shape), pick, _axis(w))
        b = one.get_state(w).reshape(a.shape)
        scale = np.abs(b).max() + 1e-6
        off = np.abs(a - b)
        # an input whose f lies within rounding of 0 may take the other end of its box in one of the two:
        # at most one in a thousand entries may read such an input
        bad = off > RTOL * (np.abs(b) + scale)
        assert bad.mean() < 1e-3, (name, w, bad.mean(), off.max(), scale)
    ref = one.bound(64)
    np.testing.assert_allclose(bound[pick], ref, rtol=1e-4, atol=1e-4)
    assert n == len(ref)
    # Saddle Point from the same duals: conversion (eq. 10), primal initialisation, then two iterations
    for ctx, part in ((big, None), (one, pick)):
        for w, v in d.items():
            ctx.set_state(w, v if part is None or w == binding.ST_ITER else np.take(v, part, _axis(w)))
    outs = [(binding.ST_SP_STATS, (4, S, big.NT), 1), (binding.ST_SP_X, (S, big.NT), 0), (binding.ST_SP_Z, (S, big.NH), 0),
            (binding.ST_ALPHA, (S, big.NH), 0)]
    # the primal initialisation leaves x and z at ends of their boxes, where beta_0's and the oracle mask's
    # gradients tie exactly (z = 0: A = Lam) and rounding picks one: the iterations start inside the boxes
    for steps in (0, 2):
        big.sp_step(0)
        one.sp_step(0)
        if steps:
            blo, bhi = (big.get_state(w).reshape(S, -1) for w in (binding.ST_LO, binding.ST_HI))
            st = {binding.ST_ITER: np.array([it, 50, 1], np.int32),
                  binding.ST_SP_X: (blo + rng.random(blo.shape, np.float32) * (bhi - blo)).astype(np.float32),
                  binding.ST_SP_Z: rng.random((S, big.NH), np.float32),
                  binding.ST_SP_STATS: big.get_state(binding.ST_SP_STATS).reshape(4, S, big.NT),
                  binding.ST_SP_CAPS: big.get_state(binding.ST_SP_CAPS).reshape(2, S, big.NH),
                  binding.ST_ALPHA: big.get_state(binding.ST_ALPHA).reshape(S, big.NH)}
            for w, v in st.items():
                ax = 1 if w in (binding.ST_SP_STATS, binding.ST_SP_CAPS) else 0
                big.set_state(w, v)
                one.set_state(w, v if w == binding.ST_ITER else np.take(v, pick, ax))
        big.sp_step(steps)
        one.sp_step(steps)
        for w, shape, ax in outs:
            a = np.take(big.get_state(w).reshape(shape), pick, ax)
            b = one.get_state(w).reshape(a.shape)
            off = np.abs(a - b)
            bad = off > RTOL * (np.abs(b) + np.abs(b).max() + 1e-6)
            # a choice (eq. 12) within rounding of a tie may fall the other way
            assert bad.mean() < 2e-3, (name, steps, w, bad.mean(), off.max())


@pytest.mark.parametrize("widths,S,nslots", [((100, 75, 33, 7), 129, 3), ((300, 130, 257, 4), 300, 0), ((520, 40, 64, 3), 41, 5)])
def test_bf16_linear_products_do_not_depend_on_their_tiles(widths, S, nslots):
    """The BF16 form's dense products (TMA, 128, 64 or 32 columns a tile): rows, columns and K that fill no
    tile. The K order of the sums is the tiles' same, so a batch (wide tiles) and each of its subproblems
    alone (narrow ones) agree bit for bit; against the oracle, test_gpu_bf16.py checks small ones."""
    net = synth.make_net(synth._mlp(list(widths)), 7)
    c, lo, hi = synth.make_boxes(widths[0], S, 0.05, 8)
    C = synth.properties_runner_up(synth.forward(net, c))
    cap = max(1, nslots)
    kw = dict(bigm_iters=10, as_iters=1000, omega=0, vars_per_add=cap, max_cuts=cap, graph_chunk=0, precision=16)
    big = binding.Context(net, lo, hi, C, options=binding.default_options(**kw))
    d = _draw(big, np.random.default_rng(9), S, nslots, 110 if nslots else 3, cap)
    outs = [binding.ST_ALPHA, binding.ST_BETA0, binding.ST_BETA1, binding.ST_SLOT_BETA]
    for w, v in d.items():
        big.set_state(w, v)
    big.as_step(2)
    for s in (0, S // 2, S - 1):
        one = binding.Context(net, lo[s:s + 1], hi[s:s + 1], C[s:s + 1], options=binding.default_options(**kw))
        for w, v in d.items():
            one.set_state(w, v if w == binding.ST_ITER else np.take(v, [s], _axis(w)))
        one.as_step(2)
        for w in outs:
            a = np.take(big.get_state(w).reshape(d[w].shape), [s], _axis(w))
            np.testing.assert_array_equal(a.ravel(), one.get_state(w))


@pytest.mark.parametrize("nslots,add,ball", [(0, False, 0), (3, True, 0), (5, False, 1), (8, False, 0)])
def test_bf16_passes_by_fours_equal_one_neuron_per_thread(nslots, add, ball):
    """The BF16 form's passes with four neurons per thread (aligned offsets) against one per thread: the same
    net with one more hidden neuron, of zero weights, has no aligned offsets; everything else is the same sums in
    the same order, which the compiler may contract into fused multiply-adds differently: a few units in the
    last place. Stride 1 and 2, channels that are no multiple of eight, several blocks of positions."""
    layers = synth._convnet((3, 12, 20), [(9, 3, 1, 1), (8, 4, 2, 1)], [24, 3])
    net = synth.make_net(layers, 11)
    S, last = 5, net[-2]["n_out"]
    wide = [dict(L) for L in net]
    wide[-2] = dict(net[-2], n_out=last + 1, W=np.vstack([net[-2]["W"], np.zeros((1, net[-2]["n_in"]), np.float32)]),
                    b=np.append(net[-2]["b"], np.float32(0)))
    wide[-1] = dict(net[-1], n_in=last + 1, W=np.hstack([net[-1]["W"], np.zeros((net[-1]["n_out"], 1), np.float32)]))
    c, lo, hi = synth.make_boxes(net[0]["n_in"], S, 0.05, 12)
    C = synth.properties_runner_up(synth.forward(net, c))
    cap = nslots + (1 if add else 0) or 1
    caps = np.array([cap, max(1, cap - 1), cap, 1, cap], np.int32)
    kw = dict(bigm_iters=10, as_iters=1000, omega=0, vars_per_add=cap, max_cuts=cap, graph_chunk=0, precision=16, input_l2=ball)
    a = binding.Context(net, lo, hi, C, caps=caps, options=binding.default_options(**kw))
    b = binding.Context(wide, lo, hi, C, caps=caps, options=binding.default_options(**kw))
    d = _draw(a, np.random.default_rng(13), S, nslots, 10 + nslots if add else 10 + 100 if nslots else 3, cap)
    for w, v in d.items():
        a.set_state(w, v)
        b.set_state(w, v if w == binding.ST_ITER else np.concatenate([v, np.zeros_like(v[..., :1])], -1))
    a.as_step(2)
    b.as_step(2)
    for w in (binding.ST_ALPHA, binding.ST_BETA0, binding.ST_BETA1, binding.ST_SLOT_BETA, binding.ST_ADAM):
        x = b.get_state(w).reshape(*d[w].shape[:-1], -1)[..., :-1]
        y = a.get_state(w).reshape(d[w].shape)
        bad = np.abs(x - y) > 2.0 ** -20 * (np.abs(x) + np.abs(x).max())
        assert bad.mean() < 1e-3, (w, bad.mean())   # an input within rounding of a tie may move its rows
    np.testing.assert_allclose(a.bound(64), b.bound(64), rtol=1e-6)
