"""Several contexts alive at once, of nets and options whose kernels need different amounts of shared memory:
each works as it does alone, whatever contexts are made after it."""
import numpy as np
import pytest

from paper_2101_05844_gb300 import binding, synth

pytestmark = pytest.mark.gpu

STATE = (binding.ST_ALPHA, binding.ST_BETA0, binding.ST_BETA1, binding.ST_SLOT_BETA)


def _problem(name, S):
    net = synth.make_net(synth.arch(name), 1)
    c, lo, hi = synth.make_boxes(net[0]["n_in"], S, 0.02, 2)
    return net, lo, hi, synth.properties_runner_up(synth.forward(net, c))


def _context(prob, max_cuts, precision=32):
    net, lo, hi, C = prob
    # masks are added from the third iteration on, one an iteration, so that every slot comes into use
    return binding.Context(net, lo, hi, C, options=binding.default_options(
        bigm_iters=2, as_iters=50, omega=0, vars_per_add=max(1, max_cuts), max_cuts=max_cuts, graph_chunk=4,
        precision=precision, sp_init_steps=2))


def _use(ctx, prob, sp):
    """A batch's whole course: interval bounds, Big-M and Active Set iterations, bound, gradient, Saddle Point."""
    import torch
    net, lo, hi, C = prob
    ctx.reset(lo, hi, C)
    out = [ctx.get_state(binding.ST_LHAT)]
    ctx.as_step(12)
    out += [ctx.get_state(w) for w in STATE] + [ctx.bound(64)]
    dlo, dhi = (torch.zeros(lo.shape, device="cuda") for _ in range(2))
    ctx.backward(np.ones(len(lo)), None, None, dlo, dhi)
    out += [dlo.cpu().numpy(), dhi.cpu().numpy()]
    if sp:
        ctx.sp_step(2)
        out += [ctx.get_state(binding.ST_SP_X), ctx.bound(64)]
    return out


# the contexts in the order they are made: (net, subproblems, max_cuts, precision); the smallest needs last
GROUPS = {
    "wide conv": [("wide_conv", 256, 8, 32), ("wide_conv", 256, 3, 32), ("wide_conv", 256, 5, 32), ("wide_conv", 256, 7, 32)],
    "other nets": [("conv4", 8, 3, 32), ("mlp_784_1024x3_10", 64, 3, 32), ("wide_conv", 64, 7, 32), ("mlp_300_65_3", 2000, 0, 32)],
    "bf16 form": [("mlp_30_21_13_5", 20, 8, 16), ("mlp_30_21_13_5", 20, 1, 16)],   # (offsets that the passes by fours refuse)
}


@pytest.mark.parametrize("group", list(GROUPS))
def test_contexts_of_other_sizes_do_not_disturb_each_other(group):
    probs = [_problem(name, S) for name, S, _, _ in GROUPS[group]]
    alone = []
    for (_, _, cuts, prec), p in zip(GROUPS[group], probs):
        ctx = _context(p, cuts, prec)
        alone.append(_use(ctx, p, prec == 32))
        ctx.close()
    ctxs = [_context(p, cuts, prec) for (_, _, cuts, prec), p in zip(GROUPS[group], probs)]
    for turn in range(2):
        for ctx, p, ref, (_, _, _, prec) in zip(ctxs, probs, alone, GROUPS[group]):
            for got, want in zip(_use(ctx, p, prec == 32), ref):
                np.testing.assert_array_equal(got, want)


def test_intermediate_bounds_leave_a_live_context_working():
    prob = _problem("wide_conv", 64)
    ctx = _context(prob, 8)
    ref = _use(ctx, prob, True)
    mlp = _problem("mlp_300_65_40_3", 20)
    binding.intermediate_bounds(mlp[0], mlp[1], mlp[2], options=binding.default_options(bigm_iters=2, as_iters=3, max_cuts=1))
    for got, want in zip(_use(ctx, prob, True), ref):
        np.testing.assert_array_equal(got, want)


def test_branch_and_bound_with_its_default_options():
    """as_bab's own contexts (max_cuts 3 and 7, batches of 256) on the Wide conv net: the search runs to its
    limit, and its bracket holds the network's values at sampled points."""
    net, lo, hi, C = _problem("wide_conv", 1)
    res = binding.bab(net, lo[0], hi[0], C[0], binding.bab_default_options(max_domains=6))
    rng = synth.SplitMix64(5)
    x = lo + rng.uniform(500 * lo.size).reshape(500, lo.size) * (hi - lo)
    vals = synth.forward(net, x) @ C[0]
    assert res["bounded"] >= 2
    assert np.isfinite(res["lower"]) and res["lower"] <= vals.min() + 1e-5 and res["lower"] <= res["upper"]


@pytest.mark.parametrize("name,S,sparse,precision", [("mlp_300_200_200_3", 600, True, 32), ("mlp_32_24_22_18_3", 6, False, 16)])
def test_a_pass_of_two_kernels_counts_once_per_iteration(name, S, sparse, precision):
    """Kernel times of a net whose layers are shared between two kernels: tiles and lane teams (a layer of mostly
    zero weights), or four neurons and one neuron a thread (offsets of some layers only are multiples of four)."""
    net, lo, hi, C = _problem(name, S)
    if sparse:
        W = net[1]["W"]
        W[np.random.default_rng(3).random(W.shape) < 0.9] = 0
    ctx = binding.Context(net, lo, hi, C, options=binding.default_options(profile=1, max_cuts=2, bigm_iters=3, as_iters=20,
                                                                         precision=precision))
    t0, l0 = ctx.kernel_times(), ctx.launch_count()
    ctx.as_step(8)
    t1, launches = ctx.kernel_times(), ctx.launch_count() - l0
    count = {k: t1[k][1] - t0[k][1] for k in t1}
    assert count["as_colA"] == count["as_rowB"] == count["counter"] == 8
    assert t1["as_colA"][0] > 0 and t1["as_rowB"][0] > 0
    # two kernels a pass, and the other kernels one launch per count
    assert launches == sum(count.values()) + 2 * 8


def test_autotune_leaves_passes_on_tiles_alone():
    """Team-size targets mean nothing to a pass whose layers are all on tiles: none is timed there, and the
    default stays; a net with a layer of mostly zero weights has targets to time."""
    net, lo, hi, C = _problem("mlp_300_200_200_3", 600)
    make = lambda tune: binding.Context(net, lo, hi, C, options=binding.default_options(  # noqa: E731
        bigm_iters=3, as_iters=20, autotune=tune))
    plain, tuned = make(0), make(1)
    assert tuned.team_targets() == plain.team_targets() == (40000, 40000)
    assert tuned.launch_count() <= 2 * plain.launch_count()   # set-up only, no timed iterations
    W = net[1]["W"]
    W[np.random.default_rng(3).random(W.shape) < 0.9] = 0
    assert make(1).launch_count() > 2 * plain.launch_count()
