"""The tiled walks (csrc/cb_tile.cuh) against the oracle, where their staging can go wrong: batches of a few
distinct subproblems repeated until the layers take tiles. Copies of a subproblem walk the same taps in the
same order wherever in a tile they lie, so they have to agree bit for bit; the first of each is compared with
the oracle, with the tolerances of tests/test_gpu_parity.py."""
import numpy as np
import pytest

from oracle import dual as du
from oracle import envelope as ev
from oracle import network as nw
from paper_2101_05844_gb300 import binding, synth
from tests.lockstep import check_active_set_step
from tests.state_helpers import draw_state, hidden_concat, oracle_bounds_f32, split_hidden
from tests.test_gpu_parity import _draw_sp_state, _install_sp_state

pytestmark = pytest.mark.gpu

DISTINCT = 7   # no divisor of a tile's 32 to 256 subproblems

# Conv layers whose window is one record: a 1x1 kernel on a plane of one position, a kernel that covers its
# plane (each stride phase of the col pass has one record), a stride that leaves one row of a taller plane
ONE_RECORD = {
    "1x1 plane": (synth._convnet((32, 1, 1), [(96, 1, 1, 0), (40, 1, 1, 0)], [24, 3]), 4103),
    "2x2 to 1x1": (synth._convnet((16, 2, 2), [(24, 2, 2, 0), (20, 1, 1, 0)], [65, 3]), 9101),
    "2x1 plane": (synth._convnet((20, 2, 1), [(12, 1, 2, 0)], [65, 40, 3]), 8401),
}


def _spread(a, S, axis):
    """Array a of the distinct subproblems, repeated along `axis` to S."""
    return np.take(a, np.arange(S) % DISTINCT, axis)


def _firsts(a, axis=0):
    """The distinct subproblems' part of a batch array whose copies are equal bit for bit."""
    first = np.take(a, np.arange(DISTINCT), axis)
    np.testing.assert_array_equal(a, _spread(first, a.shape[axis], axis))
    return first


@pytest.mark.parametrize("cap", [3, 5])
@pytest.mark.parametrize("name", list(ONE_RECORD))
def test_windows_of_one_record(name, cap):
    _check_against_oracle(*ONE_RECORD[name], cap, it=8, nslots=2)


# Planes larger and smaller than a tile, stride phases of unequal size, channels that are no multiple of a thread's,
# stride 3, narrow and odd linear layers
GENERAL = {
    "odd planes": (synth._convnet((3, 13, 11), [(5, 3, 1, 1), (9, 3, 2, 1), (12, 4, 3, 2)], [33, 3]), 701),
    "tall kernel": (synth._convnet((2, 9, 40), [(10, 5, 2, 0)], [17, 2]), 900),
    "linear": (synth._mlp([300, 65, 7, 130, 4]), 1537),
}


@pytest.mark.parametrize("cap,it,nslots", [(3, 8, 2), (8, 14, 6)])
@pytest.mark.parametrize("name", list(GENERAL))
def test_tiles_against_the_oracle(name, cap, it, nslots):
    _check_against_oracle(*GENERAL[name], cap, it, nslots)


def _check_against_oracle(layers, S, cap, it, nslots):
    """Interval bounds, the gradient and an iteration of Active Set (global iteration `it`, which adds slot nslots),
    and an iteration of Saddle Point, from drawn states."""
    import torch
    net = synth.make_net(layers, 3)
    work = S * sum(L["W"].size * (L["out_shape"][1] * L["out_shape"][2] if L["kind"] == "conv" else 1) for L in net[:-1])
    assert work >= 3e7, "the batch must be large enough for tiles"
    c, lo, hi = synth.make_boxes(net[0]["n_in"], DISTINCT, 0.1, 4)
    C = synth.properties_runner_up(synth.forward(net, c))
    dense = nw.dense_layers(net)
    prob = dict(net=net, lo=lo, hi=hi, C=C)
    Ps = nw.problems(prob, dense=dense)
    rep = lambda a, axis=0: _spread(a, S, axis)  # noqa: E731

    # interval propagation
    kw = dict(bigm_iters=5, as_iters=40, omega=3, max_cuts=cap)
    opt = binding.default_options(graph_chunk=0, **kw)
    big = binding.Context(net, rep(lo), rep(hi), rep(C), options=opt)
    hidden = lambda w, dt=np.float32: big.get_state(w, dt).reshape(S, -1)  # noqa: E731
    lh, uh = _firsts(hidden(binding.ST_LHAT)), _firsts(hidden(binding.ST_UHAT))
    for s, P in enumerate(Ps):
        rl, ru = hidden_concat(P.lhat), hidden_concat(P.uhat)
        assert (lh[s] <= rl + 1e-9 * (1 + np.abs(rl))).all() and (uh[s] >= ru - 1e-9 * (1 + np.abs(ru))).all()
        assert (np.abs(lh[s] - rl) <= 4e-6 * (1 + np.abs(rl))).all()
        assert (np.abs(uh[s] - ru) <= 4e-6 * (1 + np.abs(ru))).all()

    # an Active Set iteration from a drawn state, and the gradient there
    lh, uh = oracle_bounds_f32(Ps)
    Ps = nw.problems(prob, bounds=[(split_hidden(lh[s].astype(np.float64), Ps[0].widths)[1:],
                                    split_hidden(uh[s].astype(np.float64), Ps[0].widths)[1:])
                                   for s in range(DISTINCT)], dense=dense)
    big.reset(rep(lo), rep(hi), rep(C), rep(lh), rep(uh))
    few = binding.Context(net, lo, hi, C, lh, uh, options=opt)
    solvers = draw_state(Ps, few, kw, it, nslots, seed=31)
    shapes = {binding.ST_ALPHA: ((DISTINCT, -1), 0), binding.ST_BETA0: ((DISTINCT, -1), 0),
              binding.ST_BETA1: ((DISTINCT, -1), 0), binding.ST_ADAM: ((6, DISTINCT, -1), 1),
              binding.ST_SLOT_ADAM: ((2, DISTINCT, -1), 1), binding.ST_XSNAP: ((DISTINCT, -1), 0),
              binding.ST_ZSNAP: ((DISTINCT, -1), 0), binding.ST_SLOT_BETA: ((DISTINCT, -1), 0)}
    big.set_state(binding.ST_ITER, few.get_state(binding.ST_ITER, np.int32))
    for w, (shape, axis) in shapes.items():
        dt = np.uint8 if w in (binding.ST_XSNAP, binding.ST_ZSNAP) else np.float32
        big.set_state(w, rep(few.get_state(w, dt).reshape(shape), axis))
    n0 = lo.shape[1]
    dlo, dhi = (torch.zeros((S, n0), device="cuda") for _ in range(2))
    dW = [torch.zeros(L["W"].shape, device="cuda") for L in net]
    big.backward(np.ones(S), dW, None, dlo, dhi)
    dlo, dhi = _firsts(dlo.cpu().numpy()), _firsts(dhi.cpu().numpy())
    bound = _firsts(big.bound(64))
    refW = [np.zeros(L["W"].shape) for L in net]
    for s, sv in enumerate(solvers):
        g = ev.envelope_gradient(sv.P, sv.st)
        assert bound[s] == pytest.approx(g["value"], abs=1e-4, rel=1e-5)
        decided = np.abs(du.evaluate(sv.P, sv.st)[1][0]) > 1e-5   # x_0* of the others may be at either end
        for got, ref in ((dlo[s], g["dlo0"]), (dhi[s], g["dhi0"])):
            np.testing.assert_allclose(got[decided], ref[decided], rtol=1e-4, atol=1e-4 * np.abs(ref).max())
        copies = len(range(s, S, DISTINCT))
        for k, L in enumerate(net[:-1], start=1):
            w = g["dW"][k]
            refW[k - 1] += copies * (w if L["kind"] == "linear" else ev.filter_gradient(w, sv.P.taps[k], L["W"].shape))
        refW[-1] += copies * np.outer(C[s], g["dW"][sv.P.n][0])
    for got, ref in zip(dW, refW):
        np.testing.assert_allclose(got.cpu().numpy(), ref, rtol=1e-4, atol=1e-4 * np.abs(ref).max())
    big.as_step(1)
    al, b0, b1 = (_firsts(hidden(w)) for w in (binding.ST_ALPHA, binding.ST_BETA0, binding.ST_BETA1))
    sb = _firsts(hidden(binding.ST_SLOT_BETA)).reshape(DISTINCT, big.cap, -1)
    xstar = _firsts(hidden(binding.ST_XSTAR))
    for s, sv in enumerate(solvers):
        check_active_set_step(sv, dict(alpha=al[s], beta0=b0[s], beta1=b1[s], slots=sb[s], xstar=xstar[s]))

    # a Saddle Point iteration from a drawn iterate
    sps, st = _draw_sp_state(Ps, 50, 4)
    _install_sp_state(big, dict(x=rep(st["x"]), z=rep(st["z"]), stats=rep(st["stats"], 1), caps=rep(st["caps"], 1),
                                alpha=rep(st["alpha"])), 4)
    value = _firsts(big.bound())
    big.sp_step(1)
    sel, x, z = _firsts(hidden(binding.ST_SP_SEL, np.uint8)), _firsts(hidden(binding.ST_SP_X)), _firsts(hidden(binding.ST_SP_Z))
    al = _firsts(hidden(binding.ST_ALPHA))
    stats = _firsts(big.get_state(binding.ST_SP_STATS).reshape(4, S, -1), 1)
    tol = dict(rtol=1e-5, atol=1e-6)
    for s, sp in enumerate(sps):
        assert value[s] == pytest.approx(sp.evaluate()[0], abs=1e-5, rel=1e-5)
        sp.step(1)
        np.testing.assert_array_equal(sel[s], hidden_concat(sp.last_sel).astype(np.uint8))
        np.testing.assert_allclose(x[s], np.concatenate(sp.x), **tol)
        np.testing.assert_allclose(z[s], hidden_concat(sp.z), **tol)
        np.testing.assert_allclose(al[s], hidden_concat(sp.alpha), **tol)
        for q, ref in enumerate((sp.Sb, sp.G, sp.C)):
            np.testing.assert_allclose(stats[q, s, n0:], hidden_concat(ref), **tol)
        np.testing.assert_allclose(stats[3, s, :-big.widths[-1]],
                                   np.concatenate([sp.Pst[k] for k in range(1, sp.P.n)]), **tol)


# layers, hidden rows: taps per row that make a lane of the warp walk take one to 256 terms of it
ROWS = {
    "conv 27 taps": (synth._convnet((3, 3, 3), [(1024, 3, 1, 0)], [3]), 1200),
    "conv 576 taps": (synth._convnet((64, 3, 3), [(256, 3, 1, 0)], [3]), 256),
    "linear 100": (synth._mlp([100, 512, 3]), 640),
    "linear 784": (synth._mlp([784, 256, 3]), 160),
    "linear 8192 (split)": (synth._mlp([8192, 64, 3]), 64),
}


@pytest.mark.parametrize("name", list(ROWS))
def test_interval_sums_lose_no_accuracy_on_tiles(name):
    """Rows whose terms cancel exactly over a point box, so that the interval's ends are the rounding error of the
    row's sum and nothing else. Root mean square over at least 4096 rows, against the walk by a warp per row
    that small batches take: no larger but for the sampling error of the two (4 standard deviations of their
    ratio, at a kurtosis of 6: 10%)."""
    layers, S = ROWS[name]
    net = synth.make_net(layers, 5)
    L = net[0]
    n, m = L["n_in"], L["n_out"]
    h = n // 2
    rng = np.random.default_rng(6)
    order = rng.permutation(n)
    W = L["W"].reshape(m, n)
    x = rng.random((S, n), np.float32) + np.float32(0.1)
    W[:, order[h:2 * h]], x[:, order[h:2 * h]] = -W[:, order[:h]], x[:, order[:h]]
    W[:, order[2 * h:]] = 0
    L["b"][:] = 0
    assert S * W.size >= 3e7
    opt = binding.default_options(max_cuts=1)
    C = np.tile(np.float32([1, -1, 0]), (S, 1))
    bounds = lambda part: [binding.Context(net, x[part], x[part], C[part], options=opt).get_state(w)  # noqa: E731
                           for w in (binding.ST_LHAT, binding.ST_UHAT)]
    step = max(1, int(2.9e7 // W.size))
    starts = range(0, min(S, -(-4096 // m)), step)
    N = starts[-1] + step if starts[-1] + step < S else S
    tiles = [a.reshape(S, m)[:N] for a in bounds(slice(0, S))]
    lanes = [np.concatenate(p).reshape(N, m) for p in zip(*[bounds(slice(q, min(q + step, N))) for q in starts])]
    mag = np.abs(x[:N].astype(np.float64)) @ np.abs(W.astype(np.float64)).T
    rms = lambda b: np.sqrt(np.mean(((b[0].astype(np.float64) + b[1]) / 2 / mag) ** 2))  # noqa: E731
    assert N * m >= 4096
    # nothing but rounding: both ends are one float32 apart
    for lh, uh in (tiles, lanes):
        assert (np.abs(lh) <= 1e-13 * mag).all() and (uh >= lh).all()
    assert rms(tiles) <= 1.10 * rms(lanes), (rms(tiles), rms(lanes))
