"""Forms of a launch that compute the same thing, compared at the sizes where
the forms change or a tile is ragged."""
import dataclasses
import threading

import numpy as np
import pytest
import torch

import oracle
import paper_2304_11399_gb300 as tt
from gpu_util import dev, random_theta, synth, to_dev, configs

pytestmark = pytest.mark.gpu

BOUNDS = {1: (configs.CRS_LO, configs.CRS_HI), 2: (configs.FO_LO, configs.FO_HI)}


def _problem(n_dom, sizes, n_tr, ns, op=1, w=5, own_groups=False, seed=0):
    """n_dom domains over len(sizes) groups of the given aperture sizes;
    own_groups: the same domains, each with a group (a copy) of its own."""
    rng = np.random.default_rng(seed)
    lists = [rng.integers(0, n_tr, n).astype(np.int32) for n in sizes]
    grp = np.sort(rng.integers(0, len(sizes), n_dom))
    it0 = rng.integers(0, ns, n_dom).astype(np.int32)
    m0 = rng.uniform(0, 100, len(sizes)).astype(np.float32)
    if own_groups:
        lists, m0, grp = [lists[g] for g in grp], m0[grp], np.arange(n_dom)
    G = len(lists)
    return synth.Problem(op=op, half_window=w, group_m0=m0,
                         group_dt=np.full(G, 0.004, np.float32),
                         ap_ptr=np.concatenate([[0], np.cumsum([x.size for x in lists])]).astype(np.int32),
                         ap_idx=np.concatenate(lists + [np.zeros(0, np.int32)]).astype(np.int32),
                         dom_it0=it0, dom_group=grp.astype(np.int32),
                         group_h0=np.full(G, 400.0, np.float32) if op == 2 else None)


def _line(n_tr, ns, seed=1):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal((n_tr, ns)).astype(np.float32),
            rng.uniform(0, 100, n_tr).astype(np.float32),
            rng.uniform(0, 900, n_tr).astype(np.float32))


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("ns", [300, 2200])  # direct and moveout positions
@pytest.mark.parametrize("n_dom,sizes", [
    (31, (1,)), (32, (31, 33)), (33, (0, 32)), (700, (64, 7, 100)), (80001, (40,))])
def test_stack_lane_and_warp_per_domain_bit_identical(n_dom, sizes, ns, storage):
    """Lane-per-domain form (domains that share apertures; one sum per warp,
    and eight from about 78,000 domains on) against the warp-per-domain form
    (the same domains with apertures of their own)."""
    x, mid, off = _line(50, ns)
    th = to_dev(random_theta(n_dom, 1, *BOUNDS[1], 3)[:, 0])
    outs = []
    for own in (False, True):
        ctx = tt.tt_ctx_create(x, mid, off, _problem(n_dom, sizes, 50, ns, own_groups=own), None,
                               storage=storage, device=dev())
        outs.append(tt.tt_stack(ctx, th))
        ctx.close()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("op,w,storage,ns,sizes", [
    (1, 5, "f32", 300, (100,)), (1, 0, "f32", 2200, (57, 143)), (2, 8, "bf16", 300, (99, 101)),
    (1, 3, "bf16", 300, (300, 1, 0, 99))])
def test_slices_walked_by_one_warp_or_eight(op, w, storage, ns, sizes):
    """A launch of 160 units and one of 176 cut apertures into the same 56
    slices, the first with a warp per slice, the second (mean aperture under
    0.6 per unit) with a warp per eight: the members they share have the same
    S bit for bit. 300 entries are more than 56 chunks of 32 would hold
    per slice of one entry; 57 to 143 leave slices of one to three, 1 and 0
    leave most or all empty."""
    n_dom = 1024
    x, mid, off = _line(60, ns)
    prob = _problem(n_dom, sizes, 60, ns, op, w)
    th = to_dev(random_theta(n_dom, 11, *BOUNDS[op], 7))
    ctx = tt.tt_ctx_create(x, mid, off, prob, None, storage=storage, device=dev())
    if tt.tt_ctx_get_option(ctx, "sm_count") != 152:
        pytest.skip("launch sizes chosen for 152 multiprocessors")
    a = tt.tt_semblance_eval(ctx, th[:, :10].contiguous())
    b = tt.tt_semblance_eval(ctx, th)
    ctx.close()
    assert torch.equal(a, b[:, :10])
    if storage == "f32":
        ref = oracle.semblance.semblance_many(x, mid, off, prob, th[:, :2].cpu().numpy())
        assert np.max(np.abs(a[:, :2].cpu().numpy() - ref)) <= 1e-5


@pytest.mark.parametrize("n_dom,P,sizes,op,w,storage,ns", [
    (1, 1, (16,), 1, 5, "f32", 300), (63, 1, (64, 40), 1, 0, "f32", 300),
    (65, 1, (300,), 2, 8, "f32", 300), (130, 3, (300, 17), 1, 8, "bf16", 300),
    (500, 1, (257,), 1, 5, "f32", 2200), (40, 2, (70, 1, 33), 2, 1, "bf16", 2200),
    (9000, 1, (300, 280), 1, 3, "f32", 300), (25000, 1, (60,), 1, 5, "bf16", 300)])
def test_split_gradient(n_dom, P, sizes, op, w, storage, ns):
    """The split gradient (clusters of 9, 7 and 2 blocks) against the unsplit one.
    Both sum the same n = N (2w + 1) FP32 terms in different orders: S to
    1e-6, as elsewhere between two orders. A gradient's terms cancel to about
    1/sqrt(n) of their sum of magnitudes, so an error of at most n 2^-24 of
    that sum is n^1.5 2^-24 of a typical gradient: 2.2e-2 for the longest
    windows here (n = 5100), and 1/sqrt(n) of that, 3e-4, when roundings are
    random; 1e-3 of |G| plus the median magnitude is asked."""
    x, mid, off = _line(60, ns)
    prob = _problem(n_dom, sizes, 60, ns, op, w)
    th = to_dev(random_theta(n_dom, P, *BOUNDS[op], 5))
    ctx = tt.tt_ctx_create(x, mid, off, prob, None, storage=storage, device=dev())
    S, G = tt.tt_semblance_grad(ctx, th)
    again = tt.tt_semblance_grad(ctx, th)
    assert torch.equal(S, tt.tt_semblance_eval(ctx, th))  # the forward's slices and order
    tt.tt_ctx_set_option(ctx, "split", False)
    S0, G0 = tt.tt_semblance_grad(ctx, th)
    ctx.close()
    assert torch.equal(S, again[0]) and torch.equal(G, again[1])
    assert (S - S0).abs().max().item() <= 1e-6
    scale = G0.abs().flatten(0, 1).median(0).values
    assert ((G - G0).abs() <= 1e-3 * (G0.abs() + scale)).all()
    if storage == "f32":
        rS, _ = oracle.semblance.semblance_grad_many(x, mid, off, prob, th.cpu().numpy()) \
            if n_dom <= 500 else (None, None)
        assert rS is None or np.max(np.abs(S.cpu().numpy() - rS)) <= 1e-5


def test_split_gradient_of_one_block():
    """12 units per SM and one pair more: a unit's aperture in one block (B = 1),
    against the unsplit form, with the bounds of test_split_gradient (n = 900)."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    n_dom = 12 * n_sm * 64 + 1
    x, mid, off = _line(60, 300)
    ctx = tt.tt_ctx_create(x, mid, off, _problem(n_dom, (300,), 60, 300, w=1), None,
                           device=dev())
    th = to_dev(random_theta(n_dom, 1, *BOUNDS[1], 5))
    S, G = tt.tt_semblance_grad(ctx, th)
    assert torch.equal(S, tt.tt_semblance_eval(ctx, th))
    tt.tt_ctx_set_option(ctx, "split", False)
    S0, G0 = tt.tt_semblance_grad(ctx, th)
    ctx.close()
    assert (S - S0).abs().max().item() <= 1e-6
    scale = G0.abs().flatten(0, 1).median(0).values
    assert ((G - G0).abs() <= 1e-3 * (G0.abs() + scale)).all()


def _cfg(op, np_, ng, **kw):
    kw = {"exch_every": 0, "polish_steps": 0, "polish_lr": 2e-4, "adapt": 0, **kw}
    lo, hi = BOUNDS[op]
    return configs.DEConfig(np=np_, ng=ng, F=0.5, CR=0.9, seed=11, lo=lo, hi=hi, **kw)


@pytest.mark.parametrize("n_dom,np_,ng,op,w,storage,ns,sizes,kw", [
    (1, 4, 3, 1, 5, "f32", 300, (40,), {}), (37, 64, 0, 1, 5, "f32", 300, (40, 57), {}),
    (65, 37, 5, 2, 8, "bf16", 300, (70, 0, 33), {"adapt": 1}),
    (300, 13, 7, 1, 0, "f32", 2200, (150,), {"adapt": 1}),
    (297, 64, 4, 1, 5, "bf16", 300, (56, 1, 120), {}),
    (600, 30, 9, 1, 5, "f32", 300, (60, 20), {"grid": (20, 30), "exch_every": 3, "polish_steps": 2}),
    (60, 9, 8, 1, 2, "f32", 300, (30,), {"grid": (6, 10), "exch_every": 5, "adapt": 1})])
def test_fused_search_equals_stepwise(n_dom, np_, ng, op, w, storage, ns, sizes, kw):
    """All generations between exchanges in one launch against one launch per
    step (what a search runs while its launches are timed): the same bits."""
    kw = dict(kw)
    grid = kw.pop("grid", None)
    x, mid, off = _line(60, ns)
    prob = _problem(n_dom, sizes, 60, ns, op, w)
    if grid:
        prob.n_m0, prob.n_t0 = grid
    ctx = tt.tt_ctx_create(x, mid, off, prob, _cfg(op, np_, ng, **kw), storage=storage,
                           device=dev())
    th, S, n = tt.tt_search(ctx)
    tt.tt_ctx_set_option(ctx, "search_graph", False)
    tt.tt_ctx_stats(ctx, reset=True)
    th1, S1, n1 = tt.tt_search(ctx)
    few = tt.tt_ctx_stats(ctx, reset=True)
    tt.tt_ctx_profile(ctx, True)
    th2, S2, n2 = tt.tt_search(ctx)
    many = tt.tt_ctx_stats(ctx)
    ctx.close()
    assert torch.equal(th, th2) and torch.equal(S, S2) and n == n2
    assert torch.equal(th, th1) and torch.equal(S, S1) and n == n1
    assert few["launches"] < many["launches"] or ng == 0
    assert few["trace_evals"] == many["trace_evals"]
    assert few["semblance_launches"] == many["semblance_launches"]


@pytest.mark.parametrize("storage,w", [("f32", 5), ("f32", 6), ("bf16", 5)])
def test_two_contexts_on_two_threads(storage, w):
    """Launches of the same kernels with different amounts of shared memory, a
    context and a stream per host thread: evaluations of 8 and of 80 units
    (clusters of 9 and of 7 blocks) and searches of them (9 and 7 warps). A limit
    that one thread lowers would refuse the other's launch."""
    x, mid, off = _line(60, 300)
    errors, start = [], threading.Barrier(2, timeout=60)

    def run(n_dom):
        try:
            s = torch.cuda.Stream(device=dev())
            with torch.cuda.stream(s):
                prob = _problem(n_dom, (100,), 60, 300, w=w)
                ctx = tt.tt_ctx_create(x, mid, off, prob, _cfg(1, 64, 2), storage=storage,
                                       device=dev())
                tt.tt_ctx_set_option(ctx, "search_graph", False)
                th = to_dev(random_theta(n_dom, 64, *BOUNDS[1], 7))
                S = tt.tt_semblance_eval(ctx, th)
                best = tt.tt_search(ctx)[1]
                start.wait()
                for _ in range(500):
                    S1 = tt.tt_semblance_eval(ctx, th)
                    best1 = tt.tt_search(ctx)[1]
                assert torch.equal(S, S1) and torch.equal(best, best1)
                s.synchronize()
                ctx.close()
        except BaseException as e:  # reported by the main thread
            errors.append(e)
            start.abort()

    threads = [threading.Thread(target=run, args=(n,)) for n in (8, 80)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


@pytest.mark.parametrize("n_dom,P,sizes,op,w,ns", [
    (300, 1, (200,), 0, 5, 300), (300, 1, (300,), 1, 3, 300), (9000, 1, (300,), 2, 5, 2200)])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("bad", [float("inf"), 1e25, float("nan")])
def test_gradient_of_infinite_energy(n_dom, P, sizes, op, w, ns, storage, bad):
    """Windows with an infinite energy (an infinite sample, or 1e25, whose square
    is) have S = dS = NaN in the split gradient as in the unsplit one; with a NaN
    energy both are 0. BF16 storage sums the split form's energy in FP64, where
    1e25 squared is finite: not compared."""
    if storage == "bf16" and bad == 1e25:
        pytest.skip("finite in the split form's FP64 energy")
    x, mid, off = _line(60, ns)
    off[7] = 5.0  # an early window of every aperture that holds trace 7
    x[7, 40:60] = bad
    prob = _problem(n_dom, sizes, 60, ns, op, w)
    bounds = BOUNDS[op] if op else ((1 / 4500 ** 2,), (1 / 1400 ** 2,))
    th = to_dev(random_theta(n_dom, P, *bounds, 5))
    ctx = tt.tt_ctx_create(x, mid, off, prob, None, storage=storage, device=dev())
    out = []
    for split in (True, False):
        tt.tt_ctx_set_option(ctx, "split", split)
        out.append(tt.tt_semblance_grad(ctx, th))
        assert torch.equal(out[-1][0].isnan(), tt.tt_semblance_eval(ctx, th).isnan())
    ctx.close()
    (S, G), (S0, G0) = out
    assert torch.equal(S.isnan(), S0.isnan()) and torch.equal(G.isnan(), G0.isnan())
    assert torch.equal(S == 0, S0 == 0) and torch.equal((G == 0).all(-1), (G0 == 0).all(-1))
    if bad == bad:
        assert S.isnan().any() and G[S.isnan()].isnan().all()
    else:
        assert (S == 0).any() and not S.isnan().any() and not G.isnan().any()


@pytest.mark.parametrize("n_dom,P,sizes,op,w,storage,ns,split,launches,same", [
    (60, 2, (48,), 1, 5, "f32", 300, True, 1, True),          # the adjoint at once
    (19000, 1, (150, 140), 1, 5, "f32", 2200, True, 1, True),
    (4001, 1, (6000, 5900), 1, 5, "f32", 300, True, 2, True),  # sums, through scratch
    (3800, 1, (3000, 2990), 2, 8, "bf16", 300, True, 2, True),  # of clusters of 9
    (19456, 1, (900, 880), 1, 5, "f32", 2200, True, 2, True),  # of clusters of 7
    (19000, 3, (370, 0), 1, 3, "bf16", 300, True, 2, True),   # of clusters of 2
    (150001, 1, (130,), 1, 5, "f32", 300, True, 2, True),     # of one block
    (170000, 1, (60, 60), 1, 5, "bf16", 300, True, 2, False),  # K2 does not split
    (117001, 1, (300,), 1, 1, "f32", 300, True, 2, True),
    (300000, 1, (8,), 1, 5, "f32", 300, True, 2, True),       # too short: two launches
    (312000, 1, (20,), 1, 5, "f32", 300, True, 2, True),      # too many pairs to split
    (4001, 1, (600,), 1, 5, "f32", 300, False, 2, True)])
def test_autograd_value_and_gradient(n_dom, P, sizes, op, w, storage, ns, split, launches, same):
    """A differentiated call's value is tt_semblance_eval's bit for bit and costs
    one launch while no backward comes; its gradient is tt_semblance_grad's bit for
    bit wherever both split or neither does, and one of the same terms added in
    another order elsewhere (the bound of test_split_gradient). A backward after a
    reload is taken on the new traces."""
    x, mid, off = _line(60, ns)
    prob = _problem(n_dom, sizes, 60, ns, op, w)
    ctx = tt.tt_ctx_create(x, mid, off, prob, None, storage=storage, device=dev())
    tt.tt_ctx_set_option(ctx, "split", split)
    th = to_dev(random_theta(n_dom, P, *BOUNDS[op], 5)).requires_grad_()
    gS = torch.rand((n_dom, P), device=dev())
    E = tt.tt_semblance_eval(ctx, th.detach())
    tt.tt_ctx_stats(ctx, reset=True)
    S = tt.semblance(ctx, th)
    assert tt.tt_ctx_stats(ctx)["launches"] == 1 and torch.equal(S.detach(), E)
    S.backward(gS, retain_graph=True)
    assert tt.tt_ctx_stats(ctx)["launches"] == launches
    G = tt.tt_semblance_grad(ctx, th.detach())[1] * gS.unsqueeze(-1)

    def check(G):
        if same:
            assert torch.equal(th.grad, G)
        scale = G.abs().flatten(0, 1).median(0).values
        assert ((th.grad - G).abs() <= 1e-3 * (G.abs() + scale)).all()

    check(G)
    th.grad = None
    tt.tt_ctx_load_traces(ctx, torch.from_numpy(x[::-1].copy()))
    S.backward(gS)
    check(tt.tt_semblance_grad(ctx, th.detach())[1] * gS.unsqueeze(-1))
    ctx.close()


@pytest.mark.parametrize("op,w,storage,ns", [(1, 5, "f32", 300), (0, 3, "f32", 2200),
                                             (2, 8, "bf16", 300), (1, 4, "bf16", 2200)])
def test_uneven_slices_walked_by_one_warp_or_eight(op, w, storage, ns):
    """One unit per SM and two: the same 56 slices of apertures of 0, 1 and up to
    1.39 traces per SM, by a warp each at one unit (mean above 0.6 traces a unit),
    by a warp for eight at two (mean below that, largest below 0.7 and half the
    mean)."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [int(f * n_sm) for f in (1.3, 1.39, 1.0, 0.65, 0.8)] + [0, 1]
    n_dom = 8 * n_sm
    x, mid, off = _line(60, ns)
    prob = _problem(n_dom, sizes, 60, ns, op, w)
    mean = np.diff(prob.ap_ptr)[prob.dom_group].mean()
    assert 0.6 * n_sm < mean < 1.2 * n_sm and max(sizes) < 1.4 * n_sm + 0.5 * mean
    bounds = BOUNDS[op] if op else ((1 / 4500 ** 2,), (1 / 1400 ** 2,))
    th = to_dev(random_theta(n_dom, 16, *bounds, 7))
    ctx = tt.tt_ctx_create(x, mid, off, prob, None, storage=storage, device=dev())
    a = tt.tt_semblance_eval(ctx, th[:, :8].contiguous())
    b = tt.tt_semblance_eval(ctx, th)
    ctx.close()
    assert torch.equal(a, b[:, :8])
    if storage == "f32":
        ref = oracle.semblance.semblance_many(x, mid, off, prob, th[:, :1].cpu().numpy())
        assert np.max(np.abs(a[:, :1].cpu().numpy() - ref)) <= 1e-5


@pytest.mark.parametrize("sizes,np_", [((48,) * 30 + (900,), 32), ((150,), 33)])
def test_stepwise_where_fused_is_slower(sizes, np_):
    """A long aperture among short ones, and a second wave of half-filled blocks:
    the search runs step by step (as many launches as while it is timed)."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    n_dom = 2 * n_sm + 1
    x, mid, off = _line(60, 300)
    prob = _problem(n_dom, sizes, 60, 300)
    ctx = tt.tt_ctx_create(x, mid, off, prob, _cfg(1, np_, 3), device=dev())
    tt.tt_ctx_set_option(ctx, "search_graph", False)
    tt.tt_ctx_stats(ctx, reset=True)
    th, S, _ = tt.tt_search(ctx)
    few = tt.tt_ctx_stats(ctx, reset=True)
    tt.tt_ctx_profile(ctx, True)
    th1, S1, _ = tt.tt_search(ctx)
    assert few["launches"] == tt.tt_ctx_stats(ctx)["launches"]
    ctx.close()
    assert torch.equal(th, th1) and torch.equal(S, S1)


def _device_us(fn, n=20):
    """Least of five averages over n calls."""
    best = float("inf")
    for _ in range(5):
        fn()
        t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t0.record()
        for _ in range(n):
            fn()
        t1.record()
        torch.cuda.synchronize()
        best = min(best, t0.elapsed_time(t1) * 1e3 / n)
    return best


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_stack_of_interleaved_groups(storage):
    """Domains whose group changes at every one: a warp per domain, which a launch
    with as many groups as domains takes too (the same problem with unused groups
    added; a lane per domain took 1.8 times as long, 1.4 is allowed). Sorted by
    group they have the same stack bit for bit."""
    G, n_t = 20, 1500
    n_dom = G * n_t
    x, mid, off = _line(1500, 1500)
    prob = _problem(n_dom, (1008,) * G, 1500, 1500)
    prob.dom_group = np.tile(np.arange(G), n_t).astype(np.int32)
    prob.dom_it0 = np.repeat(np.arange(n_t), G).astype(np.int32)
    th = random_theta(n_dom, 1, *BOUNDS[1], 3)[:, 0]
    by_group = np.argsort(prob.dom_group, kind="stable")
    outs, times = [], []
    for order, unused in ((np.arange(n_dom), 0), (np.arange(n_dom), n_dom), (by_group, 0)):
        p = dataclasses.replace(
            prob, dom_group=prob.dom_group[order], dom_it0=prob.dom_it0[order],
            group_m0=np.pad(prob.group_m0, (0, unused)),
            group_dt=np.pad(prob.group_dt, (0, unused), mode="edge"),
            ap_ptr=np.pad(prob.ap_ptr, (0, unused), mode="edge"))
        ctx = tt.tt_ctx_create(x, mid, off, p, None, storage=storage, device=dev())
        d_th, out = to_dev(th[order]), torch.empty(n_dom, device=dev())
        times.append(_device_us(lambda: tt.tt_stack(ctx, d_th, out)))
        ctx.close()
        back = np.empty(n_dom, np.float32)
        back[order] = out.cpu().numpy()
        outs.append(back)
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])
    assert times[0] <= 1.4 * times[1], times


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_forms_agree_on_infinities_and_nans(storage):
    """Records with infinite and NaN samples: every form of a launch has the same
    values and the same NaNs (evaluation by a warp a slice and a warp for eight;
    fused and stepwise search; stack by lanes and by warps)."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    n_dom, sizes = 8 * n_sm, (int(0.8 * n_sm),)
    x, mid, off = _line(60, 300)
    off[:4] = 5.0  # early windows read the samples below
    x[0, 30:40], x[1, 90:100], x[2, 150:160] = np.inf, np.nan, -np.inf
    prob = _problem(n_dom, sizes, 60, 300)
    th = to_dev(random_theta(n_dom, 16, *BOUNDS[1], 7))

    def same(a, b):
        return torch.equal(a.isnan(), b.isnan()) and torch.equal(a.nan_to_num(), b.nan_to_num())

    ctx = tt.tt_ctx_create(x, mid, off, prob, None, storage=storage, device=dev())
    few, many = tt.tt_semblance_eval(ctx, th[:, :8].contiguous()), tt.tt_semblance_eval(ctx, th)
    lanes = tt.tt_stack(ctx, th[:, 0].contiguous())
    ctx.close()
    own = _problem(n_dom, sizes, 60, 300, own_groups=True)
    ctx = tt.tt_ctx_create(x, mid, off, own, None, storage=storage, device=dev())
    warps = tt.tt_stack(ctx, th[:, 0].contiguous())
    ctx.close()
    assert few.isnan().any() and (few == 0).any() and same(few, many[:, :8])
    assert lanes.isnan().any() and same(lanes, warps)
    prob = _problem(2 * n_sm, (60,), 60, 300)
    ctx = tt.tt_ctx_create(x, mid, off, prob, _cfg(1, 32, 4), storage=storage, device=dev())
    th1, S1, _ = tt.tt_search(ctx)
    tt.tt_ctx_profile(ctx, True)
    th2, S2, _ = tt.tt_search(ctx)
    ctx.close()
    assert torch.equal(th1, th2) and same(S1, S2)


@pytest.mark.parametrize("storage,w,P", [("f32", 5, 8), ("bf16", 8, 8), ("f32", 0, 2),
                                         ("bf16", 3, 20)])
def test_long_split_launches_on_several_streams(storage, w, P):
    """Long apertures at unit counts (0.83, 0.41 and 0.96, 0.98 of a multiple of the
    SMs' blocks) where the blocks' sums meet in the context's scratch: the stream
    that evaluates first has it, another stream takes clusters, as a captured launch
    does. The same bits in all three, and with both streams at work at once."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    n_dom = {8: int(7.8 * n_sm), 2: int(13.2 * n_sm), 20: int(6.3 * n_sm)}[P]
    x, mid, off = _line(200, 300)
    prob = _problem(n_dom, (2000, 1500, 1700), 200, 300, w=w)
    ctx = tt.tt_ctx_create(x, mid, off, prob, None, storage=storage, device=dev())
    th = to_dev(random_theta(n_dom, P, *BOUNDS[1], 7))
    S = tt.tt_semblance_eval(ctx, th)  # the first stream: with scratch
    torch.cuda.synchronize()
    other = torch.cuda.Stream(device=dev())
    outs = [(torch.empty_like(S), torch.empty_like(S)) for _ in range(20)]
    for a, b in outs:  # nothing between the streams
        tt.tt_semblance_eval(ctx, th, a)
        tt.tt_semblance_eval(ctx, th, b, stream=other)
    torch.cuda.synchronize()
    for a, b in outs:
        assert torch.equal(a, S) and torch.equal(b, S)
    T = torch.empty_like(S)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        tt.tt_semblance_eval(ctx, th, T)
    T.zero_()
    graph.replay()
    again = tt.tt_semblance_eval(ctx, th)
    torch.cuda.synchronize()
    ctx.close()
    assert torch.equal(T, S) and torch.equal(again, S)
    if storage == "f32":
        few = np.arange(0, n_dom, 97)
        sub = dataclasses.replace(prob, dom_it0=prob.dom_it0[few], dom_group=prob.dom_group[few])
        ref = oracle.semblance.semblance_many(x, mid, off, sub, th[few].cpu().numpy())
        assert np.max(np.abs(S[few].cpu().numpy() - ref)) <= 1e-5


def test_search_and_sweep_over_long_apertures():
    """The search's and the ENS sweep's split launches over long apertures, whose
    sums meet in scratch of their own: eager and replayed runs agree, beside
    evaluations on another stream, and the semblance reported is the evaluation's."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    n_m0, n_t0 = 4, 5 * n_sm // 4
    n_dom = n_m0 * n_t0
    x, mid, off = _line(200, 300)
    prob = _problem(n_dom, (1600,) * n_m0, 200, 300)
    prob.dom_group = np.repeat(np.arange(n_m0), n_t0).astype(np.int32)
    prob.dom_it0 = np.tile(np.arange(n_t0), n_m0).astype(np.int32)
    prob.n_m0, prob.n_t0 = n_m0, n_t0
    ctx = tt.tt_ctx_create(x, mid, off, prob, _cfg(1, 12, 5, exch_every=2, polish_steps=2),
                           device=dev())
    th = to_dev(random_theta(n_dom, 12, *BOUNDS[1], 7))
    S = tt.tt_semblance_eval(ctx, th)
    other = torch.cuda.Stream(device=dev())
    runs = []
    for graph in (True, False):
        tt.tt_ctx_set_option(ctx, "search_graph", graph)
        for call in (lambda: tt.tt_search(ctx, stream=other),
                     lambda: tt.tt_ens_search(ctx, 12, 2, 12, 2, 2, 1, 2, stream=other)):
            best, bS, n = call()
            for _ in range(4):
                assert torch.equal(tt.tt_semblance_eval(ctx, th), S)
            torch.cuda.synchronize()
            E = tt.tt_semblance_eval(ctx, best[:, None].contiguous())[:, 0]
            assert (E - bS).abs().max().item() <= 1e-5
            runs.append((best, bS, n))
    ctx.close()
    for a, b in zip(runs[:2], runs[2:]):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and a[2] == b[2]
