"""Several layers in one pass over event-major rows: every form of the rows (kept in place 1, 2 or
4 entries to an event, or end to end; one pass or several; 4 to 32 columns of sums) against the
single-layer path, bit for bit (both paths sum the same integers exactly, so no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1606_04473_gb300 as ara


def make(seed, C, n_elts, nnz, layers, f32, trials, events, mult=1.0):
    """A portfolio of `layers` (lists of ELTs) and a ragged YET with empty and one-event trials; layer
    terms at multiples of typical losses so that all clamp regimes occur."""
    g = np.random.default_rng(seed)
    ids = [g.choice(C, size=min(nnz, C), replace=False).astype(np.int32) for _ in range(n_elts)]
    loss = [np.exp(11.0 + 2.0 * g.standard_normal(i.size)) for i in ids]
    if f32:
        loss = [x.astype(np.float32).astype(np.float64) for x in loss]
    ret = np.array([np.percentile(x, 20) for x in loss])
    lim = np.array([np.percentile(x, 95) for x in loss])
    lim[::7] = np.inf
    n = len(layers)
    occ_r = g.uniform(0.0, 2e5, n)
    occ_r[::5] = 0.0
    pf = ara.Portfolio(C, ids, loss, ret, lim, layers, occ_r, g.uniform(1e5, 3e6, n),
                       g.uniform(0.0, 1e6, n) * mult, g.uniform(1e6, 5e7, n) * mult, losses_f32=f32)
    counts = g.poisson(events, trials)
    counts[:6] = [0, 1, 0, 31, 32, 33]
    counts[-1] = 0
    off = np.zeros(trials + 1, np.int64)
    np.cumsum(counts, out=off[1:])
    yet = g.integers(0, C, off[-1], dtype=np.int32)
    return pf, torch.from_numpy(off).cuda(), torch.from_numpy(yet).cuda()


def singles(pf, off, ids, sel):
    n = off.numel() - 1
    reg = torch.empty((len(sel), n), dtype=torch.uint8, device="cuda")
    ys = []
    for i, l in enumerate(sel):
        r = torch.empty((1, n), dtype=torch.uint8, device="cuda")
        ys.append(pf.run_ylt(off, ids, layers=[l], regimes=r)[0])
        reg[i] = r[0]
    pf.check()
    return torch.stack(ys), reg


def own(g, n_layers, n_elts, lo, hi):
    return [sorted(g.choice(n_elts, size=int(g.integers(lo, hi + 1)), replace=False).tolist())
            for _ in range(n_layers)]


# (catalogue, ELTs, records per ELT, layers, ELTs per layer, f32, trials, events per trial): the
# number of entries per event decides the form (in place 1, 2, 4; end to end), the number of
# layers the columns (up to 18: 32, 37-40: 16, 74: 8, else 4)
FORMS = [
    (5_003, 6, 200, 2, (1, 2), False, 700, 90.0),        # 1 in place, overflow rare
    (20_011, 12, 1_500, 9, (1, 3), True, 900, 120.0),    # 2 in place
    (4_096, 24, 300, 16, (2, 4), True, 501, 700.0),      # 4 in place, catalogue of whole tiles
    (3_000, 30, 1_400, 24, (5, 25), False, 400, 1200.0), # end to end, long rows, several drains
    (2_049, 40, 500, 64, (3, 30), True, 300, 300.0),     # end to end, 8 columns
    (1_000, 20, 700, 130, (1, 20), False, 200, 150.0),   # 4 columns, 130 layers, dense
    (777, 8, 777, 255, (1, 8), True, 65, 40.0),          # every event in every ELT, 255 layers
    (40, 3, 40, 3, (1, 3), True, 2_000, 3.0),            # a catalogue of one warp, short trials
]


@pytest.mark.parametrize("form", range(len(FORMS)))
def test_rows_equal_single_layer_runs(form):
    C, n_elts, nnz, n_layers, (lo, hi), f32, trials, events = FORMS[form]
    layers = own(np.random.default_rng(form), n_layers, n_elts, lo, hi)
    pf, off, ids = make(form, C, n_elts, nnz, layers, f32, trials, events)
    every = list(range(n_layers))
    ref, reg_ref = singles(pf, off, ids, every)
    assert 0 < int((reg_ref == 1).sum())
    some = every[::-1][: max(2, n_layers // 2)]          # a selection that is not in order
    for sel, autotune in ((every, False), (every, True), (some, False)):
        reg = torch.full((len(sel), trials), 9, dtype=torch.uint8, device="cuda")
        plan = ara.BatchedPlan(pf, off, ids, layers=sel, regimes=reg, autotune=autotune)
        y = plan.launch()
        pf.check()
        idx = torch.tensor(sel, device="cuda")
        assert torch.equal(y, ref[idx]) and torch.equal(reg, reg_ref[idx])
        rows, n_entries = plan.table()
        assert int(((rows >> 32) & 0xff).sum()) == n_entries
        plan.close()
        a = pf.run_ylt(off, ids, layers=sel, flags=ara.ARA_RUN_BATCHED)
        pf.check()
        assert torch.equal(a, ref[idx])
    pf.close()


def test_layers_in_any_elt_order_take_the_general_way():
    """Layers that do not list their ELTs in ascending order (or twice) keep their own order of the
    FP64 ELT sum: rows from the per-layer folds, equal to the single-layer runs."""
    g = np.random.default_rng(3)
    layers = [g.permutation(12)[:7].tolist() for _ in range(11)] + [[4, 4, 1], []]
    pf, off, ids = make(5, 4_000, 12, 900, layers, True, 333, 400.0)
    sel = list(range(len(layers)))
    ref, reg_ref = singles(pf, off, ids, sel)
    reg = torch.empty_like(reg_ref)
    plan = ara.BatchedPlan(pf, off, ids, regimes=reg, autotune=False)
    assert torch.equal(plan.launch(), ref) and torch.equal(reg, reg_ref)
    rows, n_entries = plan.table()
    assert int(((rows >> 32) & 0xff).sum()) == n_entries
    plan.close()
    pf.close()


@pytest.mark.parametrize("form", [0, 1, 2, 3, 5, 7])
def test_rows_of_layers_in_descending_elt_order(form):
    """The general way in every form of the rows, in place with and without overflow and end to end."""
    C, n_elts, nnz, n_layers, (lo, hi), f32, trials, events = FORMS[form]
    layers = [l[::-1] for l in own(np.random.default_rng(form), n_layers, n_elts, max(lo, 2), hi)] + [[]]
    pf, off, ids = make(form, C, n_elts, nnz, layers, f32, trials, events)
    sel = [0] + list(range(n_layers + 1))[1:][::-1]
    ref, reg_ref = singles(pf, off, ids, sel)
    for autotune in (False, True):
        reg = torch.full((len(sel), trials), 9, dtype=torch.uint8, device="cuda")
        plan = ara.BatchedPlan(pf, off, ids, layers=sel, regimes=reg, autotune=autotune)
        assert torch.equal(plan.launch(), ref) and torch.equal(reg, reg_ref)
        rows, n_entries = plan.table()
        assert int(((rows >> 32) & 0xff).sum()) == n_entries
        plan.close()
    for budget in (0, 20 * C + 8 * sum(nnz * len(l) for l in layers) + 8 * C + 4096):   # and end to end without room
        ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, budget)
        try:
            a = pf.run_ylt(off, ids, layers=sel, flags=ara.ARA_RUN_BATCHED)
        finally:
            ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, 0)
        assert torch.equal(a, ref)
    pf.check()
    pf.close()


@pytest.mark.parametrize("shape", [(2_000_000, 60, 20_000, 70, 4, 18), (1_500_000, 80, 30_000, 120, 3, 20)])
def test_tables_beyond_l2_run_in_several_passes(shape):
    """Tables large enough for several passes over the YET (8 and 4 columns): sums carried from
    pass to pass, equal to the single-layer runs; IDs outside the catalogue are still reported."""
    C, n_elts, nnz, n_layers, lo, hi = shape
    layers = own(np.random.default_rng(1), n_layers, n_elts, lo, hi)
    pf, off, ids = make(2, C, n_elts, nnz, layers, True, 1_500, 900.0, mult=3.0)
    sel = [0, n_layers // 2, n_layers - 1]
    ref, reg_ref = singles(pf, off, ids, sel)
    for autotune in (False, True):
        reg = torch.empty((n_layers, off.numel() - 1), dtype=torch.uint8, device="cuda")
        plan = ara.BatchedPlan(pf, off, ids, regimes=reg, autotune=autotune)
        y = plan.launch()
        pf.check()
        assert torch.equal(y[sel], ref) and torch.equal(reg[sel], reg_ref)
        plan.close()
    bad = ids.clone()
    bad[12_345] = C
    plan = ara.BatchedPlan(pf, off, bad, autotune=False)
    plan.launch()
    with pytest.raises(ara.AraError) as ei:
        pf.check()
    assert ei.value.status == ara.ARA_EDATA
    plan.close()
    pf.close()


def test_run_of_several_layers_takes_the_rows_and_keeps_prepared_runs():
    """An ordinary run of many layers goes through the rows (two kernels, whatever the number of
    layers) and equals the single-layer runs; a prepared run right after it, without a prepare of
    its own, still streams against the folds of those layers; a run being captured stays with the
    per-layer kernels and replays the same values."""
    g = np.random.default_rng(8)
    pf, off, ids = make(9, 50_000, 40, 3_000, own(g, 20, 40, 5, 20), True, 2_000, 500.0)
    sel = list(range(20))
    ref, reg_ref = singles(pf, off, ids, sel)
    reg = torch.empty_like(reg_ref)
    n0 = ara.launch_count()
    y = pf.run_ylt(off, ids, regimes=reg)
    assert ara.launch_count() - n0 <= 3
    assert torch.equal(y, ref) and torch.equal(reg, reg_ref)
    for layers in ([7, 3], sel):
        z = pf.run_ylt(off, ids, layers=layers, flags=ara.ARA_RUN_PREPARED)
        assert torch.equal(z, ref[layers])
    pf.check()
    s = torch.cuda.Stream()
    out = torch.zeros_like(ref)
    graph = torch.cuda.CUDAGraph()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=s):
        pf.run_ylt(off, ids, out=out, stream=s)
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    pf.check()
    pf.close()


@pytest.mark.parametrize("C,n_elts,nnz,f32", [(31, 3, 20, True), (257, 5, 200, False), (70_001, 9, 4_000, True),
                                              (200_000, 12, 9_000, False), (1_000_003, 8, 60_000, True)])
def test_fold_by_event_equals_fold_by_tiles(C, n_elts, nnz, f32):
    """The fold from the event-major records against the fold by tiles, which a layer with its ELTs in
    another order takes: two ELTs per event at most make the order of the sum irrelevant, so the
    YLTs, the maxima and the adjoints (occurrence regimes) are equal."""
    g = np.random.default_rng(C)
    ids = [np.sort(g.choice(C, size=nnz, replace=False)).astype(np.int32) for _ in range(n_elts)]
    seen = np.zeros(C, np.int32)
    keep = []
    for i in ids:                       # at most two ELTs per event
        k = seen[i] < 2
        seen[i[k]] += 1
        keep.append(i[k])
    loss = [np.exp(11.0 + 2.0 * g.standard_normal(i.size)) for i in keep]
    if f32:
        loss = [x.astype(np.float32).astype(np.float64) for x in loss]
    ret, lim = np.full(n_elts, 1e4), np.full(n_elts, 1e6)
    up = list(range(n_elts))
    part = up[: max(2, n_elts - 2)]     # a layer that does not hold every ELT
    for layer in (up, part):
        pf = ara.Portfolio(C, keep, loss, ret, lim, [layer, layer[::-1]], [2e4] * 2, [9e5] * 2, [1e5] * 2, [1e7] * 2,
                           losses_f32=f32)
        counts = g.poisson(60.0, 400)
        off = np.zeros(401, np.int64)
        np.cumsum(counts, out=off[1:])
        off, yet = torch.from_numpy(off).cuda(), torch.from_numpy(g.integers(0, C, off[-1], dtype=np.int32)).cuda()
        reg = torch.empty((2, 400), dtype=torch.uint8, device="cuda")
        ys = [pf.run_ylt(off, yet, layers=[l], regimes=reg[l:l + 1]) for l in (0, 1)]
        assert torch.equal(ys[0], ys[1]) and torch.equal(reg[0], reg[1])
        f64 = [pf.run_ylt(off, yet, layers=[l], flags=ara.ARA_RUN_F64_SUM) for l in (0, 1)]
        oep = [pf.run_ylt(off, yet, layers=[l], flags=ara.ARA_RUN_OEP) for l in (0, 1)]
        assert torch.equal(f64[0], f64[1]) and torch.equal(oep[0], oep[1])
        a, b = (pf.adjoint(off, yet, ys[l], reg[l:l + 1], 0.9, layers=[l]) for l in (0, 1))
        assert torch.equal(a["layer"], b["layer"])
        k = len(layer)
        assert torch.equal(a["elt"], b["elt"].flip(1)) and k == a["elt"].shape[1]
        pf.check()
        pf.close()


@pytest.mark.parametrize("captured", ["prepared", "plain"])
def test_a_captured_fold_does_not_count_before_its_replay(captured):
    """After an ordinary run by rows the folds of its layers are missing from slot 0.  A prepared (or an
    ordinary) run that is only captured records the fold; an eager prepared run before the first replay
    still finds it missing and folds itself."""
    g = np.random.default_rng(12)
    pf, off, ids = make(13, 20_000, 30, 2_000, own(g, 12, 30, 3, 12), True, 500, 200.0)
    sel = list(range(12))
    ref, _ = singles(pf, off, ids, sel)
    # slot 0 holds other values for these layers (sums in FP64, not the fixed point of an ordinary run)
    pf.run_ylt(off, ids, layers=sel[::-1], flags=ara.ARA_RUN_F64_SUM)
    n0 = ara.launch_count()
    assert torch.equal(pf.run_ylt(off, ids, layers=sel), ref) and ara.launch_count() - n0 <= 3
    s = torch.cuda.Stream()
    out = torch.zeros_like(ref)
    graph = torch.cuda.CUDAGraph()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=s):
        pf.run_ylt(off, ids, layers=sel, out=out, flags=ara.ARA_RUN_PREPARED if captured == "prepared" else 0, stream=s)
    assert torch.equal(pf.run_ylt(off, ids, layers=sel, flags=ara.ARA_RUN_PREPARED), ref)
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    pf.check()
    pf.close()


def test_a_portfolio_without_room_for_its_event_index():
    """Room for the portfolio (13 MB here) but not for the records event by event too (5 MB): it is made all
    the same, and works through the per-layer folds."""
    args = (15, 100_000, 20, 20_000, [[2 * l, 2 * l + 1] for l in range(8)], False, 500, 200.0)
    pf, off, ids = make(*args)
    ref, reg_ref = singles(pf, off, ids, list(range(8)))
    pf.close()
    ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, 14_200_000)
    try:
        pf, off, ids = make(*args)
    finally:
        ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, 0)
    y, reg = singles(pf, off, ids, list(range(8)))
    assert torch.equal(y, ref) and torch.equal(reg, reg_ref)
    n0 = ara.launch_count()
    assert torch.equal(pf.run_ylt(off, ids), ref) and ara.launch_count() - n0 >= 8      # no rows without the index
    assert torch.equal(pf.run_ylt(off, ids, flags=ara.ARA_RUN_BATCHED), ref)
    pf.check()
    pf.close()


def test_without_room_for_the_rows_prepared_folds_stay():
    """An ordinary run whose rows do not fit the memory goes layer by layer, through its own layers' tables
    only: a fold prepared in slot 0 for other layers is still there.  (The general way of a batched run
    needs less scratch than rows in place, here 1.8 MB against 2.4, but uses the tables by slot.)"""
    pf, off, ids = make(11, 50_000, 18, 6_000, [[l] for l in range(18)], True, 900, 200.0)
    sel = list(range(2, 18))
    ref, _ = singles(pf, off, ids, list(range(18)))
    pf.prepare_ylt(layers=[0, 1], slot=0)
    for budget in (2_100_000, 1):
        ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, budget)
        try:
            n0 = ara.launch_count()
            y = pf.run_ylt(off, ids, layers=sel)
            assert ara.launch_count() - n0 >= len(sel)
        finally:
            ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, 0)
        assert torch.equal(y, ref[sel])
        z = pf.run_ylt(off, ids, layers=[0, 1], flags=ara.ARA_RUN_PREPARED)
        assert torch.equal(z, ref[[0, 1]])
    n0 = ara.launch_count()
    assert torch.equal(pf.run_ylt(off, ids, layers=sel), ref[sel]) and ara.launch_count() - n0 <= 3   # with room: rows
    pf.check()
    pf.close()


def test_largest_portfolios_run_layer_by_layer():
    """32 layers over 2^27 events, one step past what a batched pass takes: the ordinary run goes layer by
    layer, also where the rows would be the faster way."""
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 40 GB of device memory")
    C, n_layers, n = 1 << 27, 32, 64
    g = np.random.default_rng(6)
    ids = [np.sort(g.choice(C, size=5_000, replace=False)).astype(np.int32) for _ in range(4)]
    ids[0][0], ids[1][-1] = 0, C - 1
    loss = [np.full(5_000, 1e5 * (j + 1)) for j in range(4)]
    z = np.zeros(n_layers)
    pf = ara.Portfolio(C, ids, loss, np.zeros(4), np.full(4, np.inf), own(g, n_layers, 4, 1, 3), z + 1e4, z + 3e5,
                       z, z + 1e9)
    hits = np.concatenate(ids)
    yet = torch.from_numpy(g.choice(hits, size=n * 50)).cuda()
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda") * 50
    y = pf.run_ylt(off, yet)
    pf.check()
    ref, _ = singles(pf, off, yet, [0, 17, 31])
    assert torch.equal(y[[0, 17, 31]], ref) and bool((y > 0).any(1).all())
    with pytest.raises(ara.AraError) as e:
        pf.run_ylt(off, yet, flags=ara.ARA_RUN_BATCHED)
    assert e.value.status == ara.ARA_ERANGE
    pf.close()


# every row form of FORMS, and windows at both ends of the trials, inside them and of one trial
@pytest.mark.parametrize("form", [0, 1, 2, 3, 4, 6])
@pytest.mark.parametrize("window", [(0, 1), (0, 40), (7, 52), "last"])
def test_one_request_with_a_window_writes_its_own_trials_only(form, window):
    """One request over a part of the trials: rows of the window's length, equal to a run of the slice,
    and nothing before or after them."""
    import ctypes
    C, n_elts, nnz, n_layers, (lo, hi), f32, trials, events = FORMS[form]
    pf, off, ids = make(form, C, n_elts, nnz, own(np.random.default_rng(form), n_layers, n_elts, lo, hi), f32,
                        trials, events)
    t0, t1 = window if window != "last" else (trials - 1, trials)
    n, pad = n_layers * (t1 - t0), n_layers * trials
    y = torch.full((n + 2 * pad,), -7.0, dtype=torch.float64, device="cuda")
    r = torch.full((n + 2 * pad,), 77, dtype=torch.uint8, device="cuda")
    one = lambda v: (ctypes.c_int64 * 1)(v)
    st = ara.lib().ara_run_ylt_requests(
        pf._h, trials, off.data_ptr(), ids.numel(), ids.data_ptr(), 1, (ctypes.c_int32 * 2)(0, n_layers), one(t0),
        one(t1), (ctypes.c_void_p * 1)(y.data_ptr() + 8 * pad), (ctypes.c_void_p * 1)(r.data_ptr() + pad),
        torch.cuda.current_stream().cuda_stream)
    assert st == ara.ARA_OK
    pf.check()
    ref, reg_ref = singles(pf, off[t0:t1 + 1], ids, list(range(n_layers)))
    assert torch.equal(y[pad:pad + n].view(n_layers, -1), ref) and torch.equal(r[pad:pad + n].view(n_layers, -1), reg_ref)
    assert bool((y[:pad] == -7.0).all() & (y[pad + n:] == -7.0).all() & (r[:pad] == 77).all() & (r[pad + n:] == 77).all())
    pf.close()


# the fold's tiles beyond those that run at once: 512 events (by size, and with enough records), 1,024 (few records)
@pytest.mark.parametrize("C,n_elts,nnz,f32", [(300_001, 6, 9_000, True), (999_999, 10, 60_000, False),
                                              (600_007, 8, 20_000, True), (1_300_000, 12, 30_000, False)])
def test_fold_by_event_in_larger_tiles(C, n_elts, nnz, f32):
    test_fold_by_event_equals_fold_by_tiles(C, n_elts, nnz, f32)
