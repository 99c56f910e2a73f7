"""The selection behind PML and TVaR at the edges of its forms (rows sorted whole, one cooperative
launch, a cluster per row, lists split a second time), against sorted rows.  PML is a copy of a YLT
entry, so it is equal; TVaR and the mean are FP64 sums of up to 3e6 values of one sign in trees of
pairwise depth, 1e-13 relative (about 500 rounding units; the trees are a few tens deep)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1606_04473_gb300 as ara

RPS = [1.0, 2.0, 10.0, 100.0, 250.0]
LEVELS = [0.0, 0.5, 0.99]


def count(x):
    r = np.rint(x)
    return int(r if abs(x - r) <= 1e-9 * max(1.0, abs(x)) else np.ceil(x))


def check(y, rps=RPS, levels=LEVELS, call=None):
    d = torch.from_numpy(y).cuda()
    call = call or ara.risk_metrics
    pml, tvar, mean = call(d, rps, levels, want_mean=True)
    s = np.sort(y, axis=1)[:, ::-1]
    n = y.shape[1]
    for i, r in enumerate(rps):
        assert np.array_equal(pml[:, i], s[:, count(n / r) - 1]), r
    for i, p in enumerate(levels):
        m = count(n * (1.0 - p))
        np.testing.assert_allclose(tvar[:, i], s[:, :m].astype(np.longdouble).mean(1).astype(float), rtol=1e-13)
    np.testing.assert_allclose(mean, y.astype(np.longdouble).mean(1).astype(float), rtol=1e-13)


def rows(seed, n_rows, n):
    """Shapes a YLT can take: lognormal years, zeros below a retention with ties at a limit, sorted
    years, few distinct values, one large value in a constant row, near-equal neighbours."""
    g = np.random.default_rng(seed)
    out = np.empty((n_rows, n))
    for i in range(n_rows):
        x = np.exp(g.normal(14.0, 2.0, n))
        k = i % 6
        if k == 1:
            x = np.clip(x - np.median(x), 0.0, np.quantile(x, 0.97))
        elif k == 2:
            x = np.sort(x)
        elif k == 3:
            x = g.integers(0, 7, n) * 1e6
        elif k == 4:
            x[:] = 3.5
            x[n // 3] = 1e9
        elif k == 5:
            x = 1e6 + np.arange(n) % 5000 * np.spacing(1e6)
        out[i] = x
    return out


@pytest.mark.parametrize("n_rows,n", [(6, 1), (6, 2), (6, 63), (6, 65), (7, 1000), (6, 4096), (6, 4097), (6, 30_011),
                                      (32, 5_000), (33, 5_000), (1, 400_003), (40, 70_001), (160, 4_100), (6, 600_000)])
def test_rows_of_every_form(n_rows, n):
    levels = [p for p in LEVELS if count(n * (1.0 - p)) >= 1]
    check(rows(n, n_rows, n), levels=levels)


def test_allocation_free_call_splits_overfull_lists():
    """Sixteen targets on a long row: the fixed array holds lists of a few thousand keys only, so the
    intervals are split a second time (for several targets that share one, too)."""
    g = np.random.default_rng(4)
    y = np.exp(g.normal(14.0, 1.0, (2, 3_000_017)))
    y[1, : 1_000_000] = 0.0
    rps = [1.0, 1.5, 2.0, 2.0000001, 2.0000002, 3.0, 10.0, 100.0, 250.0, 1000.0, 2000.0]
    check(y, rps, [0.0, 0.3, 0.5, 0.9, 0.99], ara.risk_metrics_static)


@pytest.mark.parametrize("n", [64, 1023, 1024, 1025, 2047, 2048, 2049, 4095])
def test_short_rows_at_the_widths_of_the_sort(n):
    levels = [p for p in LEVELS if count(n * (1.0 - p)) >= 1]
    check(rows(n + 1, 5, n), levels=levels)


@pytest.mark.parametrize("n,rps,levels", [(57_935, [100.0], [0.99]), (19_052, [100.0, 10.0], [0.99])])
def test_allocation_free_call_in_uneven_groups(n, rps, levels):
    """65 rows: a first group of 33 (a cluster each) would fit the array, its remainder of 32 (one cooperative
    launch, which needs class counts) would not."""
    check(rows(n, 65, n), rps, levels, ara.risk_metrics_static)


@pytest.mark.parametrize("n_rows,n", [(40, 70_001), (6, 600_000), (1, 1_000_003), (300, 5_000)])
def test_with_little_memory_the_same_bits(n_rows, n):
    """With 8 KiB for each row and target (and for a single row the least that two rounds need), the rows
    run in groups with short lists, in clusters or in the cooperative form: every result the same."""
    import ctypes
    d = torch.from_numpy(rows(n, n_rows, n)).cuda()
    want = ara.risk_metrics(d, RPS, LEVELS, want_mean=True)
    nt = len(RPS) + len(LEVELS)
    out = [torch.full((n_rows, k), -1.0, dtype=torch.float64, device="cuda") for k in (len(RPS), len(LEVELS), 1)]
    status = torch.full((1,), 9, dtype=torch.int32, device="cuda")
    arr = lambda v: (ctypes.c_double * len(v))(*v)
    for budget in (8192 * max(n_rows, 4) * nt, 8192 * max(n_rows // 4, 4) * nt):
        for call in ("wait", "queue"):
            ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, budget)
            try:
                if call == "wait":
                    got = ara.risk_metrics(d, RPS, LEVELS, want_mean=True)
                else:
                    st = ara.lib().ara_risk_metrics_async(
                        d.data_ptr(), n, n_rows, len(RPS), arr(RPS), len(LEVELS), arr(LEVELS), out[0].data_ptr(),
                        out[1].data_ptr(), out[2].data_ptr(), status.data_ptr(), torch.cuda.current_stream().cuda_stream)
                    assert st == ara.ARA_OK
                    got = [o.cpu().numpy() for o in out]
                    assert int(status) == 0
            finally:
                ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, 0)
            assert all(np.array_equal(a.reshape(b.shape), b) for a, b in zip(got, want))
    # the row sum alone has no lists
    ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, 40_000 + 200 * n_rows)
    try:
        got = ara.risk_metrics(d, [], [], want_mean=True)
    finally:
        ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, 0)
    assert np.array_equal(got[2], want[2])


def test_host_run_with_little_memory():
    """The selection of a run from host memory keeps its scratch with the portfolio: the same metrics
    where only short lists fit."""
    g = np.random.default_rng(2)
    n = 30_000
    off = np.arange(n + 1, dtype=np.int64) * 4
    ids = g.integers(0, 1000, 4 * n, dtype=np.int32)
    made = lambda: ara.Portfolio(1000, [np.arange(1000, dtype=np.int32)], [np.exp(g2.normal(10, 1, 1000))], [0.0], [np.inf],
                                 [[0]] * 3, [0.0] * 3, [1e9] * 3, [0.0, 1e4, 2e4], [1e12] * 3)
    g2 = np.random.default_rng(3)
    a = made()
    want = a.run_ylt_host(off, ids, return_periods=RPS, tvar_levels=LEVELS, want_mean=True)
    g2 = np.random.default_rng(3)
    b = made()
    # staging, offsets, rows and results, and 200 KB of the 1.2 MB of lists
    ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, 2 * (4 * ids.size + 8 * off.size) + 8 * 3 * n + 4096 + 200_000)
    try:
        got = b.run_ylt_host(off, ids, return_periods=RPS, tvar_levels=LEVELS, want_mean=True)
    finally:
        ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, 0)
    assert all(np.array_equal(x, y) for x, y in zip(got, want))
    a.close()
    b.close()


@pytest.mark.parametrize("n_rows,n", [(6, 1000), (6, 9_001), (40, 9_001), (6, 600_000)])
def test_special_values(n_rows, n):
    """Infinities, NaN, zeros of both signs and the type's extremes: in the order of the bits (a NaN above
    +inf or below -inf, by its sign); sums as IEEE gives them."""
    g = np.random.default_rng(n)
    big = np.finfo(np.float64).max
    special = np.array([np.inf, -np.inf, np.nan, -np.nan, 0.0, -0.0, big, -big, 5e-324, -5e-324])
    special = np.append(special, np.frombuffer(b"\xff" * 8 + b"\xff" * 7 + b"\x7f", dtype=np.float64))
    y = g.lognormal(3.0, 2.0, (n_rows, n))
    for i in range(n_rows):
        k = i % 6
        if k == 0:
            y[i, g.choice(n, 40, replace=False)] = np.inf
        elif k == 1:
            y[i, g.choice(n, n // 3, replace=False)] = -np.inf
        elif k == 2:
            y[i, g.choice(n, n // 2, replace=False)] = np.nan
        elif k == 3:
            y[i] = special[g.integers(0, special.size, n)]
        elif k == 4:
            y[i] = np.where(g.random(n) < 0.5, 0.0, -0.0)
        else:
            y[i] = np.inf
    levels = [p for p in LEVELS if count(n * (1.0 - p)) >= 1]
    pml, tvar, mean = ara.risk_metrics(torch.from_numpy(y).cuda(), RPS, levels, want_mean=True)
    b = y.view(np.uint64)
    key = np.where(b >> np.uint64(63), ~b, b | np.uint64(1 << 63))
    order = np.argsort(key, axis=1)[:, ::-1]
    s = np.take_along_axis(y, order, axis=1)
    same = lambda x, w: np.array_equal(x.view(np.uint64), w.view(np.uint64))
    with np.errstate(all="ignore"):
        for i, r in enumerate(RPS):
            assert same(np.ascontiguousarray(pml[:, i]), np.ascontiguousarray(s[:, count(n / r) - 1]))
        for i, p in enumerate(levels):
            m = count(n * (1.0 - p))
            want = s[:, :m].astype(np.longdouble).sum(1) / m
            rows = [r for r in range(n_rows) if r % 6 != 3]      # sums near the largest double may overflow on the way
            np.testing.assert_allclose(tvar[rows, i], want[rows].astype(np.float64), rtol=1e-13)
        want = (y.astype(np.longdouble).sum(1) / n).astype(np.float64)
        np.testing.assert_allclose(mean[rows], want[rows], rtol=1e-13)


@pytest.mark.parametrize("n_rows,n", [(40, 100_000), (33, 5_000), (8, 4_097), (24, 300_001), (100, 9_000)])
def test_allocation_free_call_has_the_bits_of_the_allocating_one(n_rows, n):
    """Where the request fits the fixed array with tight lists, it runs in one go in the same form."""
    d = torch.from_numpy(rows(n, n_rows, n)).cuda()
    rps, levels = [100.0, 250.0], [0.99]
    n0 = ara.launch_count()
    got = ara.risk_metrics_static(d, rps, levels, want_mean=True)
    assert ara.launch_count() - n0 == 1
    assert all(np.array_equal(a, b) for a, b in zip(got, ara.risk_metrics(d, rps, levels, want_mean=True)))
