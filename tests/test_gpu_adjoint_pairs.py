"""The adjoint of several layers in one pass, whose histogram adds to two entries of an event's row at
once and whose rows come from the event-major records (ELTs listed in ascending order) or from the
layers' folds (any other order): equal, bit for bit, to the pass over the event-major index and to one
pass per layer.  The counts are integers, so no tolerance."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1606_04473_gb300 as ara


# layers at the edges of the slot widths of a row descriptor; rows from mostly empty to one entry per layer
@pytest.mark.parametrize("n_layers", [2, 3, 16, 17, 64, 65, 255])
@pytest.mark.parametrize("nnz", [60, 2_000, 4_999])
@pytest.mark.parametrize("ascending", [True, False])
def test_pairs_equal_the_other_passes(n_layers, nnz, ascending):
    g = np.random.default_rng(1000 * n_layers + nnz)
    C, n_elts, trials = 5_000, 12, 700
    ids = [g.choice(C, size=nnz, replace=False).astype(np.int32) for _ in range(n_elts)]
    loss = [np.exp(11.0 + 2.0 * g.standard_normal(nnz)) for _ in ids]
    layers = [sorted(g.choice(n_elts, size=int(g.integers(2, 5)), replace=False).tolist(), reverse=not ascending)
              for _ in range(n_layers)]
    z = np.zeros(n_layers)
    pf = ara.Portfolio(C, ids, loss, np.full(n_elts, 1e4), np.full(n_elts, 1.5e6), layers, z + 1e4, z + 2e6,
                       g.uniform(0.0, 1e6, n_layers), z + 1e13)
    counts = g.poisson(300, trials)
    counts[[0, 5, trials - 1]] = 0
    off = np.zeros(trials + 1, np.int64)
    np.cumsum(counts, out=off[1:])
    off, ev = torch.from_numpy(off).cuda(), torch.from_numpy(g.integers(0, C, off[-1], dtype=np.int32)).cuda()
    reg = torch.empty((n_layers, trials), dtype=torch.uint8, device="cuda")
    ylt = pf.run_ylt(off, ev, regimes=reg)
    pf.check()
    a = pf.adjoint(off, ev, ylt, reg, 0.98)
    assert float(a["loss"].abs().sum()) > 0
    others = [pf.adjoint(None, None, ylt, reg, 0.98, index=pf.yet_index(off, ev))]
    if n_layers <= 17:
        ara.debug_set(ara.ARA_DBG_ADJOINT_PER_LAYER, 1)
        try:
            others.append(pf.adjoint(off, ev, ylt, reg, 0.98))
        finally:
            ara.debug_set(ara.ARA_DBG_ADJOINT_PER_LAYER, 0)
    for b in others:
        assert all(torch.equal(a[k], b[k]) for k in ("elt", "layer", "loss")) and np.array_equal(a["ties"], b["ties"])
    pf.close()


def test_longest_yets_count_single_entries():
    """A YET of 2^32 occurrences and more keeps one 32-bit add per entry; here its trials cover the first few."""
    g = np.random.default_rng(3)
    C, n_elts, trials, n_layers = 5_000, 12, 300, 20
    ids = [g.choice(C, size=3_000, replace=False).astype(np.int32) for _ in range(n_elts)]
    loss = [np.exp(11.0 + 2.0 * g.standard_normal(3_000)) for _ in ids]
    layers = [sorted(g.choice(n_elts, size=3, replace=False).tolist()) for _ in range(n_layers)]
    z = np.zeros(n_layers)
    pf = ara.Portfolio(C, ids, loss, np.full(n_elts, 1e4), np.full(n_elts, 1.5e6), layers, z + 1e4, z + 2e6,
                       g.uniform(0.0, 1e6, n_layers), z + 1e13)
    off = torch.arange(trials + 1, dtype=torch.int64, device="cuda") * 200
    ev = torch.from_numpy(g.integers(0, C, trials * 200, dtype=np.int32)).cuda()
    reg = torch.empty((n_layers, trials), dtype=torch.uint8, device="cuda")
    ylt = pf.run_ylt(off, ev, regimes=reg)
    pf.check()
    a = pf.adjoint(off, ev, ylt, reg, 0.98)
    assert float(a["loss"].abs().sum()) > 0
    longest = torch.empty(1 << 32, dtype=torch.int32, device="cuda")
    longest[: ev.numel()] = ev
    b = pf.adjoint(off, longest, ylt, reg, 0.98)
    assert all(torch.equal(a[k], b[k]) for k in ("elt", "layer", "loss")) and np.array_equal(a["ties"], b["ties"])
    pf.close()


@pytest.mark.parametrize("ascending", [True, False])
def test_with_less_memory_single_entries(ascending):
    """Without room for rows of whole pairs (13 bytes for each event more) the histogram counts single
    entries, from the folds: the same gradients down to the least memory the call runs in."""
    g = np.random.default_rng(9)
    C, n_elts, trials, n_layers = 60_000, 12, 700, 6
    ids = [g.choice(C, size=20_000, replace=False).astype(np.int32) for _ in range(n_elts)]
    loss = [np.exp(11.0 + 2.0 * g.standard_normal(20_000)) for _ in ids]
    layers = [sorted(g.choice(n_elts, size=4, replace=False).tolist(), reverse=not ascending) for _ in range(n_layers)]
    z = np.zeros(n_layers)
    pf = ara.Portfolio(C, ids, loss, np.full(n_elts, 1e4), np.full(n_elts, 1.5e6), layers, z + 1e4, z + 2e6, z + 1e5,
                       z + 1e13)
    off = torch.arange(trials + 1, dtype=torch.int64, device="cuda") * 200
    ev = torch.from_numpy(g.integers(0, C, trials * 200, dtype=np.int32)).cuda()
    reg = torch.empty((n_layers, trials), dtype=torch.uint8, device="cuda")
    ylt = pf.run_ylt(off, ev, regimes=reg)
    want = pf.adjoint(off, ev, ylt, reg, 0.98)

    def within(budget):
        ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, budget)
        try:
            return pf.adjoint(off, ev, ylt, reg, 0.98)
        except ara.AraError as e:
            assert e.status == ara.ARA_ENOMEM
            return None
        finally:
            ara.debug_set(ara.ARA_DBG_MEMORY_BUDGET, 0)

    lo, hi = 1, 64 << 20                       # the least budget, to 1 KB
    while hi - lo > 1024:
        mid = (lo + hi) // 2
        got = within(mid)
        if got is None:
            lo = mid
        else:
            hi = mid
            assert all(torch.equal(got[k], want[k]) for k in ("elt", "layer", "loss"))
            assert np.array_equal(got["ties"], want["ties"])
    entries = sum(20_000 * len(l) for l in layers)
    assert hi < 13 * (entries + C) + n_layers * C + 12 * C + (2 << 20)
    pf.close()
