"""Distinct portfolios are independent: two host threads run two portfolios whose kernels are the same
functions with different amounts of shared memory, on a stream each, and every result equals the
one computed alone.  Likewise a plan whose function a later, narrower plan uses too."""
import ctypes
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_1606_04473_gb300 as ara


def world(seed, C, n_elts, nnz, n_layers, trials=60, events=400):
    """Every event in about the same number of entries per event whatever the layers: the rows' form
    depends on n_layers * nnz / C."""
    g = np.random.default_rng(seed)
    ids = [g.choice(C, size=nnz, replace=False).astype(np.int32) for _ in range(n_elts)]
    loss = [np.exp(11.0 + 2.0 * g.standard_normal(nnz)) for _ in ids]
    layers = [[l % n_elts] for l in range(n_layers)]
    z = np.zeros(n_layers)
    pf = ara.Portfolio(C, ids, loss, np.full(n_elts, 1e4), np.full(n_elts, 1e6), layers, z + 1e4, z + 9e5, z + 1e5,
                       z + 1e7)
    counts = g.poisson(events, trials)
    off = np.zeros(trials + 1, np.int64)
    np.cumsum(counts, out=off[1:])
    return pf, torch.from_numpy(off).cuda(), torch.from_numpy(g.integers(0, C, off[-1], dtype=np.int32)).cuda()


def run(w, stream, kind):
    pf, off, ids = w
    n_layers = pf.n_layers
    if kind == "single":
        return pf.run_ylt(off, ids, layers=[0], stream=stream)
    if kind == "adjoint":
        reg = torch.empty((1, off.numel() - 1), dtype=torch.uint8, device="cuda")
        y = pf.run_ylt(off, ids, layers=[0], regimes=reg, stream=stream)
        return pf.adjoint(off, ids, y, reg, 0.9, layers=[0], stream=stream)["layer"]
    flags = ara.ARA_RUN_BATCHED if kind == "batched" else 0
    return pf.run_ylt(off, ids, layers=list(range(n_layers)), flags=flags, stream=stream)


# the rows in place (32 columns of sums, 16 and 3 layers) as an ordinary and as a batched run, rows end to
# end, and the single-layer stream and histogram over a small and a large catalogue
@pytest.mark.parametrize("kind,a,b", [
    ("plain", (20_000, 16, 900, 16), (20_000, 3, 4_500, 3)),
    ("batched", (20_000, 16, 900, 16), (20_000, 3, 4_500, 3)),
    ("batched", (3_000, 16, 1_500, 16), (3_000, 8, 2_900, 8)),
    ("single", (1_500_000, 2, 900, 1), (20_000, 2, 900, 1)),
    ("adjoint", (1_500_000, 2, 900, 1), (20_000, 2, 900, 1)),
])
def test_two_portfolios_from_two_threads(kind, a, b):
    worlds = [world(1, *a), world(2, *b)]
    streams = [torch.cuda.Stream() for _ in worlds]
    torch.cuda.synchronize()
    want = []
    for w, s in zip(worlds, streams):
        with torch.cuda.stream(s):
            want.append(run(w, s, kind))
        w[0].check(s)
    start, failed = threading.Barrier(2), []

    def work(k):
        (pf, off, ids), s = worlds[k], streams[k]
        n_sel = 1 if kind in ("single", "adjoint") else pf.n_layers
        sel = (ctypes.c_int32 * n_sel)(*range(n_sel))
        out = torch.empty_like(want[k])
        f, args = ara.lib().ara_run_ylt, (pf._h, off.numel() - 1, off.data_ptr(), ids.numel(), ids.data_ptr(), None,
                                          n_sel, sel, out.data_ptr(), None,
                                          ara.ARA_RUN_BATCHED if kind == "batched" else 0, s.cuda_stream)
        torch.cuda.synchronize()
        start.wait(timeout=60)
        for i in range(20):
            if kind == "adjoint":
                with torch.cuda.stream(s):
                    sts = {0}
                    out = run(worlds[k], s, kind)
            else:
                sts = {f(*args) for _ in range(1000)}     # back to back: the calls of the threads overlap
            s.synchronize()
            if sts != {0} or not torch.equal(out, want[k]):
                failed.append((k, i, sts))
                return
        pf.check(s)

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for w in worlds:
        w[0].close()
    assert not failed


@pytest.mark.parametrize("where", ["another thread", "the capturing thread"])
def test_an_ordinary_run_beside_a_capture(where):
    """A run of several layers (by rows, with scratch from the pool) on a stream of its own neither fails nor
    spoils the capture that is going on in the process, in any mode."""
    w = world(5, 20_000, 16, 900, 16)
    pf, off, ids = w
    side, s = torch.cuda.Stream(), torch.cuda.Stream()
    want = run(w, None, "plain")
    out = torch.zeros_like(want)
    x = torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    ara.lib().ara_release_memory()
    for mode in ("global", "thread_local", "relaxed"):
        out.zero_()
        torch.cuda.synchronize()
        graph, failed = torch.cuda.CUDAGraph(), []

        def work():
            try:
                n0 = ara.launch_count()
                pf.run_ylt(off, ids, out=out, stream=side)
                if ara.launch_count() - n0 > 3:
                    failed.append("not by rows")
            except ara.AraError as e:
                failed.append(str(e))

        with torch.cuda.graph(graph, stream=s, capture_error_mode=mode):
            x += 1
            if where == "another thread":
                t = threading.Thread(target=work)
                t.start()
                t.join()
            else:
                work()
            x += 1
        assert not failed
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert bool((x == 2).all())
    pf.check()
    pf.close()


def test_a_wide_plan_outlives_the_making_of_a_narrow_one():
    wide, narrow = world(3, 20_000, 16, 900, 16), world(4, 20_000, 3, 4_500, 3)
    want = run(wide, None, "plain")
    p = ara.BatchedPlan(wide[0], wide[1], wide[2], autotune=False)
    q = ara.BatchedPlan(narrow[0], narrow[1], narrow[2], autotune=False)
    assert torch.equal(p.launch(), want)
    q.launch()
    assert torch.equal(p.launch(), want)
    wide[0].check()
    for x in (p, q, wide[0], narrow[0]):
        x.close()
