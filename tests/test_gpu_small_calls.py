"""Calls that must not cost more than larger ones of the same kind, and the
sums behind them at their edges. Times are compared within one process, with
wide margins, as the best of several runs."""
import time

import numpy as np
import pytest

import oracle
import paper_2506_01752_gb300 as mocd
import synth

pytestmark = pytest.mark.gpu


def _regular(n, d, seed):
    """About d neighbours for each of n nodes."""
    rng = np.random.default_rng(seed)
    u = np.repeat(np.arange(n), d // 2)
    return synth.csr_from_edges(n, u, rng.integers(0, n, u.size))


def _best(f, times=7):
    f()
    best = float("inf")
    for _ in range(times):
        t = time.perf_counter()
        f()
        best = min(best, time.perf_counter() - t)
    return best


# Up to 32 nodes share a warp in a small population: their sums must not take
# turns on the same words of shared memory.
def test_small_populations_cost_no_more_than_large_ones():
    rp, ci, _ = synth.planted_partition(5, 100, 0.1, 0.005, seed=1)
    h = mocd.graph_upload(rp, ci)

    def run(np_):
        mocd.population_init(h, mocd.Params(pop_size=np_, n_parents=4, seed=2))
        mocd.generation(h, 48)
        mocd.synchronize(h)
    try:
        large = _best(lambda: run(100))
        for np_ in (2, 4, 8):
            assert _best(lambda: run(np_)) < 1.2 * large, np_
    finally:
        mocd.destroy(h)


# Sums of squares past 2^44, the third limb of a block's sum: 2 m is above
# 2^22 and every node of a labelling is in one community, or in two.
@pytest.mark.parametrize("n,d", [(41_000, 104), (40_000, 108), (9000, 480)])
@pytest.mark.parametrize("count", [1, 3, 20])
def test_scoring_of_collapsed_labellings(n, d, count):
    torch = pytest.importorskip("torch")
    rp, ci = _regular(n, d, seed=n)
    assert int(rp[-1]) > 1 << 22
    lab = np.zeros((count, n), dtype=np.int32)
    lab[0] = n - 1
    if count > 1:
        lab[1, ::2] = 7
    ref = oracle.objectives(rp, ci, lab)
    assert int(ref[1].max()) > 1 << 44
    h = mocd.graph_upload(rp, ci)
    try:
        got = mocd.evaluate(h, lab)
    finally:
        mocd.destroy(h)
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    rows = torch.zeros((n, (count + 3) // 4 * 4), dtype=torch.int32)
    rows[:, :count] = torch.from_numpy(lab.T.copy())
    rows, out = rows.cuda(), torch.full((2, count), -1, dtype=torch.int64, device="cuda")
    d_rp, d_ci = torch.from_numpy(rp.astype(np.int32)).cuda(), torch.from_numpy(ci).cuda()
    mocd.evaluate_noalloc(d_rp.data_ptr(), d_ci.data_ptr(), n, rows.data_ptr(), count, out[0].data_ptr(),
                          out[1].data_ptr(), torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert np.array_equal(out[0].cpu().numpy(), ref[0]) and np.array_equal(out[1].cpu().numpy(), ref[1])


def _scoring(torch, rp, ci, lab):
    count, n = lab.shape
    rows = torch.zeros((n, (count + 3) // 4 * 4), dtype=torch.int32)
    rows[:, :count] = torch.from_numpy(lab.T.copy())
    rows, out = rows.cuda(), torch.full((2, count), -1, dtype=torch.int64, device="cuda")
    d_rp, d_ci = torch.from_numpy(rp.astype(np.int32)).cuda(), torch.from_numpy(ci).cuda()

    def run():
        mocd.evaluate_noalloc(d_rp.data_ptr(), d_ci.data_ptr(), n, rows.data_ptr(), count, out[0].data_ptr(),
                              out[1].data_ptr(), torch.cuda.current_stream())
        return out
    return run


def _pass_us(torch, run, passes=50):
    for _ in range(10):
        run()
    best = float("inf")
    for _ in range(7):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(passes):
            run()
        torch.cuda.synchronize()
        best = min(best, (time.perf_counter() - t) / passes * 1e6)
    return best


# Where the scoring's histograms move between shared and global memory, by the
# nodes (27,000, 30,000, 40,960) and the row (32 and 64 labellings, 25 to 48).
@pytest.mark.parametrize("n", [27_000, 27_001, 30_001, 40_961])
@pytest.mark.parametrize("count", [24, 25, 29, 32, 33, 48, 49, 61, 64, 65])
def test_scoring_in_either_histogram(n, count):
    torch = pytest.importorskip("torch")
    rp, ci = _regular(n, 6, seed=n)
    lab = synth.random_labels(n, count, seed=count, n_distinct=200)
    lab[:, -1] = n - 1
    lab[-1] = n - 1  # the last labelling's last label, everywhere
    ref = oracle.objectives_parallel(rp, ci, lab)
    run = _scoring(torch, rp, ci, lab)
    for _ in range(2):  # the second call finds what the first left
        got = run().cpu().numpy()
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])


# Few communities: the labellings' cells must not share sectors, where the
# additions of all nodes would take turns.
def test_scoring_of_few_communities_is_no_cliff():
    torch = pytest.importorskip("torch")
    rp, ci = _regular(60_000, 10, seed=2)
    many = synth.random_labels(60_000, 64, seed=1, n_distinct=600)
    few = np.broadcast_to(many[:1] % 2, many.shape)
    assert _pass_us(torch, _scoring(torch, rp, ci, few)) < 3 * _pass_us(torch, _scoring(torch, rp, ci, many))


# A row of 128 bytes, which a histogram block reads slowest.
def test_scoring_of_32_labellings_costs_little_more_than_20():
    torch = pytest.importorskip("torch")
    rp, ci = _regular(40_000, 16, seed=2)
    t = {c: _pass_us(torch, _scoring(torch, rp, ci, synth.random_labels(40_000, c, seed=1, n_distinct=400)))
         for c in (20, 32)}
    assert t[32] < 1.25 * t[20], t


# mocd_set_population checks up to 32,768 labels on the host, more on the
# device. Either way a label out of range is refused and the population that
# was there stays.
@pytest.mark.parametrize("n,np_", [(64, 1), (256, 128), (257, 128), (8191, 4), (8193, 4)])
def test_set_population_refuses_labels_out_of_range(n, np_):
    rp, ci = _regular(n, 6, seed=n)
    good = synth.random_labels(n, np_, seed=1)
    params = mocd.Params(pop_size=np_, n_parents=1, seed=3)
    h = mocd.graph_upload(rp, ci)
    try:
        mocd.set_population(h, params, good, 5)
        before = mocd.get_population(h)
        assert np.array_equal(before[0], good)
        for at, label in ((0, -1), (-1, n), (good.size // 2, -2**31), (-1, 2**31 - 1)):
            bad = good.copy()
            bad.reshape(-1)[at] = label
            with pytest.raises(mocd.MocdError):
                mocd.set_population(h, params, bad, 7)
            after = mocd.get_population(h)
            assert all(np.array_equal(x, y) for x, y in zip(before, after))
        mocd.generation(h, 1)  # and it still runs
        ref = oracle.run(rp, ci, oracle.Params(pop_size=np_, n_parents=1, seed=3),
                         oracle.State(good, before[1], before[2], 5), 1)
        assert np.array_equal(mocd.get_population(h)[0], ref.labels)
    finally:
        mocd.destroy(h)


def test_set_population_of_few_labels_costs_little_more_than_an_init():
    rp, ci = _regular(200, 6, seed=1)
    params = mocd.Params(pop_size=1, n_parents=1, seed=3)
    lab = synth.random_labels(200, 1, seed=1)
    h = mocd.graph_upload(rp, ci)
    try:
        init = _best(lambda: mocd.population_init(h, params), times=60)
        assert _best(lambda: mocd.set_population(h, params, lab, 0), times=60) < 1.45 * init
    finally:
        mocd.destroy(h)


# nodes_per_warp is for the many short items: the votes of degrees 33 to 128 must
# not queue up behind each other on few warps. 60 nodes of degree about 100.
def test_nodes_per_warp_leaves_long_votes_alone():
    hs = []
    try:
        for seed in range(8):
            rng = np.random.default_rng(seed)
            u = np.concatenate([np.repeat(np.arange(1000), 10), np.repeat(np.arange(60), 80)])
            rp, ci = synth.csr_from_edges(1000, u, rng.integers(0, 1000, u.size))
            d = np.diff(rp)
            assert ((d > 64) & (d <= 128)).sum() >= 50
            hs.append(mocd.graph_upload(rp, ci))
            mocd.population_init(hs[-1], mocd.Params(seed=seed))
        batch = mocd.batch_create(hs)
        t = {}
        try:
            for npw in (1, 8):
                mocd.batch_configure(batch, npw, 0)

                def run():
                    mocd.batch_generation(batch, 10)
                    mocd.batch_synchronize(batch)
                t[npw] = _best(run)
        finally:
            mocd.batch_destroy(batch)
        assert t[8] < 1.5 * t[1], t
    finally:
        for h in hs:
            mocd.destroy(h)


# Nodes of degree 129..512 of a settled population, whose pairs are settled by
# counting the own label first: by quads up to 65,536 quads, by quarters above.
@pytest.mark.parametrize("n", [2600, 2660])
def test_wide_nodes_of_a_settled_population(n):
    rng = np.random.default_rng(n)
    u = np.repeat(np.arange(n), 130)
    v = np.where(rng.random(u.size) < 0.9, u // 400 * 400 + rng.integers(0, 400, u.size), rng.integers(0, n, u.size))
    rp, ci = synth.csr_from_edges(n, u, np.minimum(v, n - 1))
    deg = np.diff(rp)
    wide = int(((deg > 128) & (deg <= 512)).sum())
    assert (wide * 25 > 65536) == (n == 2660) and wide > 0.9 * n
    lab = np.repeat((np.arange(n) // 400 * 400).astype(np.int32)[None], 100, 0)
    stray = rng.random(lab.shape) < 0.05 * rng.random((100, 1))
    lab[stray] = rng.integers(0, n, int(stray.sum()))
    k1, k2 = oracle.objectives_parallel(rp, ci, lab)
    op = oracle.Params(pop_size=100, seed=n)
    ref = oracle.State(lab, int(rp[-1]) // 2 - k1, k2, 0)
    h = mocd.graph_upload(rp, ci)
    try:
        mocd.set_population(h, mocd.Params(pop_size=100, seed=n), lab, 0)
        for _ in range(3):  # the second and third know what the one before settled
            mocd.generation(h, 1)
            ref = oracle.run_parallel(rp, ci, op, ref, 1)
            labels, g1, g2, gen = mocd.get_population(h)
            assert np.array_equal(g1, ref.k1) and np.array_equal(g2, ref.k2) and np.array_equal(labels, ref.labels)
    finally:
        mocd.destroy(h)
