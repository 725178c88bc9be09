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
