"""The sizes at which a kernel or a launch shape changes: each against the
oracle or the step-by-step form, element by element (all values are integers
or bit patterns)."""
import numpy as np
import pytest

import oracle
import paper_2506_01752_gb300 as mocd
import synth

pytestmark = pytest.mark.gpu


def _state_equals(h, ref):
    labels, k1, k2, gen = mocd.get_population(h)
    assert gen == ref.generation
    assert np.array_equal(k1, ref.k1) and np.array_equal(k2, ref.k2)
    assert np.array_equal(labels, ref.labels)


def _regular(n, d, seed):
    """About d neighbours for each of n nodes."""
    rng = np.random.default_rng(seed)
    u = np.repeat(np.arange(n), d // 2)
    return synth.csr_from_edges(n, u, rng.integers(0, n, u.size))


# 40,960 labels are the largest histogram of one block; above it (and for a
# stride that is no multiple of 4) the histogram is global memory.
@pytest.mark.parametrize("n", [40_959, 40_960, 40_961])
@pytest.mark.parametrize("count", [1, 4, 33])
def test_scoring_at_the_histogram_limit(n, count):
    torch = pytest.importorskip("torch")
    rp, ci = _regular(n, 6, seed=n)
    lab = synth.random_labels(n, count, seed=count, n_distinct=n if count == 4 else 300)
    lab[:, -1] = n - 1
    ref = oracle.objectives(rp, ci, lab)
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
    for _ in range(2):  # the second call finds what the first left
        mocd.evaluate_noalloc(d_rp.data_ptr(), d_ci.data_ptr(), n, rows.data_ptr(), count, out[0].data_ptr(),
                              out[1].data_ptr(), torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert np.array_equal(out[0].cpu().numpy(), ref[0]) and np.array_equal(out[1].cpu().numpy(), ref[1])


# 24 generations are the shortest run that launches eights; 31 and 41 leave
# remainders, before and after the eights' graph exists.
@pytest.mark.parametrize("runs", [(23,), (24,), (31, 41), (8, 40, 7)])
def test_runs_in_eights_equal_single_generations(runs):
    rp, ci, _ = synth.planted_partition(5, 30, 0.3, 0.02, seed=4)
    params, op = mocd.Params(pop_size=20, seed=3), oracle.Params(pop_size=20, seed=3)
    h = mocd.graph_upload(rp, ci)
    try:
        mocd.population_init(h, params)
        ref = oracle.population_init(rp, ci, op)
        for g in runs:
            mocd.generation(h, g)
            ref = oracle.run(rp, ci, op, ref, g)
            _state_equals(h, ref)
        mocd.population_init(h, params)  # and again from the start on the same context
        mocd.generation(h, runs[0])
        _state_equals(h, oracle.run(rp, ci, op, oracle.population_init(rp, ci, op), runs[0]))
    finally:
        mocd.destroy(h)


# Nodes of degree 129..512: a warp per quad of children up to 65,536 quads
# (2,048 nodes at N_p 128), per eighth of a node above.
@pytest.mark.parametrize("n", [2040, 2060])
def test_wide_nodes_by_quads_and_eighths(n):
    rp, ci = _regular(n, 150, seed=n)
    deg = np.diff(rp)
    assert (deg > 128).mean() > 0.9 and deg.max() <= 512
    kw = dict(pop_size=128, seed=n, p_mutation=0.3)
    params, op = mocd.Params(**kw), oracle.Params(**kw)
    ref = oracle.population_init(rp, ci, op)
    h = mocd.graph_upload(rp, ci)
    try:
        mocd.population_init(h, params)
        for _ in range(2):
            mocd.generation(h, 1)
            ref = oracle.run_parallel(rp, ci, op, ref, 1)
            _state_equals(h, ref)
    finally:
        mocd.destroy(h)


# From 2^23 edges on the selection's keys no longer fit its 24-bit limbs. A
# complete graph of 4,097 nodes has just over 2^23 edges (and only hubs).
def test_selection_keys_above_24_bits():
    n = 4097
    u, v = np.triu_indices(n, 1)
    assert u.size >= 1 << 23
    rp = np.arange(n + 1, dtype=np.int64) * (n - 1)
    ci = np.broadcast_to(np.arange(n, dtype=np.int32), (n, n))[~np.eye(n, dtype=bool)]
    rng = np.random.default_rng(1)
    lab = rng.integers(0, 1 + 40 * np.arange(8)[:, None], size=(8, n)).astype(np.int32)
    kw = dict(pop_size=8, seed=2, p_mutation=0.01)
    params, op = mocd.Params(**kw), oracle.Params(**kw)
    k1, k2 = oracle.objectives_parallel(rp, ci, lab)
    ref = oracle.State(lab, u.size - k1, k2, 0)
    h = mocd.graph_upload(rp, ci)
    try:
        mocd.set_population(h, params, lab, 0)
        for _ in range(2):
            mocd.generation(h, 1)
            ref = oracle.run_parallel(rp, ci, op, ref, 1)
            _state_equals(h, ref)
    finally:
        mocd.destroy(h)


@pytest.mark.parametrize("value", [-1, 48])
def test_refused_labels_leave_the_population_as_it_was(value):
    rp, ci, _ = synth.planted_partition(4, 12, 0.5, 0.05, seed=3)
    n = rp.size - 1
    params, op = mocd.Params(pop_size=10, seed=1), oracle.Params(pop_size=10, seed=1)
    ref = oracle.run(rp, ci, op, oracle.population_init(rp, ci, op), 2)
    h = mocd.graph_upload(rp, ci)
    try:
        mocd.population_init(h, params)
        mocd.generation(h, 2)
        for count, call in ((10, lambda lab: mocd.set_population(h, params, lab, 0)), (131, lambda lab: mocd.evaluate(h, lab))):
            lab = np.zeros((count, n), np.int32)
            lab[-1, -1] = value
            with pytest.raises(mocd.MocdError) as e:
                call(lab)
            assert e.value.status == -1
        _state_equals(h, ref)
        mocd.generation(h, 1)
        _state_equals(h, oracle.run(rp, ci, op, ref, 1))
    finally:
        mocd.destroy(h)


def test_server_result_above_a_copy_chunk():
    """A front of several MiB: copied on the worker threads."""
    rp, ci = _regular(30_000, 8, seed=5)
    params = mocd.Params(pop_size=60, seed=5)
    h = mocd.graph_upload(rp, ci)
    try:
        mocd.population_init(h, params)
        mocd.generation(h, 3)
        ref = mocd.pareto_front(h)
    finally:
        mocd.destroy(h)
    srv = mocd.Server(1 << 34)
    try:
        job = srv.submit(rp, ci, params, 3)
        while any(srv.step()[:2]):
            pass
        got = srv.result(job)
    finally:
        srv.close()
    assert ref.labels.nbytes > 2 << 20
    assert np.array_equal(got.labels, ref.labels) and np.array_equal(got.sumsq, ref.sumsq)


# Eights are captured inside generation(): on a caller's stream, and while the
# caller's thread captures another stream.
@pytest.mark.parametrize("capturing", [False, True])
def test_eights_on_a_callers_stream(capturing):
    torch = pytest.importorskip("torch")
    rp, ci, _ = synth.planted_partition(5, 30, 0.3, 0.02, seed=4)
    op = oracle.Params(pop_size=20, seed=3)
    ref = oracle.run(rp, ci, op, oracle.population_init(rp, ci, op), 41)
    x = torch.zeros(8, device="cuda")
    own, other, graph = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    h = mocd.graph_upload(rp, ci, own)
    try:
        mocd.population_init(h, mocd.Params(pop_size=20, seed=3))
        torch.cuda.synchronize()
        if capturing:
            with torch.cuda.stream(other):
                graph.capture_begin()
                x.add_(1)
                mocd.generation(h, 41)
                graph.capture_end()
            graph.replay()
        else:
            mocd.generation(h, 41)
        _state_equals(h, ref)
    finally:
        mocd.destroy(h)
    torch.cuda.synchronize()
    assert float(x.sum()) == (8 if capturing else 0)


# Both forms of the scoring's histogram, captured once and replayed twice.
@pytest.mark.parametrize("n", [1000, 40_964])
def test_noalloc_scoring_in_a_callers_graph(n):
    torch = pytest.importorskip("torch")
    rp, ci = _regular(n, 6, seed=n)
    count, graph, side = 8, torch.cuda.CUDAGraph(), torch.cuda.Stream()
    lab = synth.random_labels(n, count, seed=1, n_distinct=300)
    rows = torch.from_numpy(lab.T.copy()).cuda()
    out = torch.full((2, count), -1, dtype=torch.int64, device="cuda")
    d_rp, d_ci = torch.from_numpy(rp.astype(np.int32)).cuda(), torch.from_numpy(ci).cuda()

    def score(stream):
        mocd.evaluate_noalloc(d_rp.data_ptr(), d_ci.data_ptr(), n, rows.data_ptr(), count, out[0].data_ptr(),
                              out[1].data_ptr(), stream)

    with torch.cuda.stream(side):
        score(side)  # looks the scratch's address up
        side.synchronize()
        graph.capture_begin()
        score(side)
        graph.capture_end()
    for seed in (2, 3):
        lab = synth.random_labels(n, count, seed=seed, n_distinct=n if seed == 3 else 300)
        rows.copy_(torch.from_numpy(lab.T.copy()))
        out.fill_(-1)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        ref = oracle.objectives(rp, ci, lab)
        assert np.array_equal(out[0].cpu().numpy(), ref[0]) and np.array_equal(out[1].cpu().numpy(), ref[1])
