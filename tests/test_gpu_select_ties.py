"""Selection on populations full of identical members, long dominance chains
and fronts of every size, at the edges of its counting loops (threads per
point, eight places a lane, 32-place head masks): P order, keys and the
parents drawn from it equal the oracle's over several generations."""
import numpy as np
import pytest

import oracle
import paper_2506_01752_gb300 as mocd
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("np_", [1, 2, 3, 8, 9, 31, 32, 33, 63, 65, 100, 127, 128])
@pytest.mark.parametrize("kind", ["copies", "chain", "mixed"])
def test_selection_with_ties_matches_oracle(np_, kind):
    rp, ci, _ = synth.planted_partition(4, 12, 0.5, 0.05, seed=3)
    n = rp.size - 1
    rng = np.random.default_rng(np_)
    if kind == "copies":  # three distinct members, children are copies
        base = rng.integers(0, 4, size=(3, n), dtype=np.int64)
        lab = base[rng.integers(0, 3, size=np_)]
        kw = dict(p_crossover=0.0, p_mutation=0.0, n_parents=1)
    elif kind == "chain":  # splitting one node after the other off one community
        lab = np.zeros((np_, n), np.int64)
        for i in range(np_):
            k = i % n
            lab[i, :k] = np.arange(1, k + 1) % n
        kw = dict(p_crossover=0.5, p_mutation=0.01, n_parents=16)
    else:
        lab = rng.integers(0, 1 + np.arange(np_)[:, None] % n, size=(np_, n))
        kw = dict(p_crossover=0.8, p_mutation=0.02, n_parents=5)
    lab = np.ascontiguousarray(lab, dtype=np.int32)
    h = mocd.graph_upload(rp, ci)
    try:
        mocd.set_population(h, mocd.Params(pop_size=np_, seed=np_, **kw), lab, 0)
        k1, k2 = oracle.objectives(rp, ci, lab)
        st = oracle.State(lab, int(rp[-1] // 2) - k1, k2, 0)
        op = oracle.Params(pop_size=np_, seed=np_, **kw)
        front = mocd.pareto_front(h)
        members, best = oracle.pareto_front(st, int(rp[-1] // 2))
        assert front.best == best and np.array_equal(front.labels, st.labels[members])
        for _ in range(4):
            st = oracle.run(rp, ci, op, st, 1)
            mocd.generation(h, 1)
            labels, g1, g2, _ = mocd.get_population(h)
            assert np.array_equal(g1, st.k1) and np.array_equal(g2, st.k2)
            assert np.array_equal(labels, st.labels)
        front = mocd.pareto_front(h)
        members, best = oracle.pareto_front(st, int(rp[-1] // 2))
        assert front.best == best and np.array_equal(front.labels, st.labels[members])
    finally:
        mocd.destroy(h)
