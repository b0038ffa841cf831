"""Chains of cached nodes in the pass over cached nodes: a climb takes their
descriptors 32 and their operands 8 at a time, so the chains end on and beside
those borders, hang left, right and alternately, and meet others half way.  Root
values against the CPU oracle bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LENGTHS = (1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 39, 40, 41, 63, 64, 65, 72, 96, 97, 130, 700)


def _chain(n, side, rng, leaf):
    """n functions above one leaf, each with a leaf on the right (0), the left (1) or either side (2)."""
    out, right = [], []
    for _ in range(n):
        out.append(int(rng.integers(4)))
        if side == 1 or (side == 2 and rng.random() < 0.5):
            out.append(leaf())
        else:
            right.append(leaf())
    return out + [leaf()] + right[::-1]


@pytest.mark.parametrize("kind,C,K", [("f32", 48, 2), ("f32", 20, 1), ("f32", 300, 4), ("i32", 48, 2), ("i32", 100, 1),
                                      ("mux6", 64, 1), ("mux11", 2048, 2)])
@pytest.mark.parametrize("T", [2, 16])
def test_chains(kind, C, K, T):
    import oracle
    import synth
    import paper_2205_03251_gb300 as gp
    gp.build()
    rng = np.random.default_rng(17)
    n_in = {"mux6": 6, "mux11": 11}.get(kind)

    def leaf():
        return int(rng.integers(4, 4 + n_in)) if n_in else (4 if rng.random() < 0.5 else int(rng.integers(5, 256)))

    trees = [_chain(n, side, rng, leaf) for n in LENGTHS for side in (0, 1, 2)]
    trees += [[int(rng.integers(4))] + _chain(a, 2, rng, leaf) + _chain(b, 2, rng, leaf)
              for a, b in zip(LENGTHS, LENGTHS[::-1])]
    off = np.zeros(len(trees) + 1, np.uint64)
    off[1:] = np.cumsum([len(s) for s in trees])
    ops = np.concatenate([np.asarray(s, np.uint8) for s in trees])
    (x, t), k = (synth.cases_int(5, C), synth.consts_int(5)) if kind == "i32" else (synth.cases(5, C), synth.consts(5))
    pop = gp.Population(x, t, k, ops, off, max_nodes=2000, cache_threshold=T, cases_per_lane=K, integer=kind == "i32",
                        boolean=bool(n_in), mux_k=3 if kind == "mux11" else 2)
    pop.eval_full()
    vals = pop.root_values()
    pop.close()
    if kind == "f32":
        ov, _ = oracle.eval_pop_f32(ops, off, k, x, t)
        assert np.array_equal(oracle.canon_nan(vals), oracle.canon_nan(ov))
    elif kind == "i32":
        ov, _ = oracle.eval_pop_i32(ops, off, k, x, t)
        assert np.array_equal(vals, ov)
    else:
        for i, s in enumerate(trees):
            want = oracle.eval_node_mux(np.asarray(s, np.uint8), 0, 3 if kind == "mux11" else 2)
            assert np.array_equal(np.atleast_1d(vals[i]), np.atleast_1d(want)), i
