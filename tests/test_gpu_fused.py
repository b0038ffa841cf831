"""The fused interpreter at the sizes where it can go wrong: runs that end
on and around the edges of its 128-node chunks, stacks that stay just inside,
cross and return through the shared window, leaves and functions on either
side of a chunk's edge.  Root values and fitness against the CPU oracle, bit
for bit (NaN patterns canonicalised): the same operations on the same operands
leave no tolerance."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _comb(n, left, rng, leaf):
    """n functions in a chain: a left comb keeps n leaves pending, a right comb none."""
    if left:
        return [int(rng.integers(4)) for _ in range(n)] + [leaf() for _ in range(n + 1)]
    return sum(([int(rng.integers(4)), leaf()] for _ in range(n)), []) + [leaf()]


def _bushes(n, depth, rng, leaf):
    """n left combs of `depth` pending leaves, one after another along a right spine: the stack goes up to depth and
    back n times, crossing a window of that depth in every chunk."""
    out = []
    for _ in range(n):
        out += [int(rng.integers(4))] + _comb(depth, True, rng, leaf)
    return out + [leaf()]


def _trees(kind):
    import synth
    rng = np.random.default_rng(20220503)
    if kind == "f32" or kind == "i32":
        def leaf():
            return 4 if rng.random() < 0.5 else int(rng.integers(5, 256))
        nin = None
    else:
        nin = {"mux6": 6, "mux11": 11}[kind]

        def leaf():
            return int(rng.integers(4, 4 + nin))
    trees = [[leaf()], [int(rng.integers(4)), leaf(), leaf()]]
    for n in (1, 2, 7, 15, 16, 17, 31, 32, 33, 61, 63, 64, 65, 66, 127, 128, 129, 255, 256, 511):
        trees += [_comb(n, True, rng, leaf), _comb(n, False, rng, leaf)]
    for depth in (13, 14, 15, 16, 17, 30, 31, 32, 33, 62, 63, 64, 65, 66):
        trees.append(_bushes(max(1, 900 // (2 * depth + 2)), depth, rng, leaf))
    sizes = np.array([2 * (int(s) // 2) + 1 for s in
                      list(range(3, 80)) + list(range(119, 139)) + list(range(247, 267)) +
                      [381, 383, 385, 387, 511, 513, 1021, 1023, 1025, 2045, 2047, 2049, 4095, 5001, 20001]], np.uint64)
    kw = {} if nin is None else {"boolean": True, "n_inputs": nin}
    ops, off = synth.population("remy", 77, len(sizes), sizes=sizes, **kw)
    trees += [list(ops[int(off[i]):int(off[i + 1])]) for i in range(len(sizes))]
    o = np.zeros(len(trees) + 1, np.uint64)
    o[1:] = np.cumsum([len(t) for t in trees])
    return np.concatenate([np.asarray(t, np.uint8) for t in trees]), o


@pytest.mark.parametrize("kind,C,K,W", [("f32", 48, 2, 0), ("f32", 33, 1, 16), ("f32", 130, 4, 32), ("f32", 64, 2, 64),
                                        ("f32", 1, 1, 64), ("i32", 48, 2, 0), ("i32", 20, 1, 32), ("mux6", 64, 1, 0),
                                        ("mux11", 2048, 2, 0), ("mux11", 2048, 1, 64)])
def test_full_evaluation_at_the_edges(kind, C, K, W):
    import oracle
    import synth
    import paper_2205_03251_gb300 as gp
    gp.build()
    ops, off = _trees(kind)
    boolean = kind.startswith("mux")
    if kind == "i32":
        (x, t), k = synth.cases_int(5, C), synth.consts_int(5)
    else:
        (x, t), k = synth.cases(5, C), synth.consts(5)
    for T in (1024, 128):
        pop = gp.Population(x, t, k, ops, off, max_nodes=20001, cache_threshold=T, cases_per_lane=K, stack_window=W,
                            boolean=boolean, integer=kind == "i32", mux_k=3 if kind == "mux11" else 2)
        pop.eval_full()
        vals = pop.root_values()
        fit = pop.fitness()
        pop.close()
        if kind == "f32":
            ov, of = oracle.eval_pop_f32(ops, off, k, x, t)
            assert np.array_equal(oracle.canon_nan(vals), oracle.canon_nan(ov)), T
            assert np.array_equal(oracle.canon_nan(fit), oracle.canon_nan(of)), T
        elif kind == "i32":
            ov, of = oracle.eval_pop_i32(ops, off, k, x, t)
            assert np.array_equal(vals, ov) and np.array_equal(fit, of), T
        else:
            for i in range(len(off) - 1):
                want = oracle.eval_node_mux(ops[int(off[i]):int(off[i + 1])], 0, 3 if kind == "mux11" else 2)
                assert np.array_equal(np.atleast_1d(vals[i]), np.atleast_1d(want)), (T, i)
