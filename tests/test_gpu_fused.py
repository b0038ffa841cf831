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


@pytest.mark.parametrize("C,K", [(1, 1), (48, 1), (48, 2), (33, 2), (130, 4), (97, 4)])
@pytest.mark.parametrize("integer", [False, True])
def test_every_pair_of_functions(C, K, integer):
    """f g L L with every pair of functions and leaf kinds: each operation rounds by itself (a joined product and sum
    would not), against the oracle bit for bit."""
    import itertools
    import oracle
    import synth
    import paper_2205_03251_gb300 as gp
    if integer and K == 4:
        pytest.skip("binary32 only")
    gp.build()
    (x, t), k = (synth.cases_int(9, C), synth.consts_int(9)) if integer else (synth.cases(9, C), synth.consts(9))
    trees = [[f, g, a, b, c] for f, g, a, b, c in itertools.product(range(4), range(4), (4, 10), (4, 20), (4, 30))]
    trees += [[h] + s + [31] for h, s in itertools.product((0, 2), list(trees))]      # the running value is kept
    o = np.zeros(len(trees) + 1, np.uint64)
    o[1:] = np.cumsum([len(s) for s in trees])
    ops = np.concatenate([np.asarray(s, np.uint8) for s in trees])
    pop = gp.Population(x, t, k, ops, o, max_nodes=16, cases_per_lane=K, integer=integer)
    pop.eval_full()
    vals, fit = pop.root_values(), pop.fitness()
    pop.close()
    ov, of = (oracle.eval_pop_i32 if integer else oracle.eval_pop_f32)(ops, o, k, x, t)
    canon = (lambda v: v) if integer else oracle.canon_nan
    assert np.array_equal(canon(vals), canon(ov)) and np.array_equal(canon(fit), canon(of))


def _remy(sizes, seed):
    import synth
    return synth.population("remy", seed, len(sizes), sizes=np.asarray(sizes, np.uint64))


@pytest.mark.parametrize("C", [64, 65, 128, 129, 193, 1023, 1025, 1056, 2049, 4096])
def test_case_blocks_of_the_skeleton(C):
    """Trees with cached nodes over case counts on either side of the lane rules (64 x odd and even, four cases per
    lane or two) and of 32 case blocks, which the pass over cached nodes takes in groups."""
    import oracle
    import synth
    import paper_2205_03251_gb300 as gp
    gp.build()
    ops, off = _remy([1, 3, 255, 257, 1023, 1025, 3001, 9001], 13)
    (x, t), k = synth.cases(6, C), synth.consts(6)
    ov, of = oracle.eval_pop_f32(ops, off, k, x, t)
    for K in (0, 1, 2, 4):
        pop = gp.Population(x, t, k, ops, off, max_nodes=9001, cache_threshold=128, cases_per_lane=K)
        pop.eval_full()
        vals, fit = pop.root_values(), pop.fitness()
        pop.close()
        assert np.array_equal(oracle.canon_nan(vals), oracle.canon_nan(ov)), K
        assert np.array_equal(oracle.canon_nan(fit), oracle.canon_nan(of)), K


@pytest.mark.parametrize("T", [2, 16, 32, 64, 128, 256, 512, 1024])
def test_cached_nodes_at_every_threshold(T):
    """The structure pass marks exactly the nodes that head T nodes or more and the root, for trees that end around
    its 32-node chunks and 1,024-node blocks; the subtree sizes are recounted here."""
    import synth
    import paper_2205_03251_gb300 as gp
    gp.build()
    ops, off = _remy([1, 3, 31, 33, 63, 65, 127, 1023, 1025, 1055, 1057, 2047, 2049, 2111, 4095, 9217, 30001], 29)
    trees = [ops[int(off[i]):int(off[i + 1])] for i in range(len(off) - 1)]
    rng = np.random.default_rng(3)
    for n in (31, 32, 33, 511, 512, 513, 1023, 1024, 1500):
        for left in (True, False):
            trees.append(np.asarray(_comb(n, left, rng, lambda: 4), np.uint8))
    o = np.zeros(len(trees) + 1, np.uint64)
    o[1:] = np.cumsum([len(s) for s in trees])
    x, t = synth.cases(6, 5)
    pop = gp.Population(x, t, synth.consts(6), np.concatenate(trees), o, max_nodes=30001, cache_threshold=T)
    pop.eval_full()
    for i, s in enumerate(trees):
        size, stack = np.zeros(len(s), np.int64), []
        for p in range(len(s) - 1, -1, -1):
            size[p] = 1 + (stack.pop() + stack.pop() if s[p] < 4 else 0)
            stack.append(int(size[p]))
        want = [p for p in range(len(s)) if size[p] >= T or p == 0]
        pos, end, _ = pop.cache_entries(i)
        pos = np.asarray(pos, np.int64)
        assert np.array_equal(pos, want), (i, len(s))
        assert np.array_equal(np.asarray(end, np.int64) - pos, size[want]), (i, len(s))
    pop.close()


@pytest.mark.parametrize("P,C", [(1, 4096), (2, 4096), (300, 2), (300, 32), (300, 33), (200, 512)])
def test_allocation_free_batches_at_the_edges(P, C):
    """Few trees over many cases (tasks by block), many trees over few cases, and stacks beyond the shared window in
    more warps than there are overflow stacks, which then take turns."""
    import oracle
    import synth
    import torch
    import paper_2205_03251_gb300 as gp
    gp.build()
    gp.load()
    deep = np.array([2] * 511 + [4] + [5 + (j % 9) for j in range(511)], np.uint8)
    mid = np.array([1] * 97 + [4] * 98, np.uint8)
    trees = [(deep, mid, np.array([4], np.uint8))[i % 3] for i in range(P)]
    o = np.zeros(P + 1, np.uint64)
    o[1:] = np.cumsum([len(s) for s in trees])
    ops = np.concatenate(trees)
    (x, t), k = synth.cases(8, C), synth.consts(8)
    dev = torch.device("cuda", 0)
    d_ops = torch.zeros((len(ops) + 15) // 16 * 16, dtype=torch.uint8, device=dev)
    d_ops[:len(ops)] = torch.from_numpy(ops).to(dev)
    d = [torch.from_numpy(np.ascontiguousarray(v)).to(dev) for v in (o.astype(np.int64), x, t, np.asarray(k, np.float32))]
    vals = torch.empty((P, C), dtype=torch.float32, device=dev)
    fit = torch.empty((P,), dtype=torch.float32, device=dev)
    assert gp.gp_eval_small_noalloc(d_ops, *d, vals, fit) == 0
    ov, of = oracle.eval_pop_f32(ops, o, k, x, t)
    assert np.array_equal(oracle.canon_nan(vals.cpu().numpy()), oracle.canon_nan(ov))
    assert np.array_equal(oracle.canon_nan(fit.cpu().numpy()), oracle.canon_nan(of))
