"""f g L L over the Boolean sets: every pair of functions with every choice of
leaves, alone, with a running value kept beside it, and on a stack that a chunk
of 128 nodes drives past the shared window.  Bit for bit against the CPU oracle."""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _check(trees, mux_k, K, W):
    import oracle
    import paper_2205_03251_gb300 as gp
    gp.build()
    off = np.zeros(len(trees) + 1, np.uint64)
    off[1:] = np.cumsum([len(s) for s in trees])
    ops = np.concatenate([np.asarray(s, np.uint8) for s in trees])
    pop = gp.Population(None, None, np.zeros(251, np.float32), ops, off, max_nodes=max(map(len, trees)), boolean=True,
                        mux_k=mux_k, cases_per_lane=K, stack_window=W)
    pop.eval_full()
    vals = pop.root_values()
    pop.close()
    for i, s in enumerate(trees):
        want = oracle.eval_node_mux(np.asarray(s, np.uint8), 0, mux_k)
        assert np.array_equal(np.atleast_1d(vals[i]), np.atleast_1d(want)), (i, s[:12])


@pytest.mark.parametrize("mux_k,K", [(2, 1), (3, 1), (3, 2)])
def test_every_pair(mux_k, K):
    rng = np.random.default_rng(mux_k)
    n = {2: 6, 3: 11}[mux_k]
    leaf = list(range(4, 4 + n))
    three = [tuple(int(v) for v in rng.choice(leaf, 3)) for _ in range(6)] + [(leaf[0], leaf[-1], leaf[1]), (leaf[5],) * 3]
    pairs = [[f, g, a, b, c] for f, g, (a, b, c) in itertools.product(range(4), range(4), three)]
    trees = pairs + [[h] + s + [leaf[2]] for h, s in itertools.product(range(4), pairs[::3])]
    trees += [[h, leaf[3]] + s for h, s in itertools.product(range(4), pairs[1::3])]
    trees += [[h] + s + r for h, s, r in zip(itertools.cycle(range(4)), pairs, pairs[::-1])]
    _check(trees, mux_k, K, 16)


@pytest.mark.parametrize("W", [16, 32])
@pytest.mark.parametrize("mux_k,K", [(2, 1), (3, 1), (3, 2)])
def test_pairs_past_the_window(mux_k, K, W):
    """n pending operands of five nodes each: about 25 of them in a chunk, where the window holds 16; with operands of
    one node between them more than 32."""
    rng = np.random.default_rng(7 + mux_k)
    n = {2: 6, 3: 11}[mux_k]

    def pair():
        return [int(v) for v in rng.integers(0, 4, 2)] + [int(v) for v in rng.integers(4, 4 + n, 3)]

    trees = []
    for m in (8, 15, 16, 17, 24, 30, 40, 100):
        for every in (1, 4):
            operands = [pair() if j % every == 0 else [int(rng.integers(4, 4 + n))] for j in range(m + 1)]
            trees.append([int(v) for v in rng.integers(0, 4, m)] + sum(operands, []))
    _check(trees, mux_k, K, W)
