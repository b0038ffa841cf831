"""Protected binary32 division wherever trees are evaluated, against the CPU
oracle bit for bit (NaN patterns canonicalised).  Pairs whose operands all lie
within [2^-60, 2^60] take a short sequence that must be the correctly rounded
quotient; one operand outside sends its whole warp to the machine's division.
So the operands stand at both bounds and one unit either side, with zeros,
subnormals, infinities and NaN in all, some and single lanes of a warp, beside
random significands."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

F = np.float32


def _edges():
    lo, hi = F(2.0 ** -60), F(2.0 ** 60)
    v = []
    for b in (lo, hi):
        v += [np.nextafter(b, F(0)), b, np.nextafter(b, F(np.inf))]
    v += [F(1), np.nextafter(F(1), F(0)), np.nextafter(F(1), F(2)), F(3), F(1) / F(3)]
    out = [F(0), F(np.inf), F(1e-45), F(1.1754942e-38), F(1.1754944e-38), F(3.4028235e38), F(2.0 ** 61), F(2.0 ** -61)]
    inside = np.array([x for x in v if lo <= x <= hi], F)
    outside = np.array([x for x in v if not lo <= x <= hi] + out, F)
    return np.concatenate([inside, -inside]), np.concatenate([outside, -outside, np.array([np.nan], F)])


def _random(rng, n):
    """Random significands, exponents over all of the short sequence's range."""
    bits = rng.integers(0, 1 << 23, n, dtype=np.uint32) | (rng.integers(67, 187, n, dtype=np.uint32) << 23)
    return (bits | (rng.integers(0, 2, n, dtype=np.uint32) << 31)).view(F)


def _inputs(seed, C):
    """x: blocks of 128 cases in turn all inside the range, with one lane outside, and mixed; the constants: both kinds."""
    rng = np.random.default_rng(seed)
    inside, outside = _edges()
    x = _random(rng, C)
    for b in range(0, C, 128):
        blk = x[b:b + 128]
        at = rng.permutation(len(blk))
        n = len(blk) // 4
        blk[at[:n]] = rng.choice(inside, n)
        if (b // 128) % 3 == 1:
            blk[at[n]] = rng.choice(outside)
        elif (b // 128) % 3 == 2:
            blk[at[n:2 * n]] = rng.choice(outside, n)
    k = np.concatenate([inside, outside, _random(rng, 251 - len(inside) - len(outside))])
    return x.astype(F), rng.uniform(-1, 1, C).astype(F), k


def _trees(seed):
    """Quotients of leaves in every order, and of quotients: as right, left and both operands."""
    rng = np.random.default_rng(seed)
    const = list(range(5, 256))
    two = [[3, 4, a] for a in const] + [[3, a, 4] for a in const] + [[3, 4, 4]]
    two += [[3, int(a), int(b)] for a, b in zip(rng.integers(5, 256, 600), rng.integers(5, 256, 600))]
    q = [two[int(i)] for i in rng.integers(0, len(two), 600)]
    more = [[3, int(rng.integers(4, 256))] + s for s in q[:150]] + [[3] + s + [int(rng.integers(4, 256))] for s in q[150:300]]
    more += [[3] + a + b for a, b in zip(q[300:450], q[450:600])]
    trees = two + more
    off = np.zeros(len(trees) + 1, np.uint64)
    off[1:] = np.cumsum([len(s) for s in trees])
    return np.concatenate([np.asarray(s, np.uint8) for s in trees]), off


def _same(oracle, got, want):
    got, want = oracle.canon_nan(got), oracle.canon_nan(want)
    bad = np.argwhere(got.view(np.uint32) != want.view(np.uint32))
    assert not len(bad), (len(bad), bad[:3].tolist(), got[tuple(bad[0])], want[tuple(bad[0])])


@pytest.mark.parametrize("T", [1024, 2])              # 2: every node is cached, the pass over cached nodes divides
@pytest.mark.parametrize("C,K", [(32, 1), (300, 1), (64, 2), (333, 2), (128, 4), (400, 4)])
def test_full_evaluation(C, K, T):
    import oracle
    import paper_2205_03251_gb300 as gp
    gp.build()
    x, t, k = _inputs(C + K, C)
    ops, off = _trees(C)
    pop = gp.Population(x, t, k, ops, off, max_nodes=16, cases_per_lane=K, cache_threshold=T)
    pop.eval_full()
    vals, fit = pop.root_values(), pop.fitness()
    pop.close()
    ov, of = oracle.eval_pop_f32(ops, off, k, x, t)
    _same(oracle, vals, ov)
    _same(oracle, fit, of)


@pytest.mark.parametrize("C", [20, 64, 300])
def test_allocation_free_batch(C):
    import oracle
    import torch
    import paper_2205_03251_gb300 as gp
    gp.build()
    x, t, k = _inputs(C, C)
    ops, off = _trees(C + 1)
    dev = torch.device("cuda", 0)
    d_ops = torch.zeros((len(ops) + 15) // 16 * 16, dtype=torch.uint8, device=dev)
    d_ops[:len(ops)] = torch.from_numpy(ops).to(dev)
    d = [torch.from_numpy(np.ascontiguousarray(v)).to(dev) for v in (off.astype(np.int64), x, t, k)]
    P = len(off) - 1
    vals, fit = torch.empty((P, C), device=dev), torch.empty((P,), device=dev)
    assert gp.gp_eval_small_noalloc(d_ops, *d, vals, fit) == 0
    ov, of = oracle.eval_pop_f32(ops, off, k, x, t)
    _same(oracle, vals.cpu().numpy(), ov)
    _same(oracle, fit.cpu().numpy(), of)


@pytest.mark.parametrize("T,onepass", [(2, -1), (2, 0), (1024, 0)])       # walked level by level, or in one pass
@pytest.mark.parametrize("C,K", [(32, 1), (96, 2), (200, 4)])
def test_generations(C, K, T, onepass):
    import oracle
    import paper_2205_03251_gb300 as gp
    gp.build()
    x, t, k = _inputs(C + 7, C)
    ops, off = _trees(C + 2)
    pop = gp.Population(x, t, k, ops, off, max_nodes=256, cases_per_lane=K, cache_threshold=T, seed=3,
                        onepass_nodes=onepass)
    pop.eval_full()
    fit = pop.fitness()
    for g in range(3):
        pl = oracle.plan(ops, off, fit, T=7, seed=3, gen=g, max_nodes=256)
        ops, off = oracle.breed(ops, off, pl)
        pop.crossover(g)
        pop.eval_incremental()
        ov, of = oracle.eval_pop_f32(ops, off, k, x, t)
        fit = pop.fitness()
        _same(oracle, fit, of)
        _same(oracle, pop.root_values(), ov)
    pop.close()


def test_random_significands():
    """8 million quotients of random significands over the short sequence's whole range."""
    import oracle
    import paper_2205_03251_gb300 as gp
    gp.build()
    ops = np.concatenate([np.array([3, 4, a], np.uint8) for a in range(5, 256)])
    off = np.arange(252, dtype=np.uint64) * 3
    for seed in range(8):
        rng = np.random.default_rng(100 + seed)
        x, k = _random(rng, 4096), _random(rng, 251)
        t = np.zeros(4096, F)
        pop = gp.Population(x, t, k, ops, off, max_nodes=16, cases_per_lane=(1, 2, 4)[seed % 3])
        pop.eval_full()
        vals = pop.root_values()
        pop.close()
        _same(oracle, vals, np.where(k[:, None] == 0, F(1), x[None, :] / k[:, None]).astype(F))
